"""A batch of more scenes than a block has threads, with and without rigid bodies: every tile finds
its scene past the first 256, in both launch structures that look it up; each scene as stepped
alone, bit for bit."""
import numpy as np
import pytest

from paper_2511_15908_gb300 import scenes

from test_gpu_parity import sph  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bps", [0, 1])
def test_many_scenes_equal_each_alone(sph, bps):  # noqa: F811
    scs = [scenes.tiny(seed=s, n=(2 + s % 3, 2, 2 + s % 2), with_bodies=s % 3 > 0) for s in range(263)]
    sims = [sph.Simulation(sc) for sc in scs]
    batch = sph.Batch(sims)
    batch.configure(bps, 1)
    batch.step(2)
    batch.sync()
    for i in (0, 1, 127, 255, 256, 257, 262):
        alone = sph.Simulation(scs[i])
        alone.step(2)
        a, b = alone.state(), sims[i].state()
        for key in ("x", "v", "rho"):
            np.testing.assert_array_equal(a[key], b[key])
        alone.close()
    batch.close()
    for s in sims:
        s.close()

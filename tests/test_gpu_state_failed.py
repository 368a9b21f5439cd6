"""A state read that fails leaves the caller's arrays as they were."""
import numpy as np
import pytest

from paper_2511_15908_gb300 import scenes

from test_gpu_failed_call import read_under_capture
from test_gpu_parity import sph  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", ["pinned", "direct"])
def test_failed_read_keeps_the_arrays(sph, size):  # noqa: F811
    sc = (scenes.dam_break(seed=1, grab=True) if size == "pinned" else
          scenes.coupled(seed=0, n_fluid=30_000, cols=(40, 30), tank=(0.4, 0.3, 0.5), n_substeps=10, probe_r=0.04, soft_n=6))
    sim = sph.Simulation(sc)
    sim.step(1)
    sim.sync()
    x, v = np.full((sim.n, 3), 7.0, np.float32), np.full((sim.n, 3), 8.0, np.float32)
    read_under_capture(sph, sim, x, v)
    assert np.all(x == 7.0) and np.all(v == 8.0)
    sim.close()

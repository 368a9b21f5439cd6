"""Pinned host memory of a handle goes by its scene's size: many small scenes take little."""
import pytest
import torch

from paper_2511_15908_gb300 import scenes

from test_gpu_parity import sph  # noqa: F401

pytestmark = pytest.mark.gpu


def _shared_kb():
    """Resident shared memory of this process: the driver's pinned host allocations count here."""
    with open("/proc/self/status") as f:
        for line in f:
            if line.startswith("RssShmem:"):
                return int(line.split()[1])
    pytest.skip("no RssShmem on this system")


def test_many_small_scenes_pin_little(sph):  # noqa: F811
    stream = torch.cuda.Stream()
    sc = scenes.tiny(seed=0, n=(2, 2, 2))
    first = sph.Simulation(sc, stream=stream)
    first.step(1)
    first.state()
    before = _shared_kb()
    sims = [sph.Simulation(sc, stream=stream) for _ in range(64)]
    grown = _shared_kb() - before
    # a scene's status, haptic slot and state are under 8 KB; up to 64 KB each for the
    # driver's rounding
    assert grown <= 64 * 64, f"{grown} KB for 64 scenes of {sc.n_total} particles"
    for s in sims + [first]:
        s.close()

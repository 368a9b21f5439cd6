"""The state read, put in id order on the GPU: a scene whose arrays come through pinned memory in
one copy and one whose arrays go straight to the caller, with and without the debug record,
against the slots and ids that a checkpoint holds, bit for bit."""
import numpy as np
import pytest

from paper_2511_15908_gb300 import scenes

from test_gpu_parity import sph  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("record", [False, True])
@pytest.mark.parametrize("size", ["tiny", "pinned", "direct"])
def test_state_is_the_slots_by_id(sph, size, record):  # noqa: F811
    sc = {"tiny": lambda: scenes.tiny(seed=1, n=(2, 2, 2)),
          "pinned": lambda: scenes.dam_break(seed=1, grab=True),
          "direct": lambda: scenes.coupled(seed=0, n_fluid=30_000, cols=(40, 30), tank=(0.4, 0.3, 0.5), n_substeps=10,
                                           probe_r=0.04, soft_n=6)}[size]()
    sim = sph.Simulation(sc, flags=sc.params["flags"] | (sph.FLAG_RECORD if record else 0))
    sim.step(3)
    st = sim.state(record=record)
    n = sim.n
    raw = np.asarray(sim.checkpoint()).view(np.uint8).reshape(-1)
    x = raw[40:40 + 16 * n].view(np.float32).reshape(n, 4)      # behind the header: positions, then
    v = raw[40 + 16 * n:40 + 32 * n].view(np.float32).reshape(n, 4)   # velocities and ids, by slot
    ids = v[:, 3].copy().view(np.int32)
    np.testing.assert_array_equal(np.sort(ids), np.arange(n))
    np.testing.assert_array_equal(st["x"][ids], x[:, :3])
    np.testing.assert_array_equal(st["v"][ids], v[:, :3])
    assert np.all(st["rho"] > 0.0)
    if record:
        assert st["nnbr"].max() > 0 and np.isfinite(st["acc"]).all()
    again = sim.state()
    np.testing.assert_array_equal(again["rho"], st["rho"])
    sim.close()

"""Lists too short for most particles in a scene large enough for the passes that small scenes do
not take: four lanes per rigid particle beside one thread per particle, sixteen lanes with the
low-latency flag (those that overflow walk beside those that do not), the force pass's two shares
to a lane, the volume variant.  Against the oracle under the parity bar, and alone against a batch
of one bit for bit."""
import numpy as np
import pytest

from paper_2511_15908_gb300 import scenes

from test_gpu_parity import check_one_substep, sph  # noqa: F401

pytestmark = pytest.mark.gpu

SLOTS = 24                              # a fluid particle has some 34 neighbours, a rigid one 226


def _scene():
    return scenes.with_velocity_noise(
        scenes.coupled(seed=0, n_fluid=60_000, cols=(60, 40), tank=(0.6, 0.4, 0.4), n_substeps=10, probe_r=0.04,
                       soft_n=8), seed=4, sigma=0.2)


@pytest.mark.parametrize("flag", ["", "FLAG_LOW_LATENCY", "FLAG_VOLUME_BOUNDARY"])
def test_against_the_oracle(sph, flag):  # noqa: F811
    sc = _scene()
    assert sc.n_total > 60_000
    if flag:
        sc.params["flags"] |= getattr(scenes, flag, None) or getattr(sph, flag)
    check_one_substep(sph, sc, mode=1, max_neighbours=SLOTS)


def test_alone_equals_a_batch_of_one(sph):  # noqa: F811
    sims = [sph.Simulation(_scene(), max_neighbours=slots) for slots in (SLOTS, SLOTS, 0)]
    batch = sph.Batch(sims[:1])
    batch.configure(0)
    batch.step(3)
    batch.sync()
    for s in sims[1:]:
        s.step(3)
    states = [s.state() for s in sims]
    for other in states[1:]:            # the short lists alone, and lists that hold everything
        for key in ("x", "v", "rho"):
            np.testing.assert_array_equal(states[0][key], other[key])
    for k in range(len(sims[0].scene.bodies)):
        np.testing.assert_array_equal(sims[0].body_wrench(k), sims[1].body_wrench(k))
    batch.close()
    for s in sims:
        s.close()

"""The neighbour search and the density sum over its lists at the sizes where they can go
wrong: scenes of a few particles, counts around the tiles' edges, rows of candidates longer
than a chunk, lists exactly full or too short, bodies sampled far more finely than the fluid.
Every case against the oracle under the parity bar (counts exact), and the two ways of walking
(one thread per particle, as a batch does; cooperating lanes, as a small scene does) against
each other bit for bit."""
import numpy as np
import pytest

from paper_2511_15908_gb300 import scenes

from test_gpu_parity import check_one_substep, sph  # noqa: F401

pytestmark = pytest.mark.gpu


def _cloud(n, seed=0, spacing=0.02, body=0.0):
    """n fluid particles at random in a small box, optionally a rigid cube sampled at `body`."""
    rng = np.random.default_rng(seed)
    side = max(1, int(np.ceil(n ** (1.0 / 3.0))))
    x = scenes._lattice((side, side, side), spacing, (0.0, 0.0, 0.0))[:n]
    x = (x + rng.uniform(-0.3, 0.3, x.shape) * spacing).astype(np.float32)
    v = rng.normal(0.0, 0.2, x.shape).astype(np.float32)
    bodies = []
    if body:
        loc, _ = scenes.solid_box((2.5 * spacing,) * 3, body)
        pose = np.array([side * spacing + 0.5 * spacing, 0.5 * side * spacing, 0.5 * side * spacing, 1, 0, 0, 0], np.float32)
        bodies.append(scenes.Body(scenes.KIND_RIGID, loc, body, mass=0.01, inertia=np.eye(3, dtype=np.float32) * 1e-5,
                                  pose=pose, vel=rng.normal(0.0, 0.1, 6).astype(np.float32)))
        floor = scenes._lattice((side + 2, side + 2, 1), spacing, (-spacing, -spacing, -1.2 * spacing)).astype(np.float32)
        bodies.append(scenes.Body(scenes.KIND_STATIC, floor, spacing))
    hi = (side + 5) * spacing
    params = scenes.make_params(spacing, 1e-3, (-3 * spacing,) * 3, (hi,) * 3)
    return scenes.Scene("cloud", params, x, v, spacing, bodies)


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 33, 255, 257, 513])
def test_particle_counts_around_the_tiles(sph, n):  # noqa: F811
    check_one_substep(sph, _cloud(n, seed=n), mode=0)


@pytest.mark.parametrize("body,slots", [(0.01, 0), (0.01, 32), (0.01, 36), (0.01, 4), (0.005, 0), (0.005, 2400)])
def test_finely_sampled_body_and_list_capacity(sph, body, slots):  # noqa: F811
    # at a quarter of the spacing a body particle has some 1700 neighbours: rows of more than a
    # hundred candidates, lists that overflow (288 slots) or hold them all
    check_one_substep(sph, _cloud(300, seed=7, body=body), mode=0, max_neighbours=slots)


@pytest.mark.parametrize("flags", [0, scenes.FLAG_VOLUME_BOUNDARY])
@pytest.mark.parametrize("slots", [0, 24])
def test_cooperating_lanes_equal_one_thread(sph, flags, slots):  # noqa: F811
    scs = [_cloud(300, seed=3, body=0.01), scenes.with_velocity_noise(scenes.dam_break(seed=4, grab=True), seed=5)]
    for sc in scs:
        sc.params["flags"] |= flags
    alone = [sph.Simulation(sc, max_neighbours=slots) for sc in scs]
    batched = [sph.Simulation(sc, max_neighbours=slots) for sc in scs]
    batch = sph.Batch(batched)
    batch.configure(0)
    for s in alone:
        s.step(5)
    batch.step(5)
    batch.sync()
    for a, b in zip(alone, batched):
        sa, sb = a.state(), b.state()
        for key in ("x", "v", "rho"):
            np.testing.assert_array_equal(sa[key], sb[key])
        for k in range(len(a.scene.bodies)):
            np.testing.assert_array_equal(a.body_wrench(k), b.body_wrench(k))
    batch.close()
    for s in alone + batched:
        s.close()

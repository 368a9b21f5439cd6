"""Several scenes stepped at once on their own streams, where lanes that share a particle's work
cost the other scenes theirs: scenes of 30,000 to 60,000 particles take together about what a batch
of them takes, whose walk has one thread per particle.  And the walks on both sides of the sizes
where the rule changes, alone against a batch bit for bit."""
import numpy as np
import pytest
import torch

from paper_2511_15908_gb300 import scenes

from test_gpu_parity import sph  # noqa: F401

pytestmark = pytest.mark.gpu


def _time(first, streams, run):
    """Device time of run() over the streams, best of five, in ms."""
    best = float("inf")
    for _ in range(5):
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(first)
        for s in streams:
            s.wait_event(a)
        run()
        for s in streams:
            e = torch.cuda.Event()
            e.record(s)
            first.wait_event(e)
        b.record(first)
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_scenes_side_by_side_cost_about_their_batch(sph):  # noqa: F811
    scs = scenes.batched(seed=5, n_scenes=8, lo=8_000, hi=20_000, n_substeps=400)
    assert all(30_000 < sc.n_total <= 60_000 for sc in scs)
    sims = [sph.Simulation(sc) for sc in scs]
    batched = [sph.Simulation(sc) for sc in scs]
    batch = sph.Batch(batched)
    batch.configure(0)
    for s in sims:
        s.step(10)
    batch.step(10)
    batch.sync()

    def alone():
        for _ in range(16):
            for s in sims:
                s.step(1)

    t_batch = _time(batch.stream, [], lambda: batch.step(16))
    t_alone = _time(sims[0].stream, [s.stream for s in sims[1:]], alone)
    print(f"8 scenes, 16 substeps: side by side {t_alone:.2f} ms, batch {t_batch:.2f} ms")
    # each scene's own launches and their gaps beside the batch's: up to half as much again
    assert t_alone <= 1.5 * t_batch
    batch.close()
    for s in sims + batched:
        s.close()


def _with_body(n, seed):
    """n particles in all: jittered fluid, a rigid cube at half its spacing and a floor."""
    s = 0.02
    rng = np.random.default_rng(seed)
    loc, _ = scenes.solid_box((6 * s,) * 3, s / 2)
    side = int(np.ceil((n / 1.0) ** (1.0 / 3.0)))
    floor = scenes._lattice((side, side, 1), s, (0.0, 0.0, -1.2 * s)).astype(np.float32)
    nf = n - len(loc) - len(floor)
    x = scenes._lattice((side, side, side), s, (0.0,) * 3)[:nf]
    x = (x + rng.uniform(-0.3, 0.3, x.shape) * s).astype(np.float32)
    v = rng.normal(0.0, 0.2, x.shape).astype(np.float32)
    top = float(x[:, 2].max())
    pose = np.array([0.4 * side * s, 0.5 * side * s, top + 3.2 * s, 1, 0, 0, 0], np.float32)
    bodies = [scenes.Body(scenes.KIND_RIGID, loc, s / 2, mass=1.0, inertia=np.eye(3, dtype=np.float32) * 1e-3, pose=pose,
                          vel=rng.normal(0.0, 0.1, 6).astype(np.float32)),
              scenes.Body(scenes.KIND_STATIC, floor, s)]
    hi = (side + 3) * s
    params = scenes.make_params(s, 1e-3, (-3 * s,) * 3, (hi, hi, top + 12 * s))
    sc = scenes.Scene("with a body", params, x, v, s, bodies)
    assert sc.n_total == n
    return sc


@pytest.mark.parametrize("slots", [0, 24])
@pytest.mark.parametrize("n", [20_000, 20_001, 30_000, 30_001, 60_000, 60_001])
def test_sizes_where_the_walk_changes(sph, n, slots):  # noqa: F811
    sc = _with_body(n, seed=n)
    alone, batched = (sph.Simulation(sc, max_neighbours=slots, flags=sc.params["flags"] | sph.FLAG_RECORD) for _ in range(2))
    batch = sph.Batch([batched])
    batch.configure(0)
    alone.step(3)
    batch.step(3)
    batch.sync()
    a, b = alone.state(record=True), batched.state(record=True)
    assert a["nnbr"].max() > 100
    for key in ("x", "v", "rho", "nnbr", "acc"):
        np.testing.assert_array_equal(a[key], b[key])
    np.testing.assert_array_equal(alone.body_wrench(0), batched.body_wrench(0))
    batch.close()
    alone.close()
    batched.close()

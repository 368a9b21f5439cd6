"""Particles outside the grid: clamped into its border cells, they keep all their neighbours.
Blocks of fluid that cross each of the six faces and a corner, reaching four to five cells out,
in every way the search walks: cooperating lanes (a small scene alone), one thread per particle
(the same in a batch, and a scene above 60,000 particles), the low-latency walk, with lists that
hold every neighbour and lists that overflow.  Every case against the oracle under the parity bar
(neighbour counts exact; all pairs for the small scene), and alone against batched bit for bit."""
import numpy as np
import pytest

from paper_2511_15908_gb300 import scenes

import test_gpu_parity
from test_gpu_parity import sph  # noqa: F401

pytestmark = pytest.mark.gpu

S = 0.02                                           # fluid spacing = h; a cell is 1.001 h


def _crossing(n, out, inside, filled=False, seed=0):
    """Jittered blocks through the faces of a box of n^3 spacings: `out` layers beyond each face
    and `inside` within; 4^3 particles beyond the low corner; optionally the box filled."""
    rng = np.random.default_rng(seed)
    mid = (n // 2 - 2) * S
    blocks = []
    for axis in range(3):
        dims = [4, 4, 4]
        dims[axis] = out + inside
        for lo in (-out * S, (n - inside) * S):
            origin = [mid, mid, mid]
            origin[axis] = lo
            blocks.append(scenes._lattice(dims, S, origin))
    blocks.append(scenes._lattice((4, 4, 4), S, (-5.0 * S,) * 3))
    if filled:
        blocks.append(scenes._lattice((n, n, n), S, (0.0,) * 3))
    x = np.concatenate(blocks)
    x = (x + rng.uniform(-0.3, 0.3, x.shape) * S).astype(np.float32)
    v = rng.normal(0.0, 0.2, x.shape).astype(np.float32)
    return scenes.Scene("crossing", scenes.make_params(S, 1e-3, (0.0,) * 3, (n * S,) * 3), x, v, S, [])


def _reporting(sph, batched):  # noqa: F811
    """Simulation whose step takes the out-of-domain report, alone or in a batch of its own."""
    class Sim(sph.Simulation):
        def step(self, n=1):
            if batched:
                b = sph.Batch([self])
                b.configure(0)
                b.step(n)
                b.sync()
                b.close()
            else:
                super().step(n)
            with pytest.raises(sph.SphError) as e:
                self.sync()
            assert e.value.status == sph.ERR_DOMAIN
    return Sim


def _check(sph, monkeypatch, sc, batched, mode, slots):  # noqa: F811
    monkeypatch.setattr(sph, "Simulation", _reporting(sph, batched))
    return test_gpu_parity.check_one_substep(sph, sc, mode=mode, max_neighbours=slots)[0]


@pytest.mark.parametrize("slots", [0, 8])
def test_small_scene_alone_and_batched(sph, monkeypatch, slots):  # noqa: F811
    sc = _crossing(12, 5, 3)
    alone = _check(sph, monkeypatch, sc, False, 0, slots)
    monkeypatch.undo()
    batched = _check(sph, monkeypatch, sc, True, 0, slots)
    for key in ("x", "v", "rho", "nnbr", "acc"):
        np.testing.assert_array_equal(alone[key], batched[key])


def test_low_latency_walk(sph, monkeypatch):  # noqa: F811
    sc = _crossing(12, 5, 3)
    sc.params["flags"] |= sph.FLAG_LOW_LATENCY
    _check(sph, monkeypatch, sc, False, 0, 0)


@pytest.mark.parametrize("flags", [0, "FLAG_LOW_LATENCY"])
def test_scene_above_60000_particles(sph, monkeypatch, flags):  # noqa: F811
    sc = _crossing(40, 5, 0, filled=True)
    assert sc.n_total > 60_000
    sc.params["flags"] |= getattr(sph, flags) if flags else 0
    _check(sph, monkeypatch, sc, False, 1, 0)

"""The network's batch pass at the edges of its 128-row tiles, of the 16-row loss partials and of
the batch contraction's 64-row chunks: outputs, loss and every gradient against the oracle, which
rounds to BF16 at the same points, within the bounds of the surrogate's parity tests."""
import numpy as np
import pytest

from oracle import mlp as omlp

from test_gpu_surrogate import _data, sph  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 15, 16, 17, 64, 65, 127, 128, 129, 513])
def test_outputs_and_gradients_at_tile_edges(sph, B):  # noqa: F811
    import torch
    params, norm, X, T = _data(B, seed=B)
    m = sph.Surrogate(max_batch=max(B, 2))
    m.set_params(params, norm)
    x, t = torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda")
    y = m.forward(x)
    m.sync()
    ref = omlp.forward(params, norm, X, bf=True)
    got = y.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= 2.0 ** -6 * np.abs(ref) + 2.0 ** -8 * np.sqrt(np.mean(ref * ref)))
    g, loss = m.gradients(x, t)
    lref, gref = omlp.grad(params, norm, X, T, bf=True)
    # the loss follows the outputs: one BF16 unit of an output's spread, squared error's slope 2
    assert loss == pytest.approx(lref, rel=2.0 ** -6)
    rms = np.sqrt(np.mean(gref * gref))
    assert np.all(np.abs(g - gref) <= 2.0 ** -5 * np.abs(gref) + 2.0 ** -6 * rms)
    m.close()

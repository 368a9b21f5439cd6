"""The force pass, two partners at a time: odd and even partner counts (down to none), particle
counts around its 128-particle blocks, full and overflowing lists, its three variants.  Every
case against the oracle under the parity bar."""
import pytest

from paper_2511_15908_gb300 import scenes

from test_gpu_parity import check_one_substep, sph  # noqa: F401
from test_gpu_walk import _cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["mass", "volume", "low_latency"])
@pytest.mark.parametrize("n,slots", [(1, 0), (2, 0), (3, 0), (5, 0), (127, 0), (128, 0), (129, 0), (300, 24)])
def test_partner_pairs_and_block_edges(sph, n, slots, variant):  # noqa: F811
    sc = _cloud(n, seed=40 + n, body=0.0 if n < 128 else 0.01)
    sc.params["flags"] |= {"mass": 0, "volume": scenes.FLAG_VOLUME_BOUNDARY, "low_latency": sph.FLAG_LOW_LATENCY}[variant]
    check_one_substep(sph, sc, mode=0, max_neighbours=slots)

"""Context tokens and the attention to them: observation widths that do not fill a step of the projection, both of its row-tile
heights, contexts of one 16-key tile (nothing for the second warp of a pair), of an odd number of them and of 256, one and
several query tiles, more tiles than warp pairs, verification groups whose tiles go to several blocks (three and two)."""
import pytest

from tests import helpers as hp
from tests.test_gpu_round import _round_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Tc,Do,heads,K", [(1, 5, 16, 20, 2, 2), (2, 50, 48, 33, 4, 2), (3, 64, 256, 64, 1, 2), (5, 17, 256, 31, 2, 2),
                                               (2, 50, 96, 20, 2, 6), (1, 64, 256, 20, 2, 3)])
def test_round_context_edges(B, H, Tc, Do, heads, K):
    wl = dict(H=H, A=3, To=Tc, Do=Do, T=100, precision=1, gamma=0.05,
              base=dict(arch="dit", layers=1, d=256 if heads > 1 else 128, heads=2 * heads),
              draft=dict(arch="dit", layers=1, d=128, heads=heads))
    # tolerances of the bf16 transformer rounds: bf16 operands, fp32 accumulation and softmax sums
    _round_parity(wl, B, K, hp.accept_t(), 31, 2e-2, 3e-3, [99, 60, 40, 12, 2][:B])

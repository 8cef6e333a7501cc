"""Cluster kernel as drafter and verifier against the oracle: every head width at both model widths, folded and unfolded
cross-attention (too many memory tokens, one head), resident and streamed weights, a ring that wraps inside a layer, and the
ends of what fits: one token, an odd number of them, one action dimension, 64."""
import pytest

from tests import helpers as hp
from tests.test_gpu_round import _round_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,layers,H,A,To", [
    (128, 4, 1, 16, 16, 2), (128, 2, 3, 15, 3, 3), (128, 1, 5, 9, 2, 1), (256, 8, 1, 16, 7, 1), (256, 8, 2, 5, 10, 3),
    (256, 4, 4, 4, 64, 3), (256, 2, 2, 1, 1, 2)])
def test_cluster_kernel_head_widths_and_ends(d, heads, layers, H, A, To):
    wl = hp.small_xfmr_workload(1, d=d, heads=heads, layers=layers, dd=d, dlayers=layers, H=H, A=A, To=To, Do=9)
    # tolerances of the bf16 transformer rounds: bf16 operands, fp32 accumulation, at most 8 blocks
    _round_parity(wl, 2, 3, hp.accept_t(), 21, 2e-2, 3e-3, [99, 40], drafter=2, verifier=2)

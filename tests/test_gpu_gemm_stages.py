"""Tensor-core GEMM: reductions whose number of 64-wide k-blocks is odd, or smaller than the pipeline, on the tile widths that
put two k-blocks into a stage (32 and 64) and on those that do not."""
import numpy as np
import pytest

from tests import helpers as hp
from tests.test_gpu_kernels import _gemm_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [64, 128, 192, 576, 704, 1344])
@pytest.mark.parametrize("M,N", [(130, 32), (130, 96), (2300, 320), (6000, 384)])
def test_gemm_odd_and_short_reductions(M, N, K):
    smp, *_ = hp.setup(hp.small_xfmr_workload(1), max_B=1, max_K=1)
    rng = np.random.default_rng(K + N)
    for epi in (0, 3):
        _gemm_case(smp, M, N, K, epi, rng)
    smp.close()


def test_fused_attention_gives_a_row_the_same_bits_whichever_lane_issues():
    """d = 256: four 192-wide tiles per 128 rows.  74 row tiles are two tiles for each of 148 CTAs (elected lane), one more row tile is past
    that (lane 0); a single row tile is far below."""
    import torch
    smp, *_ = hp.setup(hp.small_xfmr_workload(1), max_B=1, max_K=1)
    g = torch.Generator(device="cuda").manual_seed(1)
    d, M = 256, 74 * 128 + 16
    A = torch.randn(M, d, device="cuda", generator=g).to(torch.bfloat16)
    W = (torch.randn(3 * d, d, device="cuda", generator=g) / 16).to(torch.bfloat16)
    b = torch.randn(3 * d, device="cuda", generator=g)
    outs = {}
    for m in (128, M - 16, M):
        outs[m] = torch.full((m, d), float("nan"), device="cuda", dtype=torch.bfloat16)
        smp.gemm(A[:m].contiguous(), W, b, m, 3 * d, d, 4, outs[m])
    assert torch.isfinite(outs[M].float()).all()
    for m in (128, M - 16):
        assert torch.equal(outs[m], outs[M][:m]), m
    smp.close()

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

"""MLP kernels at the sizes where their split can go wrong: odd widths (rows that are not 16-byte aligned), more columns
than one pass of a CTA, one to eight CTAs per cluster, one and four latents per cluster with ragged last groups."""
import numpy as np
import pytest
import torch

from paper_2512_15773_b200 import binding, inputs
from tests import helpers as hp
from tests.test_gpu_round import _round_parity

pytestmark = pytest.mark.gpu


def _workload(width, layers, A, dwidth):
    return dict(H=5, A=A, To=1, Do=7, T=100, precision=0, gamma=0.05, base=dict(arch="mlp", layers=layers, width=width),
                draft=dict(arch="mlp", layers=1, width=dwidth))


@pytest.mark.parametrize("width,layers,A", [(63, 2, 3), (256, 3, 4), (300, 1, 5), (1030, 2, 1)])
@pytest.mark.parametrize("N", [1, 18, 39, 150])
def test_mlp_forward_against_oracle(width, layers, A, N):
    wl = dict(_workload(width, layers, A, 64), gamma=1.0)
    smp, S, base, _ = hp.setup(wl, max_B=N, max_K=1)
    rng = np.random.default_rng(N)
    x = rng.normal(size=(N, wl["H"], A)).astype(np.float32)
    tau = rng.integers(0, 100, size=N).astype(np.int32)
    obs = inputs.make_obs(5, N, wl["To"], wl["Do"])
    dx = torch.tensor(x, device="cuda"); out = torch.full_like(dx, float("nan"))
    smp.denoise(binding.BASE, dx, tau, torch.tensor(obs, dtype=torch.float32, device="cuda"), N, out)
    got = out.cpu().numpy()
    for n in range(0, N, max(1, N // 9)):
        # fp32 sums of at most 1030 terms: n 2^-24 of the sum of magnitudes, below 1e-4 of the largest output
        assert hp.max_rel(got[n], base(x[n].astype(np.float64), int(tau[n]), obs[n])) < 1e-4, n
    # an output does not depend on how many latents share the launch
    one = torch.full_like(dx[:1], float("nan"))
    smp.denoise(binding.BASE, dx[N - 1:].contiguous(), tau[N - 1:], torch.tensor(obs[N - 1:], dtype=torch.float32, device="cuda"), 1, one)
    assert torch.equal(one[0], out[N - 1])
    assert smp.check_guards() > 0
    smp.close()


@pytest.mark.parametrize("B,dwidth", [(2, 30), (2, 1030), (41, 64)])
def test_mlp_rollout_round_against_oracle(B, dwidth):
    wl = _workload(64, 2, 3, dwidth)
    t0s = [99, 1, 0, 3, 50, 2][:B] + [40] * (B - 6)
    _round_parity(wl, B, 5, hp.accept_t(), 9, 1e-4, 2e-5, t0s)

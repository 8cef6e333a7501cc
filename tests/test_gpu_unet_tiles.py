"""Conv UNet at the sizes where its tiles can go wrong: horizons that do not divide the 128-row tile (12, 20, 24, 64), group
widths on every GroupNorm kernel (channels not in fours, one group over everything), one level, batch sizes from one
candidate (reductions split up to eight ways) to several waves of tiles."""
import numpy as np
import pytest
import torch

from oracle import ddpm, nets
from paper_2512_15773_b200 import binding, inputs
from tests import helpers as hp
from tests.test_gpu_round import _round_parity

pytestmark = pytest.mark.gpu

CASES = [  # H, A, levels, channels, groups, obs width
    (12, 3, 3, 128, 8, 7), (20, 5, 3, 128, 16, 24), (24, 1, 2, 256, 8, 33), (64, 2, 2, 128, 4, 12), (8, 7, 1, 128, 64, 5),
    (16, 10, 3, 128, 1, 24), (16, 3, 2, 384, 8, 7)]      # (384 channels in 8 groups: a lane's values are of several channel quads)


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("N", [1, 11, 150])
def test_unet_denoiser_tiles_and_groups(case, N):
    H, A, levels, ch, groups, Do = case
    for precision, tol in ((1, 2e-2), (0, 1e-4)):
        if precision == 0 and N > 11:
            continue
        wl = dict(H=H, A=A, To=2, Do=Do, T=100, precision=precision, gamma=1.0,
                  base=dict(arch="unet", layers=levels, d=ch, heads=groups, temb=32))
        cfg = binding.make_config(H, A, 2, Do, wl["base"], dict(arch="gauss"), max_B=N, max_K=1, precision=precision)
        params = inputs.make_net(1, wl, "base")
        smp = binding.Sampler(cfg)
        smp.load_weights(binding.BASE, params)
        base = nets.make_denoiser(params, ddpm.Schedule(100, 1e-4, 0.02))
        rng = np.random.default_rng(N)
        x = rng.normal(size=(N, H, A)).astype(np.float32)
        tau = rng.integers(0, 100, size=N).astype(np.int32)
        obs = inputs.make_obs(5, N, 2, Do)
        dx = torch.tensor(x, device="cuda"); dobs = torch.tensor(obs, dtype=torch.float32, device="cuda")
        outs = []
        for _ in range(2):      # a second call: the padding rows of every buffer are still zero, the same bits come out
            out = torch.full_like(dx, float("nan"))
            smp.denoise(binding.BASE, dx, tau, dobs, N, out)
            outs.append(out.cpu().numpy())
        assert np.array_equal(outs[0], outs[1])
        for n in sorted({0, N // 2, N - 1}):
            err = hp.max_rel(outs[0][n], base(x[n].astype(np.float64), int(tau[n]), obs[n]))
            assert err < tol, (precision, n, err)
        assert smp.check_guards() > 0
        smp.close()


# One warp per group, eight groups a block: from 32 groups per SM on (4736), four channels a group at least and at most 128 quads of values.
# Two and three parts of a reduction, four to six, and none with every lane's registers full and a ragged last block (4740 groups).
@pytest.mark.parametrize("case,N", [((8, 3, 2, 128, 32, 7), 151), ((4, 5, 2, 256, 64, 12), 75), ((16, 2, 1, 128, 4, 5), 1185), ((8, 3, 1, 384, 8, 7), 593)])
def test_unet_denoiser_with_a_warp_per_group(case, N):
    test_unet_denoiser_tiles_and_groups(case, N)


# Four warps per group: the last launch whose GroupNorms fetch everything early (8 groups per SM, 1184) and the first that does not; two well past it.
@pytest.mark.parametrize("N", [148, 149, 258, 259])
def test_unet_denoiser_on_both_sides_of_the_early_fetch(N):
    test_unet_denoiser_tiles_and_groups((16, 2, 1, 128, 8, 5), N)


def test_unet_round_with_a_warp_per_group_and_few_live_candidates():
    """300 slots x 4 candidates x 4 groups; timesteps near the end leave 837 candidates alive, 3348 groups, the last block half full.
    A rejected draft's reflection multiplies the error of mu^ - mu (3e-7) by 2 sigma |xi| / |mu^ - mu|: 70 at most for this drafter, so 2e-5
    of the 6e-5 that the committed latent may be off.  (Frozen-target drafts have 490 here, beyond it.)"""
    wl = dict(H=4, A=3, To=1, Do=6, T=100, precision=0, gamma=0.05, base=dict(arch="unet", layers=1, d=128, heads=4, temb=8),
              draft=dict(arch="mlp", layers=1, width=64))
    _round_parity(wl, 300, 3, hp.accept_t(), 13, 1e-4, 2e-5, [i % 5 for i in range(299)] + [0])


def test_mish_behind_the_group_norm_keeps_fp32_accuracy():
    """Every weight but the last norm's shift and a 0/1 output matrix is zero, so eps[l, a] is Mish of shift a, nothing else.
    Above 9.5 the nearest fp32 number to Mish(v) = v (1 - 2 / (n + 2)), n = e^v (e^v + 2), is v itself (2 / (n + 2) < 2^-25).
    Elsewhere 10 units of 2^-24: the exponential (1 ulp = 2 units, its weight in the result at most 1); a quotient t <= 0.4 taken
    from 1, so of weight t / (1 - t) <= 2/3, with 3 units in its parts and 2 ulp of its own; three roundings behind it."""
    H, A, ch = 2, 64, 128
    wl = dict(H=H, A=A, To=1, Do=1, T=100, precision=0, gamma=1.0, base=dict(arch="unet", layers=1, d=ch, heads=8, temb=4))
    smp = binding.Sampler(binding.make_config(H, A, 1, 1, wl["base"], dict(arch="gauss"), max_B=1, max_K=1, precision=0))
    p = inputs.make_net(1, wl, "base")
    zero = lambda v: np.zeros_like(np.asarray(v, dtype=np.float64))
    p = {k: ([{n: zero(w) for n, w in R.items()} for R in v] if k == "blocks" else zero(v) if isinstance(v, np.ndarray) else v)
         for k, v in p.items()}
    p["W_out"][:A, :A] = np.eye(A)
    x = torch.zeros(1, H, A, device="cuda"); obs = torch.zeros(1, 1, 1, device="cuda"); out = torch.zeros_like(x)
    values = np.linspace(-25.0, 21.0, 24 * A).astype(np.float32).reshape(24, A)
    got = []
    for row in values:
        p["beh"][:A] = row
        smp.load_weights(binding.BASE, p)
        smp.denoise(binding.BASE, x, np.array([7], np.int32), obs, 1, out)
        got.append(out[0, 1].cpu().numpy())
    smp.close()
    v, got = values.reshape(-1).astype(np.float64), np.concatenate(got).astype(np.float64)
    n = np.exp(v) * (np.exp(v) + 2.0)
    err = np.abs(got - v * n / (n + 2.0)) / np.abs(v * n / (n + 2.0))
    assert np.max(err) < 10 * 2.0 ** -24
    assert np.array_equal(got[v >= 9.5], v[v >= 9.5])

"""Conv UNet at the sizes where its tiles can go wrong: horizons that do not divide the 128-row tile (12, 20, 24, 64), group
widths on every GroupNorm kernel (channels not in fours, one group over everything), one level, batch sizes from one
candidate (reductions split up to eight ways) to several waves of tiles."""
import numpy as np
import pytest
import torch

from oracle import ddpm, nets
from paper_2512_15773_b200 import binding, inputs
from tests import helpers as hp

pytestmark = pytest.mark.gpu

CASES = [  # H, A, levels, channels, groups, obs width
    (12, 3, 3, 128, 8, 7), (20, 5, 3, 128, 16, 24), (24, 1, 2, 256, 8, 33), (64, 2, 2, 128, 4, 12), (8, 7, 1, 128, 64, 5),
    (16, 10, 3, 128, 1, 24)]


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

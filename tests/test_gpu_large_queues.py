"""Queues so long that the per-request set-up has more row blocks than the second dimension of a grid may have (65535):
observation tokens of an adaLN transformer (64 rows a block), FiLM terms of a conv UNet (8 requests a block)."""
import numpy as np
import pytest
import torch

from oracle import ddpm, nets, spec
from paper_2512_15773_b200 import binding, inputs
from tests import helpers as hp

pytestmark = pytest.mark.gpu

T = 2


@pytest.mark.parametrize("base,N,To,precision,tol", [
    (dict(arch="dit", layers=1, d=128, heads=4), 65535 * 64 // 256 + 2, 256, 1, 2e-2),
    (dict(arch="unet", layers=1, d=128, heads=8, temb=4), 65535 * 8 + 9, 1, 0, 1e-4)], ids=["tokens", "film"])
def test_a_queue_beyond_a_grids_second_dimension(base, N, To, precision, tol):
    slots, seed = 4096, 5
    wl = dict(H=1, A=1, To=To, Do=1, T=T, precision=precision, gamma=1.0, base=base, draft=dict(arch="frozen"))
    cfg = binding.make_config(1, 1, To, 1, base, wl["draft"], T=T, max_B=slots, max_K=1, precision=precision)
    params = inputs.make_net(1, wl, "base")
    smp = binding.Sampler(cfg)
    smp.load_weights(binding.BASE, params)
    obs = np.random.default_rng(3).normal(size=(N, To, 1)).astype(np.float32)
    out = torch.full((N, 1, 1), float("nan"), device="cuda")
    smp.serve(torch.tensor(obs, device="cuda"), N, slots, 0, hp.accept_t(), seed, out)
    got = out.cpu().numpy()
    assert np.isfinite(got).all()
    S = ddpm.Schedule(T, 1e-4, 0.02)
    net = nets.make_denoiser(params, S)
    for i in (0, N // 2, N - 2, N - 1):      # plain DDPM: no decision that could turn
        want = spec.sample_vanilla(S, net, spec.PhiloxNoise(seed), i, obs[i], (1, 1))
        # the tolerance of a forward, times the weight of its output in the latent (below 1 at these two steps), on values of order 1
        assert np.max(np.abs(got[i] - want)) < tol * max(1.0, np.max(np.abs(want))), i
    smp.close()

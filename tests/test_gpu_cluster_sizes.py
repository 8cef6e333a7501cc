"""Clusters of 4 CTAs, which take over where there are more environments than clusters of 8, give the bits of clusters of 8: every sum
over the CTAs of a cluster has the same tree."""
import pytest
import torch

from paper_2512_15773_b200 import inputs
from tests import helpers as hp

pytestmark = pytest.mark.gpu


# d = 256: streamed weights, a head per CTA or two CTAs per head; d = 128: resident weights; short sequence, ragged latent; no observation
@pytest.mark.parametrize("d, heads, layers, H, A, To", [(256, 4, 4, 16, 10, 2), (256, 2, 1, 16, 3, 3), (128, 4, 2, 16, 2, 2), (128, 4, 3, 7, 5, 1),
                                                        (128, 2, 1, 9, 28, 0)])
def test_batches_in_clusters_of_four_equal_single_environments(d, heads, layers, H, A, To):
    """24 environments (two waves of clusters of 8, one of 4) against a queue through six slots (one wave of 8)."""
    wl = hp.small_xfmr_workload(1, d=128, heads=4, layers=1, dd=d, dlayers=layers, H=H, A=A, To=To, Do=12, gamma=0.05)
    wl["draft"]["heads"] = heads
    B, K = 24, 5
    obs = torch.tensor(inputs.make_obs(4, B, To, 12), dtype=torch.float32, device="cuda")
    out = []
    for slots in (B, 6):
        smp, *_ = hp.setup(wl, max_B=slots, max_K=K, drafter=2, verifier=1)
        o = torch.full((B, H, A), float("nan"), device="cuda")
        smp.serve(obs, B, slots, K, hp.accept_t(), 7, o)
        assert smp.check_guards() >= 20
        out.append(o)
        smp.close()
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])


def test_verification_in_clusters_of_four_equals_clusters_of_eight():
    """4 environments x 6 candidates in one call against the same environments one by one."""
    wl = dict(inputs.WORKLOADS["pusht_xfmr"])
    wl["base"] = dict(wl["base"], layers=3)
    B, K = 4, 5
    obs = torch.tensor(inputs.make_obs(4, B, 2, 20), dtype=torch.float32, device="cuda")
    out = []
    for slots in (B, 1):
        smp, *_ = hp.setup(wl, max_B=slots, max_K=K, drafter=2, verifier=2)
        o = torch.full((B, 16, 2), float("nan"), device="cuda")
        smp.serve(obs, B, slots, K, hp.accept_t(), 7, o)
        out.append(o)
        smp.close()
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])

"""Clusters of 4 CTAs, which take over where there are more environments than clusters of 8, give the bits of clusters of 8: every sum
over the CTAs of a cluster has the same tree."""
import re

import pytest
import torch

from paper_2512_15773_b200 import inputs
from tests import helpers as hp

pytestmark = pytest.mark.gpu


def _sizes(call):
    """CTAs per cluster of the cluster kernels that a call launches; None where this process cannot record launches."""
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA], acc_events=True) as p:
        call()
        torch.cuda.synchronize()
    names = {e.name for e in p.events() if "tsdp::" in e.name}
    return {int(m.group(1)) for m in (re.search(r"drafter_cluster_kernel<\d+, \d+, (\d+)>", n) for n in names) if m} if names else None


def _chunks(wl, B, slots, K, verifier=1):
    """Chunks of B environments through `slots` slots, and the cluster sizes they were drafted (or verified) in."""
    smp, *_ = hp.setup(wl, max_B=slots, max_K=K, drafter=2, verifier=verifier)
    obs = torch.tensor(inputs.make_obs(4, B, wl["To"], wl["Do"]), dtype=torch.float32, device="cuda")
    out = torch.full((B, wl["H"], wl["A"]), float("nan"), device="cuda")
    sizes = _sizes(lambda: smp.serve(obs, B, slots, K, hp.accept_t(), 7, out))
    assert smp.check_guards() >= 20
    smp.close()
    assert torch.isfinite(out).all()
    return out, sizes


def _workload(d, heads, layers, H, A, To):
    wl = hp.small_xfmr_workload(1, d=128, heads=4, layers=1, dd=d, dlayers=layers, H=H, A=A, To=To, Do=12, gamma=0.05)
    wl["draft"]["heads"] = heads
    return wl


# streamed weights, d = 256: a head per CTA or two CTAs per head; d = 128, of which clusters of 4 hold one block at most: short sequence,
# ragged latent; resident weights: with and without observation tokens
@pytest.mark.parametrize("d, heads, layers, H, A, To", [(256, 4, 4, 16, 10, 2), (256, 2, 1, 16, 3, 3), (128, 4, 2, 16, 2, 2), (128, 4, 3, 7, 5, 1),
                                                        (128, 2, 1, 9, 28, 0), (128, 4, 1, 16, 2, 2)])
def test_batches_in_clusters_of_four_equal_single_environments(d, heads, layers, H, A, To):
    """24 environments (two waves of clusters of 8, one of 4) against a queue through six slots (one wave of 8)."""
    wl = _workload(d, heads, layers, H, A, To)
    four, eight = (_chunks(wl, 24, slots, 5) for slots in (24, 6))
    assert four[1] in ({4}, None) and eight[1] in ({8}, None)
    assert torch.equal(four[0], eight[0])


# A cluster goes from one environment to the next: ring, stage and buffer parities, tables and latents carry over, and from the first
# finished environment on some of them are skipped.  41: two waves of at most 33 clusters, 70: three.
@pytest.mark.parametrize("d, layers, B", [(256, 4, 41), (128, 1, 70), (128, 2, 70)])
def test_several_environments_per_cluster_of_four_equal_single_environments(d, layers, B):
    wl = _workload(d, 4, layers, 16, 7, 2)
    four, eight = (_chunks(wl, B, slots, 5) for slots in (B, 6))
    assert four[1] in ({4}, None) and eight[1] in ({8}, None)
    assert torch.equal(four[0], eight[0])


@pytest.mark.parametrize("switch", ["TSDP_NO_FOLD", "TSDP_NO_ASYNC_BCAST"])
@pytest.mark.parametrize("d, heads, layers, B", [(256, 4, 2, 41), (256, 2, 1, 24), (128, 4, 1, 24)])
def test_clusters_of_four_without_the_fold_and_with_cluster_barriers(monkeypatch, switch, d, heads, layers, B):
    """The cross-attention by its own products (two more exchanges a block), and exchanges by plain stores and barriers."""
    monkeypatch.setenv(switch, "1")
    wl = _workload(d, heads, layers, 16, 7, 2)
    four, eight = (_chunks(wl, B, slots, 4) for slots in (B, 6))
    assert four[1] in ({4}, None) and eight[1] in ({8}, None)
    assert torch.equal(four[0], eight[0])


@pytest.mark.parametrize("B", [4, 9])
def test_verification_in_clusters_of_four_equals_clusters_of_eight(B):
    """B environments x 6 candidates in one call (24: one wave of clusters of 4; 54: two) against the same environments one by one."""
    wl = dict(inputs.WORKLOADS["pusht_xfmr"])
    wl["base"] = dict(wl["base"], layers=3)
    many, one = (_chunks(wl, B, slots, 5, verifier=2) for slots in (B, 1))
    assert many[1] in ({8, 4}, None) and one[1] in ({8}, None)      # (the drafts of B environments run in clusters of 8)
    assert torch.equal(many[0], one[0])

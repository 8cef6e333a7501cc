"""The cluster kernel reads its own copy of a network's weights, one per cluster size: a context holds the copies that it can run, no others."""
import pytest
import torch

from paper_2512_15773_b200 import binding, inputs

pytestmark = pytest.mark.gpu

WL = dict(inputs.WORKLOADS["pusht_xfmr"], draft=dict(arch="xfmr", layers=8, d=256, heads=4))


def _loaded_bytes(which, **kw):
    smp = binding.Sampler(binding.make_config(WL["H"], WL["A"], WL["To"], WL["Do"], WL["base"], WL["draft"], T=WL["T"], max_B=2, max_K=2,
                                              precision=1, **kw))
    params = inputs.make_net(1, WL, "base" if which == binding.BASE else "draft")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    smp.load_weights(which, params)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    smp.close()
    return used


def test_only_the_cluster_forms_that_can_run_are_held():
    """8 blocks of d = 256 take 14.7 MB in clusters of 4 and 17.8 MB in clusters of 8 (allocations come in pieces of 2 MB)."""
    base = {v: _loaded_bytes(binding.BASE, verifier=v) for v in (0, 1, 2)}
    assert base[2] - base[0] > 10e6      # clusters of 4: only where the cluster kernel verifies whatever the number of candidates
    assert base[0] - base[1] > 13e6      # none: layer by layer
    draft = {v: _loaded_bytes(binding.DRAFT, drafter=v) for v in (0, 1, 2)}
    assert draft[0] - draft[1] > 25e6 and draft[0] == draft[2]

"""How a sampling call waits for its rounds, and what it leaves behind when it ends early."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2512_15773_b200 import binding, inputs
from tests import helpers as hp

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

BLOCKING = """
import ctypes, time
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0
assert cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0      # CU_CTX_SCHED_BLOCKING_SYNC
import torch
from paper_2512_15773_b200 import binding, inputs
wl = dict(inputs.WORKLOADS["serving_xfmr"])
cfg = binding.make_config(wl["H"], wl["A"], wl["To"], wl["Do"], wl["base"], dict(arch="frozen"), max_B=256, max_K=1)
smp = binding.Sampler(cfg)
smp.load_weights(binding.BASE, inputs.make_net(1, wl, "base"))
obs = torch.randn(256, wl["To"], wl["Do"], device="cuda")
out = torch.zeros(256, wl["H"], wl["A"], device="cuda")
call = lambda: smp.sample_chunk(obs, 256, 0, binding.AcceptT(0, 1.0, 1.0, 1), 1, out)
call()
wall, cpu = time.perf_counter(), time.thread_time()
call()
wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
print("wall %.4f s, of which the calling thread ran %.4f s" % (wall, cpu))
assert cpu < 0.5 * wall
"""


def test_a_process_that_asked_for_blocking_waits_does_not_spin():
    """100 rounds of a full batch (tens of milliseconds of GPU work): issuing them takes the host a few, the rest it sleeps."""
    r = subprocess.run([sys.executable, "-c", BLOCKING], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("call", ["chunk", "round"])
def test_a_call_after_one_that_failed_half_way_sees_nothing_of_it(call):
    """99 rounds of plain DDPM are in flight when the 100th is refused on the host.  The next call has other parameters; its result
    and, for a chunk, its number of rounds are those of a context that never failed."""
    wl = dict(inputs.WORKLOADS["serving_xfmr"], base=dict(arch="xfmr", layers=4, d=512, heads=8))
    B, K, D = 64, 4, wl["H"] * wl["A"]
    obs = torch.tensor(inputs.make_obs(3, B, wl["To"], wl["Do"]), dtype=torch.float32, device="cuda")
    outs = []
    for fail in (False, True):
        smp, *_ = hp.setup(wl, max_B=B, max_K=K)
        out = torch.zeros(B, wl["H"], wl["A"], device="cuda")
        smp.sample_chunk(obs, B, K, hp.accept_t(), 1, out)                  # graphs exist
        before = smp.stats()["rounds"]
        if fail:
            smp.arm_round_failure(100)
            with pytest.raises(binding.TsdpError) as e:
                smp.sample_chunk(obs, B, 0, hp.accept_t(), 2, out)
            assert e.value.status == 4                                      # TSDP_ERR_CUDA
            before += 99
        if call == "chunk":
            smp.sample_chunk(obs, B, K, hp.accept_t(), 9, out)
            outs.append((out.clone(), smp.stats()["rounds"] - before))
        else:
            x = torch.tensor(inputs.make_obs(7, B, wl["H"], wl["A"]), dtype=torch.float32, device="cuda").reshape(B, D)
            h_t = (torch.arange(B, dtype=torch.int32) + 20).numpy()
            smp.round(obs, B, K, hp.accept_t(), 9, x, h_t)
            outs.append((x.clone(), h_t.tolist()))
        smp.close()
    assert torch.equal(outs[0][0], outs[1][0])
    assert outs[0][1] == outs[1][1]

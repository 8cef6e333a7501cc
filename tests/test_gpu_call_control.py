"""How a sampling call waits for its rounds, and what it leaves behind when it ends early."""
import os
import subprocess
import sys

import pytest

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

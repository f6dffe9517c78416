"""How a waited call waits.  Behind work that the caller queued on its own
stream, in a process that asks for blocking synchronisation, it leaves the core
after its short poll (thread time well under the wall time), on device pointers
and on host arrays; and small host calls right after waited device calls on a
caller's stream, whose kernels may still be retiring, give the same results."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import workload as W
import paper_2608_14575_gb300 as H

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, sys, time
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0 and cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0     # CU_CTX_SCHED_BLOCKING_SYNC
import numpy as np, torch
import workload as W, paper_2608_14575_gb300 as H
dtype, kind = sys.argv[1:]
p = W.make_problem(Q=2000 if kind == "device" else 1, M=4, G=3, F=24, H1=128, H2=128, E=64, dtype=dtype, lam=0.4,
                   slo=2.0, seed=3, bias_std=0.05)
st = torch.cuda.Stream()
r = H.Router(p, stream=st.cuda_stream)
Q = p["Q"]
ins = [torch.from_numpy(p[k].view(np.int16) if p[k].dtype == np.uint16 else p[k]).cuda() for k in ("in_len", "out_len", "emb")]
out = [torch.empty(Q, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32)]
torch.cuda.synchronize()
call = (lambda: r.route_device(*ins, *out, slo=2.0, lam=0.4)) if kind == "device" else (lambda: r.route())
for _ in range(3):
    call()
with torch.cuda.stream(st):
    torch.cuda._sleep(400_000_000)
w, c = time.perf_counter(), time.thread_time()
call()
w, c = time.perf_counter() - w, time.thread_time() - c
r.close()
print(w, c)
"""


@pytest.mark.parametrize("kind", ["device", "host"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_a_call_behind_long_work_leaves_the_core(dtype, kind):
    H.build()
    o = subprocess.run([sys.executable, "-c", CHILD, dtype, kind], cwd=ROOT, check=True, capture_output=True,
                       text=True, timeout=300, env=dict(os.environ, PYTHONPATH=ROOT)).stdout
    wall, core = map(float, o.split())
    assert wall > 0.1, "the queued work was too short to show anything"
    assert core < 0.25 * wall, (wall, core)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_small_host_calls_after_waited_device_calls(dtype):
    p = W.make_problem(Q=1500, M=4, G=3, F=24, H1=128, H2=128, E=64, dtype=dtype, lam=0.4, slo=2.0, seed=4,
                       bias_std=0.05)
    st = torch.cuda.Stream()
    r = H.Router(p, stream=st.cuda_stream)
    ins = [torch.from_numpy(p[k].view(np.int16) if p[k].dtype == np.uint16 else p[k]).cuda()
           for k in ("in_len", "out_len", "emb")]
    out = [torch.empty(1500, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32)]
    torch.cuda.synchronize()
    few = [p[k][:3] for k in ("in_len", "out_len", "emb")]
    small = r.route(*few)
    r.route_device(*ins, *out, slo=p["slo"], lam=p["lam"])
    large = [o.cpu().numpy() for o in out]
    for i in range(40):
        if i % 8 == 7:      # work of the caller's own in between
            with torch.cuda.stream(st):
                torch.cuda._sleep(200_000)
        for o in out:
            o.zero_()
        torch.cuda.current_stream().synchronize()
        r.route_device(*ins, *out, slo=p["slo"], lam=p["lam"])
        got = r.route(*few)
        for g, w in zip(got, small):
            assert np.array_equal(g, w, equal_nan=True)
        for g, w in zip(out, large):
            assert np.array_equal(g.cpu().numpy(), w, equal_nan=True)
    r.close()

"""Waited device calls: the call returns on the host word that its last block
sets.  Outputs copied on another stream right after the return, without any
synchronisation, must be complete; inputs may be overwritten from another
stream; the synchronising fallback (limit 0) and calls behind queued work give
the same results.  Fused fp32 kernel and tensor path, split and whole tiles.
That the word does end such calls, over many grids and both paths in turn, is
asked for by HWR_TEST_POLL_ONLY, under which a call that falls back fails."""
import numpy as np
import pytest
import torch

import workload as W
import paper_2608_14575_gb300 as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    H.build()


@pytest.mark.parametrize("poll_us", [None, "0"])
@pytest.mark.parametrize("dtype,M,G,H1,Q", [("f32", 2, 2, 32, 256), ("f32", 4, 3, 64, 1500), ("bf16", 4, 3, 128, 1),
                                            ("bf16", 4, 3, 128, 4096), ("bf16", 8, 4, 64, 20001)])
def test_outputs_are_complete_at_the_return(monkeypatch, dtype, M, G, H1, Q, poll_us):
    if poll_us is not None:
        monkeypatch.setenv("HWR_TEST_POLL_US", poll_us)
    p = W.make_problem(Q=2 * Q, M=M, G=G, F=M + G + 9, H1=H1, H2=H1, E=64, dtype=dtype, lam=0.4, slo=2.0,
                       seed=M + Q, bias_std=0.05)
    st, other = torch.cuda.Stream(), torch.cuda.Stream()
    r = H.Router(p, stream=st.cuda_stream)
    flags = H.HWR_PATH_TENSOR if dtype == "bf16" else H.HWR_PATH_SIMT
    want = [r.route(*(p[k][a * Q:(a + 1) * Q] for k in ("in_len", "out_len", "emb")), flags=flags) for a in (0, 1)]
    src = [[torch.from_numpy(np.ascontiguousarray(p[k][a * Q:(a + 1) * Q]).view(np.int16 if p[k].dtype == np.uint16 else p[k].dtype)).cuda()
            for k in ("in_len", "out_len", "emb")] for a in (0, 1)]
    ins = [t.clone() for t in src[0]]
    out = [torch.empty(Q, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32)]
    kept = [[torch.empty_like(o) for o in out] for _ in range(20)]
    torch.cuda.synchronize()
    for i in range(20):
        if i % 5 == 4:     # behind queued work of the same context
            r.route_device(*src[1], *out, slo=p["slo"], lam=p["lam"], flags=flags | H.HWR_ASYNC)
        r.route_device(*ins, *out, slo=p["slo"], lam=p["lam"], flags=flags)
        with torch.cuda.stream(other):
            for k, o in zip(kept[i], out):
                k.copy_(o)
            for t, s in zip(ins, src[(i + 1) % 2]):
                t.copy_(s)
        other.synchronize()
    torch.cuda.synchronize()
    for i in range(20):
        for k, w in zip(kept[i], want[i % 2]):
            assert np.array_equal(k.cpu().numpy(), w, equal_nan=True), i
    r.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_the_host_word_ends_waited_calls(monkeypatch, dtype):
    monkeypatch.setenv("HWR_TEST_POLL_ONLY", "1")
    p = W.make_problem(Q=3000, M=4, G=2, F=18, H1=64, H2=64, E=64, dtype=dtype, lam=0.4, slo=2.0, seed=6,
                       bias_std=0.05)
    st = torch.cuda.Stream()
    r = H.Router(p, stream=st.cuda_stream)
    ins = [torch.from_numpy(p[k].view(np.int16) if p[k].dtype == np.uint16 else p[k]).cuda()
           for k in ("in_len", "out_len", "emb")]
    out = [torch.empty(3000, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32)]
    torch.cuda.synchronize()
    for i, Q in enumerate((3000, 97, 1024, 2999, 100, 513, 1500, 3000) * 4):
        path = H.HWR_PATH_TENSOR if dtype == "bf16" and i % 3 else H.HWR_PATH_SIMT
        r.route_device(*(t[:Q] for t in ins), *(o[:Q] for o in out), slo=p["slo"], lam=p["lam"], flags=path)
    r.close()
    # the fallback shows: nothing polls here
    monkeypatch.setenv("HWR_TEST_POLL_US", "0")
    r = H.Router(p, stream=st.cuda_stream)
    with pytest.raises(H.HwrError, match="host word"):
        r.route_device(*ins, *out, slo=p["slo"], lam=p["lam"], flags=path)
    r.close()

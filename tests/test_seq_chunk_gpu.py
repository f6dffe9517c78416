"""Chunks of a sequential call on the SIMT table: the results and the persisted
picks do not depend on the chunk size, and the size chosen takes no longer than
others do, with layer widths that are equal and not."""
import numpy as np
import pytest
import torch

import workload as W
import paper_2608_14575_gb300 as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,G,H1,H2", [(4, 3, 64, 256), (8, 4, 32, 256), (16, 4, 32, 256), (16, 4, 64, 256),
                                       (8, 4, 256, 32), (4, 3, 128, 128)])
def test_the_chunk_size_chosen_is_a_good_one(M, G, H1, H2, monkeypatch):
    H.build()
    Q, E = 1000, 64
    p = W.make_problem(Q=Q, M=M, G=G, F=M + G + 9, H1=H1, H2=H2, E=E, dtype="f32", lam=0.4, slo=3.0, seed=8,
                       bias_std=0.05)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        ins = [torch.from_numpy(p[k]).cuda() for k in ("in_len", "out_len", "emb")]
        out = [torch.empty(Q, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32)]
    st.synchronize()
    t, got = {}, {}
    for n in ("0", "16", "24", "32", "48", "64"):
        monkeypatch.setenv("HWR_TEST_SEQ_CHUNK", n)
        r = H.Router(p, stream=st.cuda_stream)
        best = 1e9
        for _ in range(5):
            r.update_snapshot(p["snap"])
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(st)
            r.route_device(*ins, *out, slo=3.0, lam=0.4, flags=H.HWR_SEQUENTIAL | H.HWR_ASYNC)
            b.record(st)
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        t[n], got[n] = best, [o.cpu().numpy() for o in out] + [r.get_snapshot()]
        r.close()
    for n in t:
        for x, y in zip(got[n], got["0"]):
            assert np.array_equal(x, y, equal_nan=True), n
    # (by H1 alone 1.3 times the best of them at 64 x 256 and 32 x 256)
    assert t["0"] < 1.22 * min(t.values()), t

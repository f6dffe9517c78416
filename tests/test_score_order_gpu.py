"""Scores queued back to back on the tensor-core path, where a call's quality
kernel starts beside the previous call's predictor and writes the caller's
array itself: two batches scored in turn into the same arrays, each with a
copy of its results queued behind it, and the quality array of one call as the
lengths of the next; every result equals the same call run alone.  Model
counts whose rows are vectors and not, rows past the last full tile."""
import numpy as np
import pytest
import torch

import workload as W
import paper_2608_14575_gb300 as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    H.build()


@pytest.mark.parametrize("M,G,Q", [(16, 2, 700), (8, 4, 4111), (5, 3, 1000), (17, 2, 300), (3, 1, 20001)])
def test_queued_scores_equal_lone_ones(M, G, Q):
    p = W.make_problem(Q=2 * Q, M=M, G=G, F=M + G + 9, H1=64, H2=128, E=128, dtype="bf16", lam=0.4,
                       slo=2.0, seed=M, bias_std=0.05)
    st = torch.cuda.Stream()
    r = H.Router(p, stream=st.cuda_stream)
    with torch.cuda.stream(st):
        il, ol = (torch.from_numpy(p[k]).cuda() for k in ("in_len", "out_len"))
        emb = torch.from_numpy(p["emb"].view(np.int16)).cuda()
        parts = [tuple(t[k * Q:(k + 1) * Q].contiguous() for t in (il, ol, emb)) for k in range(2)]
        cost = torch.empty(Q, p["D"], device="cuda")
        # a caller's array that starts on a 4-byte boundary only, and one that does not
        for off in (0, 1):
            qual = torch.empty(Q * M + off, device="cuda")[off:].view(Q, M)
            alone = []
            for part in parts:
                r.score_device(*part, cost, qual, flags=H.HWR_PATH_TENSOR)
                alone.append((cost.clone(), qual.clone()))
            st.synchronize()
            for _ in range(3):
                got = []
                for k in (0, 1, 1, 0, 1):
                    r.score_device(*parts[k], cost, qual, flags=H.HWR_PATH_TENSOR | H.HWR_ASYNC)
                    if k == 1:
                        got.append((k, cost.clone(), qual.clone()))
                got.append((1, cost.clone(), qual.clone()))
                r.synchronize()
                for k, c, q in got:
                    assert torch.equal(c, alone[k][0]) and torch.equal(q, alone[k][1])
            # the quality scores as the next call's input lengths
            lens = qual.view(-1)[:Q]
            r.score_device(*parts[0], cost, qual, flags=H.HWR_PATH_TENSOR | H.HWR_ASYNC)
            r.score_device(lens, parts[1][1], parts[1][2], cost, None, flags=H.HWR_PATH_TENSOR | H.HWR_ASYNC)
            chained = cost.clone()
            r.synchronize()
            r.score_device(lens.clone(), parts[1][1], parts[1][2], cost, None, flags=H.HWR_PATH_TENSOR)
            assert torch.equal(chained, cost)
    r.close()

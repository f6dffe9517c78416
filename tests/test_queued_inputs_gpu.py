"""Queued tensor-core calls that read what an earlier queued call wrote, with
other calls between the two: kernels of a queued route start before those of
the routes before it have finished, so the library has to notice such inputs
however far back their writer is.  Lengths, budgets and embeddings taken from a
large call's scores, behind 0 to 30 small calls into their own arrays (more
arrays than the library keeps note of), and from a decision's outputs; every
result equals the one with a wait between the calls."""
import numpy as np
import pytest
import torch

import workload as W
import paper_2608_14575_gb300 as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    H.build()


@pytest.mark.parametrize("between", [0, 1, 2, 5, 30])
@pytest.mark.parametrize("what", ["lengths", "budgets", "embeddings"])
def test_inputs_written_by_an_earlier_queued_call(what, between):
    Q, n, E = 20001, 1000, 64
    p = W.make_problem(Q=Q, M=8, G=4, F=21, H1=64, H2=128, E=E, dtype="bf16", lam=0.4, slo=2.0, seed=9,
                       bias_std=0.05)
    D = p["D"]
    st = torch.cuda.Stream()
    r = H.Router(p, stream=st.cuda_stream)
    flags = H.HWR_PATH_TENSOR
    with torch.cuda.stream(st):
        il, ol = (torch.from_numpy(p[k]).cuda() for k in ("in_len", "out_len"))
        emb = torch.from_numpy(p["emb"].view(np.int16)).cuda()
        new = lambda: [torch.empty(n, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32)]  # noqa: E731
        cost = torch.empty(Q, D, device="cuda")
        route, side, last = [torch.empty(Q, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32)], \
            [new() for _ in range(between)], new()

        def chain(wait):
            cost.fill_(0.25)
            route[1].fill_(0.25)
            for o in last:
                o.zero_()
            f = flags if wait else flags | H.HWR_ASYNC
            if what == "budgets":
                r.route_device(il, ol, emb, *route, slo=p["slo"], lam=p["lam"], flags=f)
            else:
                r.score_device(il, ol, emb, cost, flags=f)
            for o in side:
                r.route_device(il[:n], ol[:n], emb[:n], *o, slo=p["slo"], lam=p["lam"], flags=f)
            # the writer's last rows: its last tile finishes last
            if what == "lengths":
                r.route_device(cost.view(-1)[-n:], ol[:n], emb[:n], *last, slo=p["slo"], lam=p["lam"], flags=f)
            elif what == "budgets":
                b = route[1][-n:]
                r.route_device_slo(il[:n], ol[:n], emb[:n], *last, budgets=b, lam=p["lam"], flags=f)
            else:
                e = cost.view(-1)[-n * E // 2:].view(torch.bfloat16).view(n, E)
                assert e.data_ptr() % 16 == 0
                r.route_device(il[:n], ol[:n], e, *last, slo=p["slo"], lam=p["lam"], flags=f)
            r.synchronize()
            return [o.cpu().numpy().view(np.int32) for o in last + [x for s in side for x in s]]

        want = chain(True)
        for _ in range(5):
            for g, w in zip(chain(False), want):
                assert np.array_equal(g, w)
    r.close()

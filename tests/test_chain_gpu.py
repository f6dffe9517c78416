"""The serial walk of sequential mode (k_seq_chain) at its edges, bit for bit
against the oracle: chunks of one query up to several chunks and their
remainders, deployments below, at and above the 32 of one half, a utility that
overflows to -inf and costs that overflow to inf (the walk's long way, with and
without a budget that lets them in), ties, all costs NaN, and every mix of
feasible and infeasible steps."""
import numpy as np
import pytest

import oracle as O
import workload as W
import paper_2608_14575_gb300 as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    H.build()


def _problem(Q, M, G, heads=2):
    return W.make_problem(Q=Q, M=M, G=G, F=M + G + 9, H1=32, H2=32, E=64, dtype="f32", lam=0.5,
                          slo=1.0, seed=M + Q, bias_std=0.05, n_heads=heads)


def _check(p, **kw):
    r = H.Router(p)
    got = r.route(flags=H.HWR_SEQUENTIAL)
    want = O.Problem(p).route(mode=O.F32, sequential=True)
    for g, w, t in zip(got, want, (np.int32, np.float32, np.float32)):
        assert np.array_equal(g, np.asarray(w).astype(t), equal_nan=True)
    assert np.array_equal(r.get_snapshot(), want[3])
    r.close()


@pytest.mark.parametrize("M,G", [(1, 1), (5, 1), (31, 1), (8, 4), (11, 3), (16, 4)])
@pytest.mark.parametrize("Q", [1, 2, 31, 32, 33, 64, 65, 150])
def test_shapes(M, G, Q):
    p = _problem(Q, M, G)
    p["slo"] = float(np.median([0.5, 1.0, 2.0])) * (1 + Q % 3)
    _check(p)


@pytest.mark.parametrize("slo", [float("inf"), 2.0, 0.0, float("-inf")])
@pytest.mark.parametrize("what", ["huge_lambda", "huge_cost", "some_huge", "nan_cost", "ties"])
@pytest.mark.parametrize("M,G", [(4, 3), (13, 3)])
def test_values_off_the_ordinary_range(M, G, what, slo):
    p = _problem(70, M, G)
    p["slo"] = slo
    rng = np.random.default_rng(1)
    if what == "huge_lambda":
        p["lam"] = 3e38                       # utilities overflow to -inf
    elif what == "huge_cost":
        p["out_len"] = np.full_like(p["out_len"], 3e38)
        p["b3"] = p["b3"].copy()
        p["b3"][1] = 20.0                     # costs overflow to inf
    elif what == "some_huge":
        p["out_len"] = np.where(rng.random(70) < 0.4, np.float32(3e38), p["out_len"])
        p["b3"] = p["b3"].copy()
        p["b3"][1] = 3.0
    elif what == "nan_cost":
        p["W3"] = p["W3"].copy()
        p["W3"][0, :] = np.nan
    else:                                     # every deployment alike
        p["W1"] = np.zeros_like(p["W1"])
        p["memb"] = np.zeros_like(p["memb"])
    _check(p)


@pytest.mark.parametrize("M,G,Q", [(4, 3, 1024), (5, 1, 1025), (4, 3, 2100), (16, 4, 1200)])
def test_runs_of_chunks(M, G, Q):
    """Calls longer than one run of prepared prefixes, and a second call that
    continues from the first one's counts."""
    p = _problem(Q, M, G)
    p["slo"] = 4.0
    _check(p)
    r = H.Router(p)
    orc = O.Problem(p)
    running = p["snap"]["running"]
    for lo, hi in ((0, 130), (130, Q)):
        s = W.query_slice(p, lo, hi)
        got = r.route(s["in_len"], s["out_len"], s["emb"], flags=H.HWR_SEQUENTIAL)
        want = orc.route(s["in_len"], s["out_len"], s["emb"], mode=O.F32, sequential=True, running=running)
        for g, w, t in zip(got, want, (np.int32, np.float32, np.float32)):
            assert np.array_equal(g, np.asarray(w).astype(t), equal_nan=True)
        running = want[3]
        assert np.array_equal(r.get_snapshot(), running)
    # a batch route after it sees the prefixes of the final counts
    got = r.route(p["in_len"][:50], p["out_len"][:50], p["emb"][:50], flags=H.HWR_PATH_SIMT)
    snap = dict(p["snap"], running=running)
    orc.set_snapshot(snap)
    want = orc.route(p["in_len"][:50], p["out_len"][:50], p["emb"][:50], mode=O.F32)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1].astype(np.float32))
    r.close()

"""The selection over several lambdas (k_select_multi): every number of
lambdas, so every template and its padding, deployments short of a group of
four and of the four lanes' share, cost rows read as vectors and one by one,
query counts that end inside a warp; each row equals the single-lambda route."""
import numpy as np
import pytest

import workload as W
import paper_2608_14575_gb300 as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    H.build()


@pytest.mark.parametrize("M,G,Q,dtype,flags", [
    (1, 1, 3, "f32", 0), (3, 1, 70, "f32", 0), (2, 2, 333, "f32", H.HWR_SCORE_CONVEX),
    (5, 1, 41, "f32", 0), (4, 4, 129, "f32", 0), (17, 1, 65, "f32", 0), (5, 9, 77, "f32", 0),
    (16, 4, 201, "bf16", 0), (7, 5, 300, "bf16", H.HWR_SCORE_CONVEX),
])
def test_rows_equal_single_lambda_routes(M, G, Q, dtype, flags):
    p = W.make_problem(Q=Q, M=M, G=G, F=M + G + 9, H1=64, H2=64, E=64, dtype=dtype, lam=0.4,
                       slo=2.0, seed=M + G, bias_std=0.05)
    lams = np.linspace(0.0, 1.0, 16).astype(np.float32)
    r = H.Router(p)
    if dtype == "bf16":
        flags |= H.HWR_PATH_TENSOR
    single = [r.route(lam=float(x), flags=flags) for x in lams]
    for K in (1, 3, 4, 5, 8, 9, 12, 13, 16):
        got = r.route_multi(lams[:K], flags=flags)
        for k in range(K):
            for a, b in zip(got, single[k]):
                assert np.array_equal(a[k], b, equal_nan=True), (K, k)
    r.close()

"""A sequential call that finds no memory for the layer-1 prefixes of a whole run
of chunks prepares them chunk by chunk: same results, same persisted picks.  The
allocations of the call fail in turn on the host; the one that holds the
prefixes is the only one whose failure does not end the call."""
import numpy as np
import pytest

import oracle as O
import workload as W
import paper_2608_14575_gb300 as H
from paper_2608_14575_gb300 import _hwr

pytestmark = pytest.mark.gpu


def test_prefixes_fall_back_to_one_chunk(monkeypatch):
    H.build()
    p = W.make_problem(Q=300, M=4, G=3, F=24, H1=32, H2=32, E=64, dtype="f32", lam=0.4, slo=3.0, seed=5,
                       bias_std=0.05)
    want = O.Problem(p).route(mode=O.F32, sequential=True)
    n, created, fell_back = 1, False, 0
    while True:
        monkeypatch.setenv("HWR_TEST_FAIL_ALLOC", str(n))
        n += 1
        try:
            r = H.Router(p)
        except H.HwrError:
            assert not created
            continue
        created = True
        try:
            got = r.route(flags=H.HWR_SEQUENTIAL)
        except H.HwrError as e:
            assert e.status == _hwr.HWR_ERR_OOM
            r.close()
            continue
        for g, w, t in zip(got, want, (np.int32, np.float32, np.float32)):
            assert np.array_equal(g, np.asarray(w).astype(t), equal_nan=True)
        assert np.array_equal(r.get_snapshot(), want[3])
        failed = "test hook" in H.hwr_last_error(r.ctx)
        r.close()
        if not failed:
            break               # no allocation of the call is left to fail
        fell_back += 1
    assert fell_back == 1

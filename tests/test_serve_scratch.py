"""Requests at the limit of the serving budget: one whose walks in flight and query order would
need more than the budget runs with fewer walks and in query order, so the smallest budget that
serves a request in query order serves it whatever its order."""
import re

import numpy as np
import pytest

from paper_1804_09996_gb300 import lc
from test_serve import _alone, _run, served  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [40, 420, 1500])
def test_smallest_budget_serves_every_order(served, nq):  # noqa: F811
    h, xq, _ = served
    q = np.ascontiguousarray(np.tile(xq, (nq // len(xq) + 1, 1))[:nq], np.float32)
    sp = lc.lc_default_search_params(10, 64, order=lc.LC_ORDER_NEVER)
    srv = lc.lc_serve_open(h, 4096, 1, nq)
    try:
        with pytest.raises(lc.LcError) as e:
            lc.lc_serve_submit(srv, q, sp, lc.make_request_cb(lambda *a: None))
        assert e.value.status == lc.LC_ERR_BUDGET
        least = int(re.search(r"needs (\d+) bytes", e.value.message).group(1))
    finally:
        lc.lc_serve_close(srv)
    ref = _alone(h, q, sp)
    srv = lc.lc_serve_open(h, least, 1, nq)
    try:
        reqs = [(q, lc.lc_default_search_params(10, 64, order=o)) for o in (lc.LC_ORDER_NEVER, lc.LC_ORDER_AUTO, lc.LC_ORDER_ALWAYS)]
        ids, results, cbs = _run(srv, reqs)
        for rid in ids:
            st, i, d = results[rid]
            assert st == lc.LC_OK
            assert np.array_equal(i, ref[0]) and np.array_equal(d.view(np.int32), ref[1].view(np.int32))
    finally:
        lc.lc_serve_close(srv)

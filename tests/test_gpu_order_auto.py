"""The automatic choice of the query order: a batch of which every query walks at once is never
ordered, however small (an eighth of fewer than eight walks is less than one query), and one with a
second round of walks is."""
import numpy as np
import pytest

from paper_1804_09996_gb300 import lc
from test_gpu_order import search
from test_gpu_parity import handle

pytestmark = pytest.mark.gpu


def descent_ms(h, q, order):
    lc.lc_profile(h, True)
    try:
        ms = []
        for _ in range(5):
            search(h, q, 10, 64, order)
            ms.append(lc.lc_profile_phases(h)[1])
        return float(np.median(ms))
    finally:
        lc.lc_profile(h, False)


@pytest.mark.parametrize("name", ["mix3k", "sift2k"])
@pytest.mark.parametrize("nq,ordered", [(1, False), (2, False), (7, False), (8, False), (200, False), (8000, True)])
def test_auto_order(request, name, nq, ordered):
    # (without an order there is nothing between the two events; an ordered search has two kernels)
    ix, xb, xq = request.getfixturevalue(name)
    h = handle(name, ix)
    q = np.tile(xq, (nq // len(xq) + 1, 1))[:nq]
    auto, always, never = (descent_ms(h, q, o) for o in (lc.LC_ORDER_AUTO, lc.LC_ORDER_ALWAYS, lc.LC_ORDER_NEVER))
    assert never < 0.5 * always
    assert (auto > 0.5 * always) == ordered, (auto, always, never)

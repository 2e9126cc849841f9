"""Ordered searches whose re-rank reads the level-2 codebook through the cache (d > 104: the two
FP32 codebooks do not fit in shared memory together) are the same bit for bit as query-order ones,
with one warp and with teams of warps per query."""
import numpy as np
import pytest

from test_gpu_full_walk_splits import index
from test_gpu_order import same, search
from test_gpu_parity import handle

from paper_1804_09996_gb300 import lc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [40, 1300, 6000])
@pytest.mark.parametrize("shortlist,beam", [(0, 1), (100, 4)])
@pytest.mark.parametrize("split", [(128, 16, 16), (207, 16, 40)])
def test_ordered_equals_query_order(split, shortlist, beam, nq):
    ix, xq = index(split)
    h = handle(f"split{split}", ix)
    q = np.tile(xq, (nq // len(xq) + 1, 1))[:nq]
    a = search(h, q, 10, 40, lc.LC_ORDER_ALWAYS, beam=beam, shortlist=shortlist)
    same(a, search(h, q, 10, 40, lc.LC_ORDER_NEVER, beam=beam, shortlist=shortlist))
    m = min(nq, len(xq))
    same([x[:m] for x in a], search(h, xq[:m], 10, 40, lc.LC_ORDER_NEVER, beam=beam, shortlist=shortlist))

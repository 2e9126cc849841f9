"""A re-rank that reads the level-2 codebook through the cache (d = 128) runs beside the walks of an
ordered search or after them, by one warp or a team per query, by the number of candidates, efSearch
and the form of the walk: the same bit for bit on both sides of the line."""
import numpy as np
import pytest

from test_gpu_full_walk_splits import index
from test_gpu_order import same, search
from test_gpu_parity import handle

from paper_1804_09996_gb300 import lc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,ef,shortlist,beam,full", [
    (9_000, 256, 0, 4, 0), (30_000, 256, 0, 4, 0),          # one warp per query: beside, after
    (5_200, 256, 32, 1, 0), (5_200, 128, 32, 1, 0),         # teams: beside (by one warp each), after
    (40, 256, 100, 1, 0), (3_000, 16, 0, 4, 1), (3_700, 16, 0, 4, 1),
])
def test_beside_or_after_the_walks(nq, ef, shortlist, beam, full):
    ix, xq = index((128, 16, 16))
    h = handle("split(128, 16, 16)", ix)
    q = np.tile(xq, (nq // len(xq) + 1, 1))[:nq]
    form = dict(beam=beam, shortlist=shortlist, walk_full=full)
    same(search(h, q, 10, ef, lc.LC_ORDER_ALWAYS, **form), search(h, q, 10, ef, lc.LC_ORDER_NEVER, **form))

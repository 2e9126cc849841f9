"""Walks by teams of warps (small batches) on graphs whose upper levels have rows without
neighbours: a lone entry point on the top level, and empty levels below it.  The same bits, visit
counts included, as the walks of one warp each."""
import numpy as np
import pytest

from paper_1804_09996_gb300 import lc
from test_gpu_order import same
from test_gpu_visited import search

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("empty_from", [1, 2])
@pytest.mark.parametrize("name", ["mix3k", "opq3k", "odd2k"])
@pytest.mark.parametrize("beam,full", [(1, 0), (4, 0), (1, 1)])
def test_rows_without_neighbours(request, name, beam, full, empty_from):
    ix, xb, xq = request.getfixturevalue(name)
    # the entry point alone on three more levels; rows from level empty_from on are empty
    levels = ix.levels.copy()
    levels[ix.ep] += 3
    rows, r = [], 0
    for i, old in enumerate(ix.levels):
        for l in range(1, levels[i] + 1):
            keep = l <= old and l < empty_from
            rows.append(ix.upper_adj[r + l - 1] if keep else np.full(32, -1, np.int32))
        r += old
    h = lc.lc_create(lc.lc_default_params(ix.d, ix.M1, ix.M2))
    try:
        lc.lc_import(h, ix.N, ix.R, ix.C1, ix.C2, ix.codes1, ix.codes2, ix.beta, ix.B, ix.adj0, levels,
                     np.ascontiguousarray(rows, np.int32), ix.ep)
        big = search(h, np.tile(xq, (1000 // len(xq) + 1, 1)), 10, 48, beam, 0, walk_full=full)      # one warp each
        assert (big[2][:, 0] > 100).all()
        for n in (1, 7, len(xq)):
            same(search(h, xq[:n], 10, 48, beam, 0, walk_full=full), [x[:n] for x in big])
            same(search(h, xq[:n], 10, 48, beam, 0, walk_full=full, warps=3), [x[:n] for x in big])
    finally:
        lc.lc_free(h)

"""The two storages of a walk's visited set (16-bit tags, the automatic choice; 32-bit ids, when
a caller asks for a table size) hold the same set under the same limits, so every search must
be the same bit for bit: ids, distances, visit counts.  Wide searches on small indexes visit
every node, more than the buckets of tags hold, so the overflow tables (shared, then global) are
covered; adjacency rows with repeated ids too (an imported graph may have them)."""
import numpy as np
import pytest

from paper_1804_09996_gb300 import lc
from test_gpu_order import same
from test_gpu_parity import handle

pytestmark = pytest.mark.gpu


def search(h, xq, k, ef, beam, vlog, **more):
    import torch
    nq = len(xq)
    sp = lc.lc_default_search_params(k, ef, visited_log=vlog, **more)
    if beam > 1:
        sp.mode, sp.beam = lc.LC_MODE_BATCHED, beam
    q = torch.from_numpy(np.ascontiguousarray(xq, np.float32)).cuda()
    ids = torch.full((nq, k), -7, dtype=torch.int32, device="cuda")
    ds = torch.full((nq, k), -7.0, dtype=torch.float32, device="cuda")
    st = torch.full((nq, 3), -7, dtype=torch.int32, device="cuda")
    lc.lc_search(h, q, nq, sp, ids, ds, st, torch.cuda.current_stream())
    return ids.cpu().numpy(), ds.cpu().numpy(), st.cpu().numpy()


@pytest.mark.parametrize("ef,beam", [(1, 1), (32, 1), (32, 4), (64, 1), (64, 8), (300, 1), (1000, 4)])
@pytest.mark.parametrize("name", ["mix3k", "opq3k", "sift2k", "odd2k"])
def test_tags_equal_ids(request, name, ef, beam):
    ix, xb, xq = request.getfixturevalue(name)
    h = handle(name, ix)
    k = min(10, ef)
    vlog = 10 if ef <= 32 else 11                              # the automatic limits at this efSearch
    got = search(h, xq, k, ef, beam, 0)
    same(got, search(h, xq, k, ef, beam, vlog))
    assert (got[2][:, 0] > 0).all()
    if ef == 1000:
        assert got[2][:, 0].max() > 1800                       # nearly the whole index


@pytest.mark.parametrize("beam", [1, 4])
def test_rows_with_repeated_ids(mix3k, beam):
    ix, xb, xq = mix3k
    adj = ix.adj0.copy()
    adj[:, 9] = adj[:, 0]                                      # a repeated neighbour in every row,
    adj[::3, 10:13] = adj[::3, :1]                             # several in some
    h = lc.lc_create(lc.lc_default_params(ix.d, ix.M1, ix.M2))
    try:
        lc.lc_import(h, ix.N, ix.R, ix.C1, ix.C2, ix.codes1, ix.codes2, ix.beta, ix.B, adj, ix.levels, ix.upper_adj, ix.ep)
        a = search(h, xq, 10, 64, beam, 0)
        same(a, search(h, xq, 10, 64, beam, 11))
        assert all(len(set(r)) == 10 for r in a[0])
    finally:
        lc.lc_free(h)


@pytest.mark.parametrize("name,u8", [("mix3k", False), ("opq3k", False), ("sift2k", True), ("odd2k", False)])
@pytest.mark.parametrize("k,shortlist,beam,prec,full", [(10, 0, 1, 0, 0), (40, 100, 4, 0, 0), (10, 0, 8, 1, 0), (10, 0, 1, 0, 1),
                                                       (5, 0, 4, 0, 1)])
def test_batch_size_does_not_matter(request, name, u8, k, shortlist, beam, prec, full):
    # large batches (tiled rotation, one warp per query) against small ones (direct rotation,
    # teams of warps in the walk and in the re-rank): the same bits for every query
    import torch
    ix, xb, xq = request.getfixturevalue(name)
    h = handle(name, ix)
    d = ix.d
    q = torch.from_numpy(np.ascontiguousarray(np.tile(xq, (4133 // len(xq) + 1, 1))[:4133], np.uint8 if u8 else np.float32)).cuda()
    sp = lc.lc_default_search_params(k, 48, shortlist=shortlist, lut_prec=prec, walk_full=full,
                                     mode=lc.LC_MODE_BATCHED if beam > 1 else lc.LC_MODE_PLAIN, beam=beam)
    out = {}
    for size in (4133, 701, 7):
        n = 4133 if size == 4133 else 3 * size
        ids = torch.empty((n, k), dtype=torch.int32, device="cuda")
        ds = torch.empty((n, k), dtype=torch.float32, device="cuda")
        for a in range(0, n, size):
            lc.lc_search_ex(h, q[a:a + size], lc.LC_QUERY_U8 if u8 else lc.LC_QUERY_F32, size, sp, None, ids[a:a + size],
                            ds[a:a + size], None, torch.cuda.current_stream())
        out[size] = ids.cpu().numpy(), ds.cpu().numpy()
    for size in (701, 7):
        n = 3 * size
        assert np.array_equal(out[size][0], out[4133][0][:n])
        assert np.array_equal(out[size][1].view(np.int32), out[4133][1][:n].view(np.int32))
    assert d % 4 == 0

"""The visited set of 16-bit tags where its tables are at their limits, against the storage of 32-bit
ids under the same limits, bit for bit (ids, distances, visit counts, failed queries):

* the capacity limit, which the automatic storage reaches in walks over a random graph;
* tags of the full 16 bits (above 2^22 ids at the smaller table size: an id whose tag is 0 never
  sits in a bucket, the entry node 0 first of all);
* the table with one more bit of buckets (above 2^23 ids there), whose tags are 16 bits again.

The graphs are random: every row brings about 32 new nodes, all over the id range."""
import numpy as np
import pytest

from paper_1804_09996_gb300 import lc
from test_gpu_order import same

pytestmark = pytest.mark.gpu


def random_index(n, d, M1, M2, degree=32):
    rng = np.random.default_rng(n)
    C1, C2 = rng.standard_normal((256, d)).astype(np.float32), 0.2 * rng.standard_normal((256, d)).astype(np.float32)
    adj = np.full((n, 32), -1, np.int32)
    adj[:, :degree] = rng.integers(0, n, (n, degree), dtype=np.int32)
    B = np.zeros((256, 9), np.float32)
    B[:, 0] = 1.0
    h = lc.lc_create(lc.lc_default_params(d, M1, M2, use_opq=0))
    lc.lc_import(h, n, np.eye(d, dtype=np.float32), C1, C2.astype(np.float32), rng.integers(0, 256, (n, M1), dtype=np.uint8),
                 rng.integers(0, 256, (n, M2), dtype=np.uint8), np.zeros(n, np.uint8), B, adj, np.zeros(n, np.int32),
                 np.zeros((0, 32), np.int32), 0)
    return h


def search(h, q, k, ef, beam, vlog, slog=0, warps=0):
    import torch
    nq = len(q)
    sp = lc.lc_default_search_params(k, ef, visited_log=vlog, spill_log=slog, warps=warps)
    if beam > 1:
        sp.mode, sp.beam = lc.LC_MODE_BATCHED, beam
    qd = torch.from_numpy(q).cuda()
    ids = torch.full((nq, k), -7, dtype=torch.int32, device="cuda")
    ds = torch.full((nq, k), -7.0, dtype=torch.float32, device="cuda")
    st = torch.full((nq, 3), -7, dtype=torch.int32, device="cuda")
    lc.lc_search(h, qd, nq, sp, ids, ds, st, torch.cuda.current_stream())
    return ids.cpu().numpy(), ds.cpu().numpy(), st.cpu().numpy()


def test_capacity_of_the_automatic_storage():
    # limits of 3/4 * 2^11 + 2^13 / 2 = 5,632 nodes at efSearch 128: a walk of 128 expansions and more
    # over rows of 32 is at about 4,000 to 6,000
    d = 16
    h = random_index(200_000, d, 16, 4)
    try:
        q = np.random.default_rng(1).standard_normal((700, d)).astype(np.float32)
        seen = []
        for ef, beam in ((128, 1), (128, 4), (128, 8), (100, 8)):
            ids = search(h, q, 10, ef, beam, 11, 13)
            failed = ids[2][:, 0] == -1
            seen.append(failed.mean())
            for n, warps in ((700, 0), (700, 3), (37, 0)):
                same(search(h, q[:n], 10, ef, beam, 0, warps=warps), [x[:n] for x in ids])
            assert (ids[0][failed] == -1).all() and (ids[0][~failed] >= 0).all()
        assert max(seen) > 0.02 and min(seen) < 0.98, seen
    finally:
        lc.lc_free(h)


@pytest.mark.parametrize("n", [(1 << 22) + 1000, (1 << 23) + 1000])
def test_tags_of_large_indexes(n):
    d = 16
    h = random_index(n, d, 16, 4, degree=24)
    try:
        q = np.random.default_rng(2).standard_normal((700, d)).astype(np.float32)
        for ef, beam in ((16, 1), (32, 4), (32, 8), (64, 1), (128, 4)):
            vlog = 10 if ef <= 32 else 11                      # the automatic limits at this efSearch
            ids = search(h, q, 10, ef, beam, vlog)
            for m in (700, 37):
                same(search(h, q[:m], 10, ef, beam, 0), [x[:m] for x in ids])
            assert (ids[2][:, 0] > 8 * ef).all() or (ids[2][:, 0] == -1).any()
    finally:
        lc.lc_free(h)

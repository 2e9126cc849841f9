"""lc_merge_topk against a sort of all keys: list counts up to one and two per lane, k of one to
200, short lists, equal keys in several shards, and lists in no order (sorted all the same)."""
import numpy as np
import pytest

from paper_1804_09996_gb300 import lc

pytestmark = pytest.mark.gpu


def reference(ids, ds, off, k):
    S, nq, _ = ids.shape
    oi, od = np.full((nq, k), -1, np.int32), np.full((nq, k), np.inf, np.float32)
    for q in range(nq):
        have = ids[:, q] >= 0
        gi = (ids[:, q].astype(np.int64) + off[:, None])[have].astype(np.int32)
        gd = ds[:, q][have]
        o = np.lexsort((gi, gd))[:k]
        oi[q, :len(o)], od[q, :len(o)] = gi[o], gd[o]
    return oi, od


@pytest.mark.parametrize("S,nq,k", [(1, 1, 1), (2, 33, 1), (8, 500, 10), (32, 70, 33), (33, 50, 7), (64, 40, 32), (3, 17, 200)])
@pytest.mark.parametrize("order", ["ascending", "none"])
def test_merge_equals_sorting(S, nq, k, order):
    import torch
    rng = np.random.default_rng(S * 1000 + k)
    ids = rng.integers(0, 5000, (S, nq, k)).astype(np.int32)
    ds = (rng.integers(0, 50, (S, nq, k)) / 8).astype(np.float32)          # many equal distances
    short = rng.integers(0, k + 1, (S, nq))
    pad = (np.arange(k) >= short[..., None]) & (rng.random((S, nq, 1)) < 0.3)
    ids[pad], ds[pad] = -1, np.inf
    off = np.zeros(S, np.int64) if S == 2 else np.arange(S) * 4000         # (S = 2: the same keys in both shards)
    if S == 2:
        ids[1], ds[1] = ids[0], ds[0]
    if order == "ascending":
        for s in range(S):
            for q in range(nq):
                o = np.lexsort((np.where(ids[s, q] < 0, 1 << 30, ids[s, q]), ds[s, q]))
                ids[s, q], ds[s, q] = ids[s, q][o], ds[s, q][o]
    ti, td = torch.from_numpy(ids).cuda(), torch.from_numpy(ds).cuda()
    oi = torch.empty((nq, k), dtype=torch.int32, device="cuda")
    od = torch.empty((nq, k), dtype=torch.float32, device="cuda")
    lc.lc_merge_topk(ti, td, S, nq, k, off, oi, od, torch.cuda.current_stream())
    ri, rd = reference(ids, ds, off, k)
    assert np.array_equal(oi.cpu().numpy(), ri)
    assert np.array_equal(od.cpu().numpy(), rd)

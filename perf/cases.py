"""Performance cases of the Link-and-Code search: what users of the library have it do, from one
query to 100,000, through the C ABI's entry points (``paper_1804_09996_gb300.lc``).

``listed()`` are the cases, ``draw(rng)`` more of the same ranges, ``prepare(case, seed)`` what
a program holds before the call (index, plan, queries), ``run(state)`` one pass, ``work(case)``
the bytes and operations a pass cannot do without, ``exact(case, seed)`` the distances in 64
bits by plain torch (the same walk and re-rank restated on the index arrays).

An index is built once per process and kept, as a serving program keeps it; its vectors are
fixed, the queries come from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1804_09996_gb300 import lc

# ------------------------------------------------------------------------------------------
# Indexes.  The sizes and codes are those of the repository's workloads (datagen.WORKLOADS,
# bench.py) and tests; "mix3m" stands for the 10M and 50M mixtures: its codes and graph
# (576 MB) are far larger than L2, at a size that is built in seconds.
INDEXES = {
    # 10k x 96, 64 centres, PQ16 + residual PQ16: the small workload
    "mix10k": dict(n=10_000, d=96, M1=16, M2=16, kind="mixture", centres=64, n_train=8_000, opq=0),
    # 1M x 96, 1,024 centres, OPQ32 + PQ31 + 1-byte codeword = 64 B/vector: the default bench
    "mix1m": dict(n=1_000_000, d=96, M1=32, M2=31, kind="mixture", centres=1024, n_train=20_000, opq=1),
    # the same codes at 3M vectors: does not fit L2
    "mix3m": dict(n=3_000_000, d=96, M1=32, M2=31, kind="mixture", centres=1024, n_train=20_000, opq=1),
    # 1M x 128 SIFT-like uint8, OPQ64 + PQ63 = 128 B/vector
    "sift1m": dict(n=1_000_000, d=128, M1=64, M2=63, kind="sift", centres=1024, n_train=20_000, opq=1),
    # product regression codebook: 8 blocks of 64 codewords (8 bytes per vector)
    "prod50k": dict(n=50_000, d=96, M1=32, M2=32, kind="mixture", centres=128, n_train=8_000, opq=1, beta_M=8, beta_K=64),
    # neither 16 nor 25 sub-spaces divide 100 coordinates: the uneven split of the paper's
    # OPQ14 / OPQ30 on 96 dimensions
    "odd20k": dict(n=20_000, d=100, M1=16, M2=25, kind="mixture", centres=64, n_train=8_000, opq=0),
}
SEED_BASE = 1804          # centres and database vectors
_index: dict = {}
_arrays: dict = {}
_plans: dict = {}


def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(seed)


def _vectors(c, n: int, seed: int) -> torch.Tensor:
    """n vectors of the index's distribution, on the GPU: unit-norm Gaussian mixture (CNN
    descriptors) float32, or SIFT-like uint8 (non-negative, heavy-tailed, many zeros)."""
    d, k = c["d"], c["centres"]
    g = _gen(seed)
    out = torch.empty((n, d), dtype=torch.uint8 if c["kind"] == "sift" else torch.float32, device="cuda")
    if c["kind"] == "sift":
        mu = torch.from_numpy(np.random.default_rng(SEED_BASE).gamma(0.5, 40.0, (k, d))).float().cuda()
    else:
        mu = torch.randn((k, d), generator=_gen(SEED_BASE), device="cuda") / math.sqrt(d)
    for a in range(0, n, 1 << 19):
        m = min(1 << 19, n - a)
        centre = mu[torch.randint(k, (m,), generator=g, device="cuda")]
        if c["kind"] == "sift":
            e = torch.empty((m, d), device="cuda").exponential_(generator=g)
            out[a:a + m] = (centre * e).floor_().clamp_(max=255).to(torch.uint8)
        else:
            x = centre + (0.6 / math.sqrt(d)) * torch.randn((m, d), generator=g, device="cuda")
            out[a:a + m] = x / x.norm(dim=1, keepdim=True)
    return out


def _params(c, **more):
    return lc.lc_default_params(c["d"], c["M1"], c["M2"], use_opq=c["opq"], opq_iters=4, kmeans_iters=10,
                                beta_train_n=50_000, beta_M=c.get("beta_M", 1), beta_K=c.get("beta_K", 256),
                                build_gpu=1, **more)


def _get_index(name: str):
    """The index of that name: trained, filled and resident on the GPU."""
    if name not in _index:
        c = INDEXES[name]
        h = lc.lc_create(_params(c))
        lc.lc_train(h, _vectors(c, c["n_train"], SEED_BASE + 1).float().cpu().numpy())
        xb = _vectors(c, c["n"], SEED_BASE + 2).cpu().numpy()
        (lc.lc_add_u8 if c["kind"] == "sift" else lc.lc_add)(h, xb)
        del xb
        out = [torch.empty((1, 1), dtype=t, device="cuda") for t in (torch.int32, torch.float32)]
        lc.lc_search(h, torch.zeros((1, c["d"]), device="cuda"), 1, lc.lc_default_search_params(1, 8), *out)
        torch.cuda.synchronize()
        _index[name] = h
    return _index[name]


def _get_arrays(name: str) -> dict:
    """The index's arrays (rotation, codebooks, codes, graph) as lc_export lays them out."""
    if name not in _arrays:
        c = INDEXES[name]
        _arrays[name] = lc.lc_export(_get_index(name), c["d"], c["M1"], c["M2"], c.get("beta_M", 1), c.get("beta_K", 256))
    return _arrays[name]


# ------------------------------------------------------------------------------------------
# Cases.  "via": search (lc_search / lc_search_ex on device buffers), host (the same call on
# pinned host buffers), plan (a captured plan), noalloc (the walk without allocation), merge
# (top-k of shards), add (filling an index with the GPU-assisted build).
def _search(name, index, nq, ef, k=10, via="search", beam=1, fp16=False, full=False, table=False, shortlist=0,
            u8=False, uneven=False, max_dist=0):
    return dict(name=name, via=via, index=index, nq=nq, ef=ef, k=k, beam=beam, fp16=fp16, full=full, table=table,
                shortlist=shortlist, u8=u8, uneven=uneven, max_dist=max_dist)


def listed():
    return [
        # one query at a time through a captured plan: interactive latency
        _search("one_query_plan", "mix1m", 1, 64, via="plan", beam=4, fp16=True),
        # a handful of queries with the library's default parameters
        _search("few_queries_default", "mix1m", 16, 64),
        # the small workload end to end from host memory (upload, search, download)
        _search("small_index_host", "mix10k", 1_000, 32, via="host"),
        # the default bench's batch with the default (plain, FP32) search
        _search("mix1m_default", "mix1m", 10_000, 64),
        # the same batch as the autotuner sets it: beam 4, FP16 codebook (the bench's headline)
        _search("mix1m_batched", "mix1m", 10_000, 64, beam=4, fp16=True),
        # large index, large batch, the full-decode walk at a small efSearch (10M / 50M headline)
        _search("mix3m_full_decode", "mix3m", 100_000, 28, beam=4, fp16=True, full=True),
        # large index, wide search: efSearch 128 with the level-1 walk, ragged batch
        _search("mix3m_wide", "mix3m", 20_011, 128, beam=4, fp16=True),
        # SIFT-like uint8 queries, each with its own efSearch out of 16 .. 256
        _search("sift1m_uneven_ef", "sift1m", 20_000, 256, beam=4, fp16=True, u8=True, uneven=True),
        # k = 100 with a product regression codebook: the re-rank of 100 candidates each
        _search("top100_product_codebook", "prod50k", 777, 128, k=100, beam=2),
        # dimensions that no sub-space count divides, ragged batch
        _search("uneven_split", "odd20k", 3_001, 48, k=5),
        # a sharded search's last step: 8 shards' lists of 10,000 queries
        dict(name="merge_8_shards", via="merge", S=8, nq=10_000, k=10),
        # filling an index: 60,000 vectors encoded, linked and assigned their codewords
        dict(name="add_60k", via="add", index="mix1m", n=60_000),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    via = rng.choices(["search", "host", "plan", "noalloc", "merge", "add"], [60, 10, 12, 6, 7, 5])[0]
    if via == "merge":
        S = rng.randint(2, 16)
        return dict(via="merge", S=S, nq=_log(rng, 1, 50_000), k=min(_log(rng, 1, 100), 2048 // S))
    if via == "add":
        return dict(via="add", index=rng.choice(["mix1m", "mix10k", "odd20k"]), n=_log(rng, 5_000, 60_000))
    index = rng.choices(list(INDEXES), [2, 6, 4, 4, 2, 2])[0]
    c = INDEXES[index]
    k = rng.choice([1, 10, 10, 10, 20, 100, rng.randint(2, 100)])
    ef = _log(rng, 16, 256)
    beam, fp16, full = rng.choice([1, 1, 2, 4, 4, 8]), rng.random() < 0.5, rng.random() < 0.25
    table = index in ("mix1m", "mix3m") and not full and rng.random() < 0.08
    if index == "odd20k" and full:
        fp16 = False                                       # the library's own limit
    shortlist = rng.choice([0, 0, 0, 0, 32, -1])
    u8, uneven = c["kind"] == "sift" and rng.random() < 0.7, rng.random() < 0.25
    max_dist = rng.choice([0] * 9 + [400])
    if via == "noalloc":
        beam, fp16, full, table, shortlist, u8, uneven, max_dist = 1, False, False, False, -1, False, False, 0
    # largest batch: no more than the largest listed case's work
    per = max(ef, k) * (3 if full else 1) * (1 if fp16 or not full else 2) + 2 * k
    nq = _log(rng, 1, min(50_000, 2_000_000 // per))
    if via == "plan":
        nq = min(nq, 4_096)
    out = _search("", index, nq, ef, k, via, beam, fp16 or table, full, table, shortlist, u8, uneven, max_dist)
    del out["name"]
    return out


def _search_params(case):
    return lc.lc_default_search_params(
        case["k"], case["ef"], shortlist=case["shortlist"], max_dist=case["max_dist"], walk_full=int(case["full"]),
        mode=lc.LC_MODE_BATCHED if case["beam"] > 1 else lc.LC_MODE_PLAIN, beam=case["beam"],
        lut_prec=lc.LC_LUT_TABLE if case["table"] else lc.LC_LUT_FP16 if case["fp16"] else lc.LC_LUT_FP32)


def _queries(case, seed):
    """Queries of the index's distribution and, for uneven searches, each one's efSearch."""
    c = INDEXES[case["index"]]
    q = _vectors(c, case["nq"], 7_000_000 + seed)
    if not case["u8"]:
        q = q.float()
    ef = None
    if case["uneven"]:
        choices = torch.tensor([e for e in (16, 32, 64, 128, 256) if e <= case["ef"]], dtype=torch.int32, device="cuda")
        ef = choices[torch.randint(len(choices), (case["nq"],), generator=_gen(8_000_000 + seed), device="cuda")]
    return q, ef


def _shard_lists(case, seed):
    """Per-shard results [S][nq][k], each list ascending by (distance, id); a tenth of the
    lists are short (-1, +inf padding), as small shards and capped searches return them."""
    S, nq, k = case["S"], case["nq"], case["k"]
    g = _gen(9_000_000 + seed)
    d = torch.rand((S, nq, k), generator=g, device="cuda").add_(0.2).sort(dim=2).values
    ids = torch.randint(1_000_000, (S, nq, k), generator=g, device="cuda", dtype=torch.int32)
    short = torch.rand((S, nq), generator=g, device="cuda") < 0.1
    have = torch.where(short, torch.randint(k + 1, (S, nq), generator=g, device="cuda"), torch.full((S, nq), k, device="cuda"))
    pad = torch.arange(k, device="cuda") >= have[..., None]
    return ids.masked_fill_(pad, -1).contiguous(), d.masked_fill_(pad, math.inf).contiguous()


def _get_plan(case):
    key = tuple(sorted((x, y) for x, y in case.items() if x != "name"))
    if key not in _plans:
        h, c = _get_index(case["index"]), INDEXES[case["index"]]
        qt = lc.LC_QUERY_U8 if case["u8"] else lc.LC_QUERY_F32
        pl = lc.lc_plan_create(h, case["nq"], _search_params(case), qt, case["uneven"])
        _plans[key] = (pl, lc.lc_plan_tensors(pl, case["nq"], c["d"], case["k"], qt))
    return _plans[key]


def prepare(case, seed):
    via = case["via"]
    if via == "merge":
        ids, dists = _shard_lists(case, seed)
        nq, k = case["nq"], case["k"]
        return dict(via=via, case=case, ids=ids, dists=dists, offsets=[1_000_000 * s for s in range(case["S"])],
                    out=dict(ids=torch.empty((nq, k), dtype=torch.int32, device="cuda"),
                             dists=torch.empty((nq, k), dtype=torch.float32, device="cuda")))
    if via == "add":
        c = INDEXES[case["index"]]
        codec = _get_arrays(case["index"])
        x = _vectors(c, case["n"], 6_000_000 + seed).cpu().numpy()
        return dict(via=via, case=case, codec={n: codec[n] for n in ("R", "C1", "C2", "B")}, x=x)
    h = _get_index(case["index"])
    q, ef = _queries(case, seed)
    nq, k = case["nq"], case["k"]
    st = dict(via=via, case=case, h=h, q=q, ef=ef, sp=_search_params(case))
    if via == "plan":
        st["plan"], st["buf"] = _get_plan(case)
        return st
    pin = dict(pin_memory=True) if via == "host" else dict(device="cuda")
    st["out"] = dict(ids=torch.empty((nq, k), dtype=torch.int32, **pin), dists=torch.empty((nq, k), dtype=torch.float32, **pin),
                     stats=torch.empty((nq, 3), dtype=torch.int32, **pin))
    if via == "host":
        st["q"] = q.cpu().pin_memory()
        st["ef"] = None if ef is None else ef.cpu().pin_memory()
    return st


def run(state):
    case, via = state["case"], state["via"]
    stream = torch.cuda.current_stream()
    if via == "merge":
        o = state["out"]
        lc.lc_merge_topk(state["ids"], state["dists"], case["S"], case["nq"], case["k"], state["offsets"], o["ids"], o["dists"], stream)
        return o
    if via == "add":
        c, a = INDEXES[case["index"]], state["codec"]
        none = np.empty(0, np.int32)
        h = lc.lc_create(_params(c))
        lc.lc_import(h, 0, a["R"], a["C1"], a["C2"], none, none, none, a["B"], none, none, none, -1)
        lc.lc_add(h, state["x"])
        got = lc.lc_export(h, c["d"], c["M1"], c["M2"], c.get("beta_M", 1), c.get("beta_K", 256))
        lc.lc_free(h)
        return {n: got[n] for n in ("codes1", "codes2", "beta", "adj0", "levels", "upper_adj", "ep")}
    if via == "plan":
        b = state["buf"]
        b["q"].copy_(state["q"])
        if state["ef"] is not None:
            b["ef"].copy_(state["ef"])
        lc.lc_plan_run(state["plan"], case["nq"], stream)
        return {n: b[n] for n in ("ids", "dists", "stats")}
    o = state["out"]
    if via == "noalloc":
        lc.lc_search_walk_noalloc(state["h"], state["q"], case["nq"], case["k"], case["ef"], o["ids"], o["dists"], o["stats"], stream)
    elif case["u8"] or case["uneven"]:
        lc.lc_search_ex(state["h"], state["q"], lc.LC_QUERY_U8 if case["u8"] else lc.LC_QUERY_F32, case["nq"], state["sp"],
                        state["ef"], o["ids"], o["dists"], o["stats"], stream)
    else:
        lc.lc_search(state["h"], state["q"], case["nq"], state["sp"], o["ids"], o["dists"], o["stats"], stream)
    return o


def work(case):
    """Bytes and operations of a pass.  A walk has to read the adjacency row of every node it
    expands and the code row of every node it scores; their counts per query depend on the
    data and are put at about what the kernels' own counters average on these indexes (1.15 ef + 4
    expansions; 9.5 new nodes each).  No array is counted more than once over, however many
    queries read it."""
    if case["via"] == "merge":
        n = case["S"] * case["nq"] * case["k"]
        return {"bytes": 8 * n + 8 * case["nq"] * case["k"], "flops": n * math.log2(case["S"])}
    c = INDEXES[case["index"]]
    d, N, M1, M2P = c["d"], c["n"], c["M1"], -(-(c["M2"] + c.get("beta_M", 1)) // 16) * 16
    if case["via"] == "add":
        # each insertion: a search at efConstruction 40 by the full decode, two encodings of
        # 256 centroids per coordinate, and the selection's distances between candidates
        n = case["n"]
        evals = 10 * 46 + 40 * 16
        return {"bytes": n * (4 * d + M1 + c["M2"] + 1 + 128 + 8 * d), "flops": n * (3.0 * d * evals + 4 * 256 * d + 2.0 * d * d)}
    nq, k = case["nq"], case["k"]
    ef = max(case["ef"], k)
    if case["uneven"]:
        ef = sum(max(e, k) for e in (16, 32, 64, 128, 256) if e <= case["ef"]) / sum(e <= case["ef"] for e in (16, 32, 64, 128, 256))
    expand = 1.15 * ef + 4
    score = min(9.5 * expand + 60, N)
    R = 0 if case["shortlist"] < 0 else max(case["shortlist"] or 10, k)
    row = M1 + (M2P if case["full"] else 0)
    read = min(nq * expand * 128, N * 128) + min(nq * score * row, N * row) + min(nq * R * 9 * (M1 + M2P), N * (M1 + M2P))
    io = nq * (d * (1 if case["u8"] else 4) + 8 * k + 12) + 4 * d * d + 2 * 1024 * d
    return {"bytes": read + io, "flops": nq * (3.0 * d * score * (4 / 3 if case["full"] else 1) + 2.0 * d * d + R * d * 30)}


# ------------------------------------------------------------------------------------------
# The same search in 64 bits, in plain torch on the index's arrays: greedy descent of the upper
# levels, best-first walk of level 0 with a result list of ef entries (`beam` expansions a
# step), re-rank of the shortlist by the regression-refined reconstruction.
def _subspace(d, M):
    return np.repeat(np.arange(M), [d // M + (j < d % M) for j in range(M)])


def _decode64(C, codes, d, M, half):
    C = torch.from_numpy(C).cuda()
    C = (C.half() if half else C).double()
    sub = torch.from_numpy(_subspace(d, M)).cuda()
    out = torch.empty((len(codes), d), dtype=torch.float64, device="cuda")
    t = torch.arange(d, device="cuda")
    for a in range(0, len(codes), 1 << 18):
        out[a:a + (1 << 18)] = C[torch.from_numpy(codes[a:a + (1 << 18)]).cuda().long()[:, sub], t]
    return out


def _by_dist_id(D, I, *more):
    """Rows sorted by (distance, id)."""
    o = torch.argsort(I, dim=1, stable=True)
    o = o.gather(1, torch.argsort(D.gather(1, o), dim=1, stable=True))
    return [x.gather(1, o) for x in (D, I) + more]


def _walk64(y, ef, a, V, up_off, beam, tcap):
    """Result lists (distances, ids) [nq][max ef] of the level-0 walk for rotated queries y."""
    dev, nq, N = "cuda", len(y), len(V)
    width = int(ef.max())
    big = torch.iinfo(torch.int64).max

    def dist(rows, ids):                                   # ids [m][w] (-1: none)
        x = V[ids.clamp(min=0)]
        return ((y[rows][:, None] - x) ** 2).sum(-1).masked_fill_(ids < 0, math.inf)

    cur = torch.full((nq,), a["ep"], device=dev)
    every = torch.arange(nq, device=dev)
    dcur = dist(every, cur[:, None])[:, 0]
    for lvl in range(int(a["levels_max"]), 0, -1):
        act = every
        while len(act):
            e = a["upper"][up_off[cur[act]] + lvl - 1].long()
            D = dist(act, e)
            m = D.min(1).values
            best = torch.where(D == m[:, None], e, torch.full_like(e, big)).min(1).values
            move = (m < dcur[act]) | ((m == dcur[act]) & (best < cur[act]))
            act = act[move]
            cur[act], dcur[act] = best[move], m[move]
    seen = torch.zeros((nq, N), dtype=torch.bool, device=dev)
    seen[every, cur] = True
    outD = torch.full((nq, width), math.inf, dtype=torch.float64, device=dev)
    outI = torch.full((nq, width), -1, device=dev)
    rows, D = every, torch.full((nq, width), math.inf, dtype=torch.float64, device=dev)
    I, F = torch.full((nq, width), -1, device=dev), torch.zeros((nq, width), dtype=torch.bool, device=dev)
    D[:, 0], I[:, 0] = dcur, cur
    count = torch.ones(nq, dtype=torch.int64, device=dev)
    pos = torch.arange(width, device=dev)
    while len(rows):
        new = (I >= 0) & ~F
        go = new.any(1) & ((count[rows] < tcap) if tcap else True)
        done = ~go
        outD[rows[done]], outI[rows[done]] = D[done], I[done]
        rows, D, I, F, new = rows[go], D[go], I[go], F[go], new[go]
        if not len(rows):
            break
        rank = new.cumsum(1)
        parts = []
        for b in range(1, beam + 1):
            hit = new & (rank == b)
            c = torch.where(hit.any(1), I.gather(1, hit.int().argmax(1, keepdim=True))[:, 0], torch.full_like(rows, -1))
            e = a["adj0"][c.clamp(min=0)].long()
            e = torch.where((c >= 0)[:, None], e, torch.full_like(e, -1))
            flat = rows[:, None] * N + e.clamp(min=0)
            fresh = (e >= 0) & ~seen.view(-1)[flat]
            seen.view(-1)[flat[fresh]] = True
            parts.append(torch.where(fresh, e, torch.full_like(e, -1)))
        F = F | (new & (rank <= beam))
        e = torch.cat(parts, 1)
        count[rows] += (e >= 0).sum(1)
        D, I, F = (torch.cat(p, 1) for p in ((D, dist(rows, e)), (I, e), (F, torch.zeros_like(e, dtype=torch.bool))))
        D, I, F = _by_dist_id(D, I, F)                     # padding (inf) last
        D, I, F = D[:, :width], I[:, :width], F[:, :width]
        over = pos >= ef[rows][:, None]
        D, I = D.masked_fill(over, math.inf), I.masked_fill(over, -1)
    return outD, outI


def exact(case, seed):
    if case["via"] == "merge":
        ids, dists = _shard_lists(case, seed)
        return {"ids": None, "dists": dists.double().permute(1, 0, 2).reshape(case["nq"], -1).sort(dim=1).values[:, :case["k"]]}
    if case["via"] == "add" or case["table"]:
        return None               # whole numbers only; tables are FP16 by definition
    c, x = INDEXES[case["index"]], _get_arrays(case["index"])
    d, k, half = c["d"], case["k"], case["fp16"]
    q, ef = _queries(case, seed)
    q = q.double() @ torch.from_numpy(x["R"]).cuda().double().T
    ef = torch.full((len(q),), case["ef"], device="cuda") if ef is None else ef.long()
    ef = ef.clamp(min=k)
    a = dict(adj0=torch.from_numpy(x["adj0"]).cuda(), upper=torch.from_numpy(x["upper_adj"]).cuda(), ep=x["ep"],
             levels_max=x["levels"].max())
    lv = torch.from_numpy(x["levels"]).cuda().long()
    up_off = lv.cumsum(0) - lv
    V = _decode64(x["C1"], x["codes1"], d, c["M1"], half)
    if case["full"]:
        V += _decode64(x["C2"], x["codes2"], d, c["M2"], half)
    G = None
    if case["shortlist"] >= 0:
        G = _decode64(x["C1"], x["codes1"], d, c["M1"], False)
        G += _decode64(x["C2"], x["codes2"], d, c["M2"], False)
        bM = c.get("beta_M", 1)
        B = torch.from_numpy(x["B"]).cuda().double().view(bM, -1, 9)
        beta = torch.from_numpy(x["beta"]).cuda().long().view(-1, bM)
        block = torch.from_numpy(_subspace(d, bM)).cuda()
        R = max(case["shortlist"] or 10, k)
    out = torch.full((len(q), k), math.inf, dtype=torch.float64, device="cuda")
    step = max(64, min(4096, int(16e9 / len(V)), int(4e9 / (32 * case["beam"] * d * 8))))
    for s in range(0, len(q), step):
        y = q[s:s + step]
        D, I = _walk64(y, ef[s:s + step], a, V, up_off, case["beam"], case["max_dist"])
        if G is None:
            out[s:s + step, :min(k, D.shape[1])] = D[:, :k]
            continue
        for r0 in range(0, len(y), 256):
            I0 = I[r0:r0 + 256, :R]
            node = I0.clamp(min=0)
            nb = a["adj0"][node][..., :8].long()                                    # [m][R][8]
            P = torch.cat([node[..., None], nb.clamp(min=0)], -1)
            W = B[torch.arange(bM, device="cuda"), beta[node]][..., block, :]       # [m][R][d][9]
            live = torch.cat([torch.ones_like(node[..., None]), (nb >= 0).long()], -1).double()
            yh = torch.einsum("mrtj,mrjt,mrj->mrt", W, G[P], live)
            D0 = ((y[r0:r0 + 256, None] - yh) ** 2).sum(-1).masked_fill_(I0 < 0, math.inf)
            m = min(k, D0.shape[1])
            out[s + r0:s + r0 + len(D0), :m] = D0.sort(dim=1).values[:, :m]
    return {"ids": None, "dists": out.cpu() if case["via"] == "host" else out, "stats": None}

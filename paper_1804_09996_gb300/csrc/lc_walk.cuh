// Device-side definitions of the search walk (shared by the element-type translation units
// lc_walk_f32.cu / lc_walk_f16.cu and by lc_search.cu): kernel arguments, shared-memory
// layouts, the scoring helpers and the walk kernel template, and the host templates that
// configure and launch one instantiation.  Not part of the ABI.
//
// walk_kernel (one warp per query; persistent CTAs take queries from an atomic counter)
//   - y' = R y from the rotation kernel (or rotated here, for the walk without allocation);
//   - the walk distance is the ADC distance ||y' - c1(x)||^2 of Section 4.1: the sum over
//     level-1 sub-spaces j of ||y'^j - C1_j[c_j]||^2, each term computed in FP32 from the
//     codebook C1, which every CTA keeps once in shared memory (a per-query table of the same
//     terms would cost 32-64 KB of shared memory per query in flight); with FQ the distance is
//     to the full two-level decode c1 + c2;
//   - greedy descent of the upper HNSW levels, then best-first search of level 0 with result
//     set W of size ef' (Section 2), in one loop with a single scoring call site.  W is a
//     sorted list of (distance, id) keys with an "expanded" flag: each step expands the best
//     unexpanded member (or the `beam` best) of W, scores all their unvisited neighbours at
//     once (one per lane) and merges them into W keeping the ef' best.  With one expansion
//     per step this expands exactly the nodes, in exactly the order, of the two-set
//     formulation (candidate heap C + result heap W);
//   - exact visited set: 16-byte buckets in shared memory (eight 16-bit tags or four ids each),
//     with a per-warp table in global memory behind it;
//   - writes the shortlist (the R best of W, Section 4.1 two-stage search) or, without
//     refinement, the top-k directly;
//   - ordered search: descent_kernel runs only the upper-level descent of every query and
//     records where it enters level 0; the walk (mode 2) runs the level-0 searches from those
//     entry nodes in the order that order_kernel sorted them (the queries whose entry node is
//     farthest from them first: they tend to walk longest, so the launch no longer ends with a
//     few long walks on an otherwise idle GPU).  Each query's result is the same as in one
//     launch (mode 0): the entry node and its distance are the ones the descent computes.
//
// FP32 walk distance: lane l holds the term of sub-space l (M1 = 32), of l mod 16 (M1 = 16)
// or the sum of sub-spaces l and l + 32 (M1 = 64), each term summed over its coordinates in
// order; the 32 lane values are added pairwise, lanes differing in bit 3 first, then bits 2,
// 1, 0 and 4.  The order is the same for every node, so a node's distance does not depend on
// where or with how many others it is scored.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "lc_device.h"

namespace lc {

#define FULL 0xffffffffu

// ------------------------------------------------------------------------------------------
// Visited set (VisitTab in lc_device.h)
constexpr uint32_t VISIT_MUL = 0x9E3779B1u;

// The storage for an index of n ids, limits of 2^hash_log; want_tag: tags where they fit.
inline VisitTab visit_tab(int64_t n, int hash_log, bool want_tag)
{
    int nb = 1;
    while (nb < 31 && ((int64_t)1 << nb) < n) nb++;
    VisitTab v{};
    for (int h = hash_log; want_tag && h <= hash_log + 1; h++) {
        const int bb = h - 3;                             // 8 tags per bucket
        nb = nb <= bb ? bb + 1 : nb;
        // Tags of more than 16 bits: one more bit of buckets, which with the stash takes an eighth more
        // than ids (2^11 limits: 9 KB and 8) but is probed once and without branches (8.4M ids, limits
        // of 2^10, 10,000 queries: 553 us against 670 with ids, batched FP16 472 and 533).
        if (nb - bb > 16) continue;
        v.tag = 1;
        v.bb = bb;
        v.tb = nb - bb;
        v.mul = VISIT_MUL << (32 - nb);
        v.bytes = 16u << bb;
        v.stash_log = h - 4;
        return v;
    }
    v.bb = hash_log - 2;                                  // 4 ids per bucket
    v.mul = VISIT_MUL;
    v.bytes = 16u << v.bb;
    v.stash_log = -1;
    return v;
}
__host__ __device__ inline size_t visit_bytes(const VisitTab &v)
{
    return v.bytes + (v.stash_log >= 0 ? (size_t)4 << v.stash_log : 0);
}
constexpr uint32_t OWNERS = 512;         // owner bytes of visit_rows (in the staging area, unused then)

// Kernel arguments
struct SplitTab {
    uint16_t off[64];
    uint8_t len[64];
};

struct WalkArgs {
    const float *Q;
    const uint8_t *Q8;     // non-null: the queries are uint8 [nq][d] (Q unused)
    const int32_t *efq;    // non-null: per-query efSearch [nq], clamped to 1..efp
    int k;
    int64_t nq;
    int d;
    const float *Rt, *C1;
    const __half *C1h;     // the same codebook in FP16 (FP16 mode); both in the walk's layout
    const uint8_t *codes1;
    const int32_t *adj0, *upper_off, *upper_adj;
    int32_t ep;
    int max_level;
    int efp;          // ef' = max(ef, k); with efq, the largest any query may use
    int efcap;        // efp rounded up to a multiple of 32
    int R;            // shortlist length (refine) or k (no refinement)
    int refine;
    int beam;         // expansions per step (1: the plain walk)
    int team;         // > 1: warps per query (small batches)
    int tcap;         // > 0: stop once that many level-0 distances were computed
    int hash_log;     // visited-set limits: 2^hash_log entries (see VisitTab) ...
    int spill_log;    // ... and a global table of 2^spill_log entries per query in flight
    VisitTab vt;      // the shared-memory part
    int32_t *spill;
    int64_t spill_tables;  // tables behind spill: one per query (nq) or one per warp
    const float *yq_in;    // non-null: y' = R y computed by rotate_kernel (read, not recomputed)
    float *yq_out;
    int32_t *short_out;
    int32_t *ids_out;
    float *dists_out;
    int32_t *stats_out;
    int32_t *status;
    unsigned long long *counter;   // next query to take (reset to 0 before each launch)
    SplitTab s1;
    // walk on the full two-level decode (kernels instantiated with FQ = true)
    const float *C2;       // [256][d] FP32, read through the cache
    const __half *C2h;     // [256][d] FP16, copied into shared memory
    const uint8_t *codes2b;
    int M2P;
    uint8_t sub2[256];     // level-2 sub-space of each coordinate
    // ordered search: descent_kernel writes each query's level-0 entry node, its walk distance
    // and the upper-level evaluations to seed / seed_d / seed_up.  walk_kernel: 0 = the whole
    // walk; 2 = level 0 only, from those, queue position i taking query order[i] (order may be
    // null: position i is query i)
    int mode;
    const int32_t *order;
    // ordered search with a re-rank: the queries walked so far, in the order they end (done_list
    // [nq], -1 where none yet; done_tail entries taken), for the re-rank that starts meanwhile
    int32_t *done_list, *done_tail;
    const __half *tab;     // table form: the queries' ADC tables [nq][256][M1] (FP16)
    int32_t *seed, *seed_up;
    float *seed_d;
};

// Programmatic dependent launch: the kernels of a search let the next one start as soon as SMs are
// free (pdl_launch), and wait for the previous one to have ended (pdl_wait) once their codebooks
// are in shared memory, before they touch anything it writes.  Each lets the next one start only
// after its own wait, so a kernel that runs has everything of the kernels before the one ahead of it.
// What the kernel ahead writes (entry nodes, distances and order of an ordered search) is read by
// plain loads: the read-only path (__ldg) is for data that no one writes while the reader's grid
// lives, and its loads may be moved ahead of the wait.
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launches kern on st; pdl: it may start before the kernel queued ahead of it has ended.  A launch
// that fails leaves no error behind for the next call to find.
template <typename... P, typename... A>
static cudaError_t launch(void (*kern)(P...), int64_t grid, int block, size_t smem, cudaStream_t st, bool pdl, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

constexpr int MAX_WALK_WARPS = 20;       // warps (queries in flight) per CTA
// threads per CTA an instantiation is compiled for: the full-decode walk and the uneven splits
// keep more per-lane state, so they get registers for 16 warps
__host__ __device__ constexpr int walk_threads(int D1, bool fq)
{
    return (fq || D1 == 0 ? 16 : MAX_WALK_WARPS) * 32;
}

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Shared memory of the walk kernel: the level-1 codebook C1 [256][d] once per CTA, then one
// region per warp.
struct WalkSmem {
    size_t yq, stage, wkey, cand, sel, ctl, slot, hash, total;
};

// Layout of the walk's level-1 codebook in shared memory, chosen so that a lane's sub-space
// term takes few loads and the lanes of one shared-memory phase hit distinct banks:
//  0 (row-major): row c holds centroid c of every sub-space in its own coordinates ([256][d]).
//    Used in FP32 with 3 or 6 dimensions per sub-space (3 j + u mod 32 permutes the lanes)
//    and for non-uniform splits.
//  1 (interleaved): the P values (D1 rounded up to 2, 4 or 8) of centroid c in sub-space j sit
//    at (c * M1 + j) * P: one vector load.  FP32 and FP16 with 2 dimensions, FP16 with 3 and 6.
__host__ __device__ constexpr int walk_layout(int D1, int es)
{
    return D1 == 0 ? 0 : D1 == 2 ? 1 : es == 4 ? 0 : 1;
}
__host__ __device__ constexpr int walk_pad(int D1) { return D1 <= 2 ? 2 : (D1 <= 4 ? 4 : 8); }
// bytes of the level-1 codebook in shared memory (es = 4: FP32, es = 2: FP16)
__host__ __device__ inline size_t walk_c1_bytes(int d, int M1, int D1, size_t es)
{
    const int L = walk_layout(D1, (int)es);
    const size_t n = L == 1 ? (size_t)256 * M1 * walk_pad(D1) : (size_t)256 * d;
    return align_up(n * es, 128);
}
// Layout of the full walk's FP16 level-2 codebook in shared memory: with 3 dimensions per
// level-1 sub-space as the level-1 codebook's layout 1 (the values of a lane's coordinates, for
// every centroid: one 8-byte load), else row-major [256][d].  The FP32 one is row-major.
__host__ __device__ constexpr bool walk_c2_lanes(int D1, int es) { return D1 == 3 && es == 2; }
__host__ __device__ inline size_t walk_c2_bytes(int d, int M1, int D1)
{
    return align_up((walk_c2_lanes(D1, 2) ? (size_t)256 * M1 * walk_pad(D1) : (size_t)256 * d) * 2, 128);
}
// shared memory before the per-warp regions: the walk's level-1 codebook and, for the full
// walk in FP16, the level-2 codebook behind it
__host__ __device__ inline size_t walk_cb_bytes(int d, int M1, int D1, size_t es, bool fq)
{
    return walk_c1_bytes(d, M1, D1, es) + (fq && es == 2 ? walk_c2_bytes(d, M1, D1) : 0);
}
// compile-time sub-space width of the uniform splits 96/16, 96/32 and 128/64 (0: other)
__host__ __device__ constexpr int walk_variant_d1(int variant) { return variant == 1 ? 6 : variant == 2 ? 3 : variant == 3 ? 2 : 0; }
inline int walk_variant(int M1, int d)
{
    return (M1 == 16 && d == 96) ? 1 : (M1 == 32 && d == 96) ? 2 : (M1 == 64 && d == 128) ? 3 : 0;
}

__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(__half x) { return __half2float(x); }

// Nodes whose code rows are staged together.  (64 where a step of the batched walk can have that
// many, so that it waits for global memory once, cost walks in flight: 2,318 against 2,195 us at
// efSearch 128 on 3M vectors.)
constexpr int STAGE_ROWS = 32;

// own_rot: the walk rotates the query itself (y' in shared memory); otherwise y' is read from
// the rotation kernel's output.
__host__ __device__ inline WalkSmem walk_smem(int M1, int d, int efcap, const VisitTab &vt, int beam, bool own_rot,
                                             int m2p = 0)
{
    WalkSmem s;
    size_t o = 0;
    s.yq = o;        o += own_rot ? align_up((size_t)d * 4, 16) : 0;
    s.stage = o;     o += (size_t)STAGE_ROWS * (M1 + m2p);   // level-1 rows, then residual rows
    s.wkey = o;      o += (size_t)efcap * 8;
    s.cand = o;      o += (size_t)32 * beam * 8 + 32;                          // candidates of a step, padded
    s.sel = o;       o += 32;                                                // nodes expanded in a step (at most 8)
    s.ctl = o;       o += 16;                                                // team: query, nodes to score
    s.slot = o;      o += (size_t)32 * beam * 4;
    s.hash = o;      o += visit_bytes(vt);
    s.total = align_up(o, 128);
    return s;
}
// The size by which a search too wide for the shared memory is refused: a walk with a table of
// 32-bit ids of its limits' size, next to codebooks without padding (so that what is accepted does
// not depend on how the walk lays out its memory).
inline size_t walk_nominal_cb_bytes(int d, int M1, bool half, bool full)
{
    const int D1 = walk_variant_d1(walk_variant(M1, d));
    const size_t plain = align_up((size_t)256 * d * 2, 128);
    return (half && D1 == 3 ? plain : walk_c1_bytes(d, M1, D1, half ? 2 : 4)) + (full && half ? plain : 0);
}
inline size_t walk_smem_nominal(int M1, int d, int efcap, int hash_log, int beam, bool own_rot, int m2p = 0)
{
    const size_t st_b = (size_t)32 * (M1 + m2p), cd_b = (size_t)32 * beam * 8;
    return align_up((own_rot ? align_up((size_t)d * 4, 16) : 0) + align_up(std::max(st_b, cd_b), 16) + (size_t)efcap * 8 +
                        align_up((size_t)efcap, 16) + (size_t)32 * beam * 12 + ((size_t)4 << hash_log), 128);
}

// Keys of the result list: distance bits, id, and the "expanded" flag as the lowest bit, which
// never decides an order (ids are distinct).
__device__ __forceinline__ uint64_t walk_key(float dist, int32_t id)
{
    return ((uint64_t)__float_as_uint(dist) << 32) | ((uint32_t)id << 1);
}
__device__ __forceinline__ int32_t walk_id(uint64_t k) { return (int32_t)((uint32_t)k >> 1); }

__device__ __forceinline__ uint64_t make_key(float dist, int32_t id)
{
    return ((uint64_t)__float_as_uint(dist) << 32) | (uint32_t)id;
}
__device__ __forceinline__ int32_t key_id(uint64_t k) { return (int32_t)(uint32_t)(k & 0xffffffffu); }
__device__ __forceinline__ float key_dist(uint64_t k) { return __uint_as_float((uint32_t)(k >> 32)); }

// Smallest (distance, id) of the lanes' pairs (distance bits ~0: none), by two warp reductions.
__device__ __forceinline__ void warp_best(uint32_t dist, uint32_t id, uint32_t *bd, uint32_t *bi)
{
    *bd = __reduce_min_sync(0xffffffffu, dist);
    *bi = __reduce_min_sync(0xffffffffu, dist == *bd ? id : 0xffffffffu);
}

// Lane bits in the order partial distances are combined: 3, 2, 1, 0, then 4.
__host__ __device__ constexpr int comb_bit(int k) { return k < 4 ? 3 - k : 4; }

// The lane bits of the first LS combinations, the first one most significant.
__device__ __forceinline__ int slot_of_lane(int lane, int LS)
{
    int s = 0;
    for (int k = 0; k < LS; k++) s = (s << 1) | ((lane >> comb_bit(k)) & 1);
    return s;
}

// Per-lane geometry: the level-1 sub-space(s) a lane scores and the query's coordinates in
// them.  M1 = 16: sub-space lane & 15 (the two half-warps score different nodes);
// M1 = 32: sub-space lane; M1 = 64: sub-spaces lane and lane + 32.  D1 > 0: every sub-space
// has D1 coordinates (compile-time); D1 = 0: lengths read at run time (uneven splits).
template <int M1, int D1>
struct LaneGeo {
    static constexpr int NSUB = M1 == 64 ? 2 : 1;
    static constexpr int DMAX = D1 > 0 ? D1 : (M1 == 16 ? 16 : (M1 == 32 ? 8 : 4));   // d <= 256
    static constexpr int M2W = (DMAX + 3) / 4;
    int off[NSUB], len[NSUB], j[NSUB];
    int maxlen;                  // longest sub-space (D1 = 0)
    float y[NSUB][DMAX];
    // full walk: the level-2 sub-space of each of the lane's coordinates, four per word, and
    // whether no lane's coordinates touch more than two (warp-uniform)
    uint32_t m2[NSUB][M2W];
    bool two;

    __device__ __forceinline__ int sub2(int k, int u) const { return (m2[k][u / 4] >> (8 * (u % 4))) & 0xff; }

    __device__ __forceinline__ void init(const SplitTab &s1, const float *yrot, const uint8_t *sub2tab, int d, int lane)
    {
        two = true;
        maxlen = D1 > 0 ? D1 : (d + M1 - 1) / M1;
#pragma unroll
        for (int k = 0; k < NSUB; k++) {
            const int jj = M1 == 16 ? (lane & 15) : lane + 32 * k;
            j[k] = jj;
            off[k] = D1 > 0 ? D1 * jj : s1.off[jj];
            len[k] = D1 > 0 ? D1 : s1.len[jj];
#pragma unroll
            for (int u = 0; u < DMAX; u++) y[k][u] = D1 > 0 || u < len[k] ? yrot[off[k] + u] : 0.f;
            if (sub2tab) {
#pragma unroll
                for (int w = 0; w < M2W; w++) m2[k][w] = 0;
#pragma unroll
                for (int u = 0; u < DMAX; u++)
                    if (D1 > 0 || u < len[k]) m2[k][u / 4] |= (uint32_t)sub2tab[off[k] + u] << (8 * (u % 4));
                if (D1 > 2) {
#pragma unroll
                    for (int u = 1; u < D1 - 1; u++)
                        two = two && (sub2(k, u) == sub2(k, 0) || sub2(k, u) == sub2(k, D1 - 1));
                }
            }
        }
        if (D1 > 2) two = __all_sync(FULL, two);
    }
};

__device__ __forceinline__ void half2_to_f(uint32_t w, float &a, float &b)
{
    const __half2 h = *reinterpret_cast<const __half2 *>(&w);
    a = __low2float(h);
    b = __high2float(h);
}

// The coordinates of centroid c in this lane's k-th sub-space, as FP32.
template <int M1, int D1, typename CT>
__device__ __forceinline__ void load_row(const CT *C1s, int d, int c, const LaneGeo<M1, D1> &g, int k,
                                         float (&x)[LaneGeo<M1, D1>::DMAX])
{
    constexpr int DMAX = LaneGeo<M1, D1>::DMAX;
    constexpr int LAYOUT = walk_layout(D1, (int)sizeof(CT));
    if constexpr (LAYOUT == 1) {
        constexpr int P = walk_pad(D1);
        const CT *p = C1s + ((size_t)c * M1 + g.j[k]) * P;
        float t[P];
        if constexpr (sizeof(CT) == 4) {                   // FP32, P = 2
            const float2 f = *reinterpret_cast<const float2 *>(p);
            t[0] = f.x;
            t[1] = f.y;
        } else if constexpr (P == 2) {
            half2_to_f(*reinterpret_cast<const uint32_t *>(p), t[0], t[1]);
        } else if constexpr (P == 4) {
            const uint2 w = *reinterpret_cast<const uint2 *>(p);
            half2_to_f(w.x, t[0], t[1]);
            half2_to_f(w.y, t[2], t[3]);
        } else {
            const uint4 w = *reinterpret_cast<const uint4 *>(p);
            half2_to_f(w.x, t[0], t[1]);
            half2_to_f(w.y, t[2], t[3]);
            half2_to_f(w.z, t[4], t[5]);
            half2_to_f(w.w, t[6], t[7]);
        }
#pragma unroll
        for (int u = 0; u < DMAX; u++) x[u] = t[u];
    } else {
        const CT *row = C1s + c * d + g.off[k];
#pragma unroll
        for (int u = 0; u < DMAX; u++)
            if (D1 > 0 || u < g.maxlen) x[u] = (D1 > 0 || u < g.len[k]) ? to_f(row[u]) : 0.f;
    }
}

__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void unpack2(unsigned long long v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// The sub-space terms of two codes c0, c1 at once with packed FP32x2 arithmetic: each half
// performs the scalar operations in the order of the sub-space's coordinates (same rounding),
// two slots per instruction.
template <int M1, int D1, typename CT>
__device__ __forceinline__ void pair_dist(const CT *C1s, int d, int c0, int c1, const LaneGeo<M1, D1> &g,
                                          int k, float &s0, float &s1)
{
    float x0[LaneGeo<M1, D1>::DMAX], x1[LaneGeo<M1, D1>::DMAX];
    load_row<M1, D1, CT>(C1s, d, c0, g, k, x0);
    load_row<M1, D1, CT>(C1s, d, c1, g, k, x1);
    unsigned long long acc = 0ull;                   // (+0.f, +0.f)
#pragma unroll
    for (int u = 0; u < D1; u++) {
        const unsigned long long yy = pack2(g.y[k][u], g.y[k][u]);
        const unsigned long long cc = pack2(x0[u], x1[u]);
        unsigned long long df;
        asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(df) : "l"(yy), "l"(cc));
        asm("fma.rn.f32x2 %0, %1, %1, %2;" : "=l"(acc) : "l"(df), "l"(acc));
    }
    unpack2(acc, s0, s1);
}

// C2 value for the full walk: FP32 codebooks are read through the cache, FP16 ones from
// shared memory.
__device__ __forceinline__ float c2_at(const float *p) { return __ldg(p); }
__device__ __forceinline__ float c2_at(const __half *p) { return __half2float(*p); }

// The level-2 values of this lane's coordinates for a node whose staged residual row is row2.
// At most two level-2 sub-spaces per lane (TWO): the first and the last coordinate's code, each
// coordinate taking the one of its sub-space; else a code per coordinate.
template <int M1, int D1, typename CT, bool TWO>
__device__ __forceinline__ void load_row2(const CT *C2, int d, const uint8_t *row2, const LaneGeo<M1, D1> &g, int k,
                                          float (&z)[LaneGeo<M1, D1>::DMAX])
{
    constexpr int DMAX = LaneGeo<M1, D1>::DMAX;
    if constexpr (walk_c2_lanes(D1, (int)sizeof(CT))) {
        auto at = [&](int c) { return *reinterpret_cast<const uint2 *>(C2 + ((size_t)c * M1 + g.j[k]) * 4); };
        const uint2 wa = at(row2[g.sub2(k, 0)]), wb = at(row2[g.sub2(k, 2)]);
        // coordinates 0 and 1 share a word, as do 2 and the padding
        float t;
        half2_to_f(wa.x, z[0], t);
        half2_to_f(wb.y, z[2], t);
        if (TWO) half2_to_f(g.sub2(k, 1) == g.sub2(k, 0) ? wa.x : wb.x, t, z[1]);
        else half2_to_f(at(row2[g.sub2(k, 1)]).x, t, z[1]);
    } else if constexpr (TWO && D1 > 0) {
        const int ca = row2[g.sub2(k, 0)], cb = row2[g.sub2(k, D1 - 1)];
        const CT *pa = C2 + (size_t)ca * d + g.off[k], *pb = C2 + (size_t)cb * d + g.off[k];
#pragma unroll
        for (int u = 0; u < D1; u++) z[u] = c2_at((g.sub2(k, u) == g.sub2(k, 0) ? pa : pb) + u);
    } else {
#pragma unroll
        for (int u = 0; u < DMAX; u++)
            z[u] = D1 > 0 || u < g.len[k] ? c2_at(C2 + (size_t)row2[g.sub2(k, u)] * d + g.off[k] + u) : 0.f;
    }
}

// Full walk, two nodes at once: sums over this lane's coordinates t of
// (y'_t - (C1[c1][t] + C2[c2_m(t)][t]))^2 in the order of the coordinates, m(t) the level-2
// sub-space of t, in packed FP32 arithmetic (the scalar operations' roundings).
template <int M1, int D1, typename CT, bool TWO>
__device__ __forceinline__ void pair_full(const CT *C1s, const CT *C2, int d, int c0, int c1, const uint8_t *ra,
                                          const uint8_t *rb, const LaneGeo<M1, D1> &g, int k, float &s0, float &s1)
{
    constexpr int DMAX = LaneGeo<M1, D1>::DMAX;
    unsigned long long acc = 0ull;
    auto add = [&](int u, float x0, float x1, float z0, float z1) {
        const unsigned long long yy = pack2(g.y[k][u], g.y[k][u]);
        unsigned long long v, df;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(pack2(x0, x1)), "l"(pack2(z0, z1)));
        asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(df) : "l"(yy), "l"(v));
        asm("fma.rn.f32x2 %0, %1, %1, %2;" : "=l"(acc) : "l"(df), "l"(acc));
    };
    if constexpr (DMAX <= 6) {
        float x0[DMAX], x1[DMAX], z0[DMAX], z1[DMAX];
        load_row<M1, D1, CT>(C1s, d, c0, g, k, x0);
        load_row<M1, D1, CT>(C1s, d, c1, g, k, x1);
        load_row2<M1, D1, CT, TWO>(C2, d, ra, g, k, z0);
        load_row2<M1, D1, CT, TWO>(C2, d, rb, g, k, z1);
#pragma unroll
        for (int u = 0; u < DMAX; u++)
            if (D1 > 0 || u < g.maxlen) add(u, x0[u], x1[u], z0[u], z1[u]);
    } else {
        // (uneven splits) coordinate by coordinate: rows of up to 16 coordinates would not fit the
        // registers; those past the lane's own length count 0
        const CT *p0 = C1s + c0 * d + g.off[k], *p1 = C1s + c1 * d + g.off[k], *q = C2 + g.off[k];
#pragma unroll
        for (int u = 0; u < DMAX; u++) {
            if (u >= g.maxlen) break;
            if (u < g.len[k])
                add(u, to_f(p0[u]), to_f(p1[u]), c2_at(q + (int)ra[g.sub2(k, u)] * d + u), c2_at(q + (int)rb[g.sub2(k, u)] * d + u));
        }
    }
    unpack2(acc, s0, s1);
}

// Scoring works on blocks of slot_block staged nodes, eight values per lane, summed over the
// lanes differing in bits 3, 2 and 1 by a reduce-scatter (seven shuffles), then over bit 0 and,
// with 32 sub-space lanes, bit 4 (one total left per lane).  With M1 = 16 the two half-warps
// score different nodes, so a block has 16.  Lane order: with s3 = the lane's bits 3, 2, 1 (bit
// 3 first), value i of a lane belongs to node i ^ s3, so at each level every lane keeps its
// lower half and sends its upper one, without selects, and ends with node s3.  A lane keeps
// the total of one node per chunk of 32: node chunk_slot(lane).
// Blocks of eight in a rolled loop, and not one unrolled pass over 16 or 32 nodes: fewer
// registers (20 warps per SM leave 102 each), no work past the last block, and code that stays in
// the instruction cache (the unrolled full-decode scoring lost two thirds of its stall cycles
// waiting for instructions).
__host__ __device__ constexpr int slot_block(int M1) { return M1 == 16 ? 16 : 8; }

// Full walk: whether C2 is read only for nodes that are there (see block_terms): in FP32, but for
// 96/32, whose whole blocks of eight keep more reads in flight: 338 against 391 us at 1,000 queries
// and 70.4 against 71.8 ms for a GPU-assisted add of 40,000 vectors (from some 1,500 queries on node
// by node is faster: 588 and 483 us at 2,000, 3,816 and 2,320 at 20,000).
__host__ __device__ constexpr bool node_by_node(int M1, int D1, int es) { return es == 4 && !(M1 == 32 && D1 == 3); }

template <int M1>
__device__ __forceinline__ int lane_block(int lane)
{
    return M1 == 16 ? (lane & 1) : ((lane & 1) | ((lane >> 3) & 2));
}

template <int M1>
__device__ __forceinline__ int chunk_slot(int lane)
{
    const int s3 = slot_of_lane(lane, 3);
    return lane_block<M1>(lane) * slot_block(M1) + (M1 == 16 ? 2 * s3 + (lane >> 4) : s3);
}

// The eight values of this lane for the block staged at `stage` (residual rows at `stage2`), whose
// first n >= 1 slots hold nodes (n may be more than a block).  The slots behind them hold stale
// bytes, which are codes all the same; their totals are not used.  TAB: C1s is the query's ADC table [256][M1] (FP16): the term of code c is its entry
// [c][lane].
template <int M1, int D1, typename CT, bool FQ, bool TAB, bool TWO>
__device__ __forceinline__ void block_terms(const CT *C1s, const uint8_t *stage, const uint8_t *stage2, int n, int d,
                                            const LaneGeo<M1, D1> &g, int lane, const CT *C2, int M2P, float (&v)[8])
{
    // node of value i for this lane, and its code in sub-space j
    const int h = M1 == 16 ? lane >> 4 : 0, j = M1 == 16 ? lane & 15 : lane, s3 = slot_of_lane(lane, 3);
    auto slot = [&](int i) { return M1 == 16 ? 2 * (i ^ s3) + h : i ^ s3; };
    if constexpr (TAB) {
        static_assert(M1 == 32 && !FQ, "the table form is built for 32 sub-spaces");
#pragma unroll
        for (int i = 0; i < 8; i++) v[i] = to_f(C1s[(int)stage[slot(i) * M1 + lane] * M1 + lane]);
    } else if constexpr (FQ && node_by_node(M1, D1, (int)sizeof(CT))) {
        // C2 comes through the cache, which bounds this form, so only nodes that are there read it: the
        // lanes take the same two nodes at a time (with M1 = 16 two per half-warp), up to the last, and
        // the values change places afterwards.  A step has about six new nodes, and a block's other
        // slots would read C2 for nothing, each lane for another node (20,000 queries, ef 64, on 20,000
        // x 96 with M1 = 16: 6,894 us with whole blocks, 2,136 now; x 128 with M1 = 64: 6,532 and 3,902;
        // x 100 with M1 = 16, where whole blocks also spill: 11,671 and 3,791).
        auto node = [&](int i) { return min(M1 == 16 ? 2 * i + h : i, n - 1); };
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            v[i] = v[i + 1] = 0.f;
            if ((M1 == 16 ? 2 * i : i) >= n) continue;
            const uint8_t *ca = stage + node(i) * M1, *cb = stage + node(i + 1) * M1;
            const uint8_t *ra = stage2 + node(i) * M2P, *rb = stage2 + node(i + 1) * M2P;
            pair_full<M1, D1, CT, TWO>(C1s, C2, d, ca[j], cb[j], ra, rb, g, 0, v[i], v[i + 1]);
            if (M1 == 64) {
                float u0, u1;
                pair_full<M1, D1, CT, TWO>(C1s, C2, d, ca[32 + j], cb[32 + j], ra, rb, g, LaneGeo<M1, D1>::NSUB - 1, u0, u1);
                v[i] += u0;
                v[i + 1] += u1;
            }
        }
#pragma unroll
        for (int b = 1; b < 8; b *= 2)
#pragma unroll
            for (int i = 0; i < 8; i++)
                if (!(i & b)) {
                    const float lo = v[i], hi = v[i | b];
                    v[i] = s3 & b ? hi : lo;
                    v[i | b] = s3 & b ? lo : hi;
                }
    } else if constexpr (FQ) {
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const uint8_t *ca = stage + slot(i) * M1, *cb = stage + slot(i + 1) * M1;
            const uint8_t *ra = stage2 + slot(i) * M2P, *rb = stage2 + slot(i + 1) * M2P;
            pair_full<M1, D1, CT, TWO>(C1s, C2, d, ca[j], cb[j], ra, rb, g, 0, v[i], v[i + 1]);
            if (M1 == 64) {
                float u0, u1;
                pair_full<M1, D1, CT, TWO>(C1s, C2, d, ca[32 + j], cb[32 + j], ra, rb, g, LaneGeo<M1, D1>::NSUB - 1, u0, u1);
                v[i] += u0;
                v[i + 1] += u1;
            }
        }
    } else if constexpr (D1 > 0) {
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const uint8_t *ca = stage + slot(i) * M1, *cb = stage + slot(i + 1) * M1;
            pair_dist<M1, D1, CT>(C1s, d, ca[j], cb[j], g, 0, v[i], v[i + 1]);
            if (M1 == 64) {
                float u0, u1;
                pair_dist<M1, D1, CT>(C1s, d, ca[32 + j], cb[32 + j], g, LaneGeo<M1, D1>::NSUB - 1, u0, u1);
                v[i] += u0;
                v[i + 1] += u1;
            }
        }
    } else {
        // uneven split: coordinate by coordinate over the eight nodes; those past a lane's own
        // length count 0 (fma(0, 0, s) = s)
#pragma unroll
        for (int k = 0; k < LaneGeo<M1, D1>::NSUB; k++) {
            const CT *row[8];
            float t[8];
#pragma unroll
            for (int i = 0; i < 8; i++) {
                row[i] = C1s + (int)stage[slot(i) * M1 + 32 * k + j] * d + g.off[k];
                t[i] = 0.f;
            }
#pragma unroll
            for (int u = 0; u < LaneGeo<M1, D1>::DMAX; u++) {
                if (u >= g.maxlen) break;
                const bool in = u < g.len[k];
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    const float df = in ? g.y[k][u] - to_f(row[i][in ? u : 0]) : 0.f;
                    t[i] = fmaf(df, df, t[i]);
                }
            }
#pragma unroll
            for (int i = 0; i < 8; i++) v[i] = k ? v[i] + t[i] : t[i];
        }
    }
}

// Sum of a block's eight values over the sub-space lanes, in the fixed order (bits 3, 2, 1, 0,
// then 4); with M1 = 16 the half-warps hold different nodes (bit 4 would add their zeros).
template <int M1>
__device__ __forceinline__ float reduce_block(float (&v)[8])
{
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const int half = 4 >> k;
#pragma unroll
        for (int i = 0; i < half; i++) v[i] += __shfl_xor_sync(FULL, v[i + half], 1 << comb_bit(k));
    }
    float r = v[0];
    r += __shfl_xor_sync(FULL, r, 1);
    if (M1 != 16) r += __shfl_xor_sync(FULL, r, 16);
    return r;
}

// Copies bytes (a multiple of 16) into shared memory with every load of a thread in flight at
// once (cp.async), so a block of a single warp does not wait for each; copy_wait before a
// barrier.
__device__ __forceinline__ void copy16(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void copy16_l2(void *dst, const void *src)      // not through L1
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void copy_async(void *dst, const void *src, size_t bytes)
{
#pragma unroll 4
    for (uint32_t i = threadIdx.x * 16; i < bytes; i += blockDim.x * 16)
        copy16(static_cast<char *>(dst) + i, static_cast<const char *>(src) + i);
}

// Code rows of the n <= STAGE_ROWS nodes in slot[0..n) into the staging area: the level-1 rows,
// then, for the full walk, the residual rows behind all of them.
template <int M1, bool FQ>
__device__ __forceinline__ void stage_codes(uint8_t *stage, const uint8_t *codes1, const uint8_t *codes2b, int M2P,
                                            const int32_t *slot, int n, int lane)
{
    __syncwarp();                                        // slot written, the staged rows read
    if (lane < n) {
        const int64_t v = slot[lane];
#pragma unroll
        for (int u = 0; u < M1 / 16; u++) copy16(stage + lane * M1 + 16 * u, codes1 + v * M1 + 16 * u);
        if constexpr (FQ)
            for (int u = 0; u < M2P; u += 16) copy16(stage + STAGE_ROWS * M1 + lane * M2P + u, codes2b + v * M2P + u);
    }
    copy_wait();
    __syncwarp();
}

// Walk distances of nf staged nodes (1 <= nf <= 32), block by block; PAIR: two blocks at once
// where there are two (their chains of shared-memory reads and shuffles overlap: 2 % for the
// batched walk, whose chunks are full; for the plain one the extra code costs more).  Returns the
// total of node chunk_slot(lane) (undefined from nf on).
template <int M1, int D1, typename CT, bool FQ, bool TAB, bool PAIR>
__device__ __forceinline__ float score_staged(const CT *C1s, const uint8_t *stage, const uint8_t *stage2, int nf, int d,
                                              const LaneGeo<M1, D1> &g, int lane, const CT *C2, int M2P)
{
    constexpr int SB = slot_block(M1);
    const int mine = lane_block<M1>(lane);
    float r = 0.f;
    auto terms = [&](int b, float (&v)[8]) {
        const uint8_t *st = stage + b * SB * M1, *st2 = stage2 + b * SB * M2P;
        const int n = nf - b * SB;
        if (FQ && D1 > 2 && !g.two) block_terms<M1, D1, CT, FQ, TAB, false>(C1s, st, st2, n, d, g, lane, C2, M2P, v);
        else block_terms<M1, D1, CT, FQ, TAB, true>(C1s, st, st2, n, d, g, lane, C2, M2P, v);
    };
#pragma unroll 1
    for (int b = 0; b * SB < nf; b += PAIR ? 2 : 1) {
        float v[8];
        if (PAIR && (b + 1) * SB < nf) {
            float v1[8];
            terms(b, v);
            terms(b + 1, v1);
            const float t = reduce_block<M1>(v), t1 = reduce_block<M1>(v1);
            if (b == mine) r = t;
            if (b + 1 == mine) r = t1;
        } else {
            terms(b, v);
            const float t = reduce_block<M1>(v);
            if (b == mine) r = t;
        }
    }
    return r;
}

__device__ __forceinline__ uint32_t hash32(int32_t e)
{
    uint32_t x = (uint32_t)e * 0x9E3779B1u;
    return x ^ (x >> 15);
}

// Ids counted to the shared part of the visited set before the walk counts to the global one.
__host__ __device__ constexpr int shared_visited_cap(int H) { return H - H / 4; }

// Open addressing with triangular probing (the p-th probe of id e at hash(e) + p(p+1)/2, mod the
// power-of-two size, visits every entry), -1 = empty.  table_insert: true if e was not there.
__device__ __forceinline__ bool table_insert(int32_t e, int32_t *tab, int log, int shift)
{
    const uint32_t m = (1u << log) - 1;
    uint32_t h = (hash32(e) >> shift) & m;
#pragma unroll 1
    for (uint32_t p = 0; p <= m; p++) {
        const int32_t old = atomicCAS(tab + h, -1, e);
        if (old == -1) return true;
        if (old == e) return false;
        h = (h + p + 1) & m;
    }
    return false;                  // unreachable: the table is never full
}
__device__ __forceinline__ bool table_find(int32_t e, const int32_t *tab, int log, int shift)
{
    const uint32_t m = (1u << log) - 1;
    uint32_t h = (hash32(e) >> shift) & m;
#pragma unroll 1
    for (uint32_t p = 0; p <= m; p++) {
        const int32_t v = tab[h];
        if (v == e) return true;
        if (v == -1) return false;
        h = (h + p + 1) & m;
    }
    return false;
}

// A halfword of v that is zero, as a mask with bit 15 or 31 set; exact for "is there one", and
// for which ones when the zero halfwords are the high ones of the word (as empty entries are:
// a bucket fills from its first entry on).
__device__ __forceinline__ uint32_t zero16(uint32_t v) { return (v - 0x00010001u) & ~v & 0x80008000u; }

// Shared-memory accesses by 32-bit address.
__device__ __forceinline__ uint4 lds128(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
// One look at the bucket of id e (e < 0: no id): SEEN; INSERT: it is not there, *at is the
// shared-memory address of the first empty entry and *bucket the bucket;
// OVERFLOW: it is not there and cannot go there.  No branches with tags: a warp's lanes mostly
// differ in the outcome, and each divergent branch costs more than computing all of it.
enum { VISIT_SEEN = 0, VISIT_INSERT = 1, VISIT_OVERFLOW = 2 };

__device__ __forceinline__ int probe_tags(const VisitTab &vt, uint32_t tab, int32_t e, uint32_t *at, uint32_t *bucket,
                                          uint32_t *neu)
{
    const uint32_t y = (uint32_t)e * vt.mul;
    const uint32_t b = y >> (32 - vt.bb);
    const uint4 w = lds128(tab + (b << 4));
    // 0 is never an entry: with 16-bit tags the ids of tag 0 always take the overflow
    const uint32_t tg = ((y << vt.bb) >> (32 - vt.tb)) + (vt.tb < 16);
    const uint32_t tt = __byte_perm(tg, 0, 0x1010);
    const uint32_t has = (zero16(w.x ^ tt) | zero16(w.y ^ tt)) | (zero16(w.z ^ tt) | zero16(w.w ^ tt));
    const uint32_t room = __popc((zero16(w.x) | (zero16(w.y) >> 1)) | ((zero16(w.z) >> 2) | (zero16(w.w) >> 3)));
    *at = tab + (b << 4) + 16 - 2 * room;                // entries fill in order
    *bucket = b;
    *neu = tg;
    const int r = room == 0 || tg == 0 ? VISIT_OVERFLOW : VISIT_INSERT;
    return e < 0 || (has != 0 && tg != 0) ? VISIT_SEEN : r;
}

// With ids in the buckets, a full one continuing in the next; closed: nothing is inserted.
__device__ __forceinline__ int probe_ids(const VisitTab &vt, uint32_t tab, int32_t e, bool closed, uint32_t *at,
                                         uint32_t *bucket, uint32_t *neu)
{
    const uint32_t v = (uint32_t)e + 1;
    uint32_t b = ((uint32_t)e * vt.mul) >> (32 - vt.bb);
    *neu = v;
    if (e < 0) return VISIT_SEEN;
    for (;;) {                                           // ends: the table is at most three quarters full
        const uint4 w = lds128(tab + b * 16);
        if (w.x == v || w.y == v || w.z == v || w.w == v) return VISIT_SEEN;
        if (w.w == 0) {
            *at = tab + b * 16 + 4 * ((w.x != 0) + (w.y != 0) + (w.z != 0));
            *bucket = b;
            return closed ? VISIT_OVERFLOW : VISIT_INSERT;
        }
        b = (b + 1) & ((1u << vt.bb) - 1);
    }
}

template <bool TAG>
__device__ __forceinline__ int bucket_probe(const VisitTab &vt, uint32_t tab, int32_t e, bool closed, uint32_t *at,
                                            uint32_t *bucket, uint32_t *neu)
{
    if (TAG) return probe_tags(vt, tab, e, at, bucket, neu);
    return probe_ids(vt, tab, e, closed, at, bucket, neu);
}
template <bool TAG>
__device__ __forceinline__ void bucket_store(uint32_t at, uint32_t v)
{
    if (TAG) asm volatile("st.shared.u16 [%0], %1;" ::"r"(at), "h"((unsigned short)v) : "memory");
    else asm volatile("st.shared.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}

// State of a query's visited set (warp-uniform).
struct Visited {
    unsigned char *tab;            // buckets
    uint32_t tab_s, own_s;         // shared-memory addresses of the buckets and the owner bytes
    int32_t *stash, *spill;        // overflow of the buckets: shared, then global
    int hcount, scount;            // ids counted to the shared and to the global limit
    int ocount;                    // ids in the stash
    bool spilled, stash_full;      // counting to the global limit; overflow goes to spill

    __device__ __forceinline__ void clear(const VisitTab &vt, int lane)
    {
#pragma unroll 1
        for (uint32_t i = lane; i < vt.bytes / 16; i += 32) reinterpret_cast<uint4 *>(tab)[i] = make_uint4(0, 0, 0, 0);
        if (vt.stash_log >= 0)
#pragma unroll 1
            for (int i = lane; i < (1 << vt.stash_log) / 4; i += 32)
                reinterpret_cast<int4 *>(stash)[i] = make_int4(-1, -1, -1, -1);
        hcount = scount = ocount = 0;
        spilled = stash_full = false;
    }
    // the level-0 entry node (one lane, into the cleared set)
    __device__ __forceinline__ void first(const VisitTab &vt, int32_t e, int lane)
    {
        hcount = 1;
        if (lane == 0) {
            uint32_t at = 0, b = 0, nw = 0;
            const int r = vt.tag ? probe_tags(vt, tab_s, e, &at, &b, &nw) : probe_ids(vt, tab_s, e, false, &at, &b, &nw);
            if (r != VISIT_INSERT) stash[hash32(e) & ((1 << vt.stash_log) - 1)] = e;
            else if (vt.tag) bucket_store<true>(at, nw);
            else bucket_store<false>(at, nw);
        }
        ocount = 1;                                      // (at most)
    }
};

// Rare parts of the visited test, out of the way of the walk's code.  (Scalar arguments: a
// reference would put the walk's state in memory.)
static __device__ __noinline__ void clear_spill(int32_t *spill, int spill_log, int lane)
{
#pragma unroll 1
    for (int i = lane; i < (1 << spill_log) / 4; i += 32)
        reinterpret_cast<int4 *>(spill)[i] = make_int4(-1, -1, -1, -1);
    __syncwarp();
}
// Id e into the overflow tables: the stash (stash_log >= 0) while it takes ids, else the global
// table; true if it was in neither.
static __device__ __noinline__ bool overflow_insert(int32_t e, int32_t *stash, int stash_log, bool stash_full, int32_t *spill,
                                             int spill_log)
{
    if (stash_log >= 0) {
        if (!stash_full) return table_insert(e, stash, stash_log, 0);
        if (table_find(e, stash, stash_log, 0)) return false;
    }
    return table_insert(e, spill, spill_log, 3);
}

// Tests and inserts one id per lane (e < 0: none) into the visited set; appends those that were not
// there to slot[ns...] and returns their number.  Insertion without atomics (one warp owns the
// table, and a compare-and-swap on random shared addresses takes 180 cycles alone and 1,024 with 16
// warps per SM): in each round the lanes that want to insert write their lane to their bucket's
// owner byte (shared by buckets OWNERS apart), and the one that is read back stores its entry; the
// others look again, so an id that two lanes hold is fresh once.
template <bool TAG>
__device__ __forceinline__ int visit_ids(Visited &V, const VisitTab &vt, int spill_log, int32_t e, int32_t *slot, int ns,
                                         int lane)
{
    const bool closed = !TAG && V.spilled;
    int32_t todo = e;
    bool fresh = false, over = false;
    do {
        uint32_t at, own = 0, nw;
        const int r = bucket_probe<TAG>(vt, V.tab_s, todo, closed, &at, &own, &nw);
        over |= r == VISIT_OVERFLOW;
        if (r != VISIT_INSERT) todo = -1;
        own = V.own_s + (own & (OWNERS - 1));
        if (todo >= 0) asm volatile("st.shared.u8 [%0], %1;" ::"r"(own), "r"(lane) : "memory");
        __syncwarp();
        uint32_t c = 0xff;
        if (todo >= 0) asm volatile("ld.shared.u8 %0, [%1];" : "=r"(c) : "r"(own) : "memory");
        __syncwarp();
        if (c == (uint32_t)lane) {
            bucket_store<TAG>(at, nw);
            fresh = true;
            todo = -1;
        }
        __syncwarp();
    } while (__any_sync(FULL, todo >= 0));
    const unsigned ov = __ballot_sync(FULL, over);
    if (ov) {
        if (TAG && !V.stash_full && V.ocount + __popc(ov) > shared_visited_cap(1 << vt.stash_log)) {
            V.stash_full = true;
            clear_spill(V.spill, spill_log, lane);
        }
        if (over) fresh = overflow_insert(e, V.stash, TAG ? vt.stash_log : -1, V.stash_full, V.spill, spill_log);
        if (!V.stash_full) V.ocount += __popc(ov);       // (at most)
        __syncwarp();
    }
    const unsigned m = __ballot_sync(FULL, fresh);
    if (fresh) slot[ns + __popc(m & ((1u << lane) - 1))] = e;
    return __popc(m);
}

// The same for the adjacency rows of cnt <= 4 nodes (ev[u]: this lane's entry of row u, -1: none);
// the caller has checked the limits for all rows.  The four rows go through one round together;
// the few ids that lose their bucket in it (four rows bring about 36 new ids, some of them twice,
// to 256 buckets) or find it full are gathered behind the fresh ones, at the end of the rows' part
// of slot[], and go through visit_ids: a second round of all four rows would be mostly idle
// (10k queries, beam 4: 650 -> 610 us).
template <bool TAG>
__device__ __forceinline__ int visit_rows(Visited &V, const VisitTab &vt, int spill_log, const int32_t (&ev)[4], int cnt,
                                          int32_t *slot, int ns, int lane)
{
    const bool closed = !TAG && V.spilled;
    const unsigned lt_mask = (1u << lane) - 1;
    uint32_t at[4], own[4] = {}, nw[4];
    int r[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
        r[u] = bucket_probe<TAG>(vt, V.tab_s, ev[u], closed, &at[u], &own[u], &nw[u]);
        own[u] = V.own_s + (own[u] & (OWNERS - 1));
    }
#pragma unroll
    for (int u = 0; u < 4; u++)
        if (r[u] == VISIT_INSERT) asm volatile("st.shared.u8 [%0], %1;" ::"r"(own[u]), "r"(lane | (u << 5)) : "memory");
    __syncwarp();
    bool won[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
        uint32_t c = 0xff;
        if (r[u] == VISIT_INSERT) asm volatile("ld.shared.u8 %0, [%1];" : "=r"(c) : "r"(own[u]) : "memory");
        won[u] = c == (uint32_t)(lane | (u << 5));
    }
    __syncwarp();
    int n = ns, end = ns + 32 * cnt;
#pragma unroll
    for (int u = 0; u < 4; u++) {
        const unsigned m = __ballot_sync(FULL, won[u]), l = __ballot_sync(FULL, r[u] != VISIT_SEEN && !won[u]);
        if (won[u]) {
            bucket_store<TAG>(at[u], nw[u]);
            slot[n + __popc(m & lt_mask)] = ev[u];
        } else if (r[u] != VISIT_SEEN) {
            slot[end - 1 - __popc(l & lt_mask)] = ev[u];
        }
        n += __popc(m);
        end -= __popc(l);
    }
    __syncwarp();
#pragma unroll 1
    for (int c = end; c < ns + 32 * cnt; c += 32) {      // (n <= end throughout: each id is listed once)
        const int32_t e = c + lane < ns + 32 * cnt ? slot[c + lane] : -1;
        __syncwarp();
        n += visit_ids<TAG>(V, vt, spill_log, e, slot, n, lane);
    }
    return n - ns;
}

// The rows of nodes sel[0..cnt) with ids in the buckets (very large indexes, table sizes asked for).
static __device__ __noinline__ int visit_rows_ids(uint32_t tab, uint32_t owners, int bb, int32_t *spill, int spill_log,
                                                  bool spilled, const int32_t *adj0, const int32_t *sel, int cnt,
                                                  int32_t *slot, int ns, int lane)
{
    VisitTab vt{};
    vt.bb = bb;
    vt.mul = VISIT_MUL;
    vt.stash_log = -1;
    Visited V{};
    V.tab_s = tab;
    V.own_s = owners;
    V.spill = spill;
    V.spilled = spilled;
    int32_t ev[4];
#pragma unroll
    for (int u = 0; u < 4; u++) ev[u] = u < cnt ? __ldg(adj0 + (int64_t)sel[u] * DEG + lane) : -1;
    return visit_rows<false>(V, vt, spill_log, ev, cnt, slot, ns, lane);
}

// Members of the sorted list W (wn keys) below k: four-way search, three reads a step in flight
// together (a binary search would wait for twice as many dependent reads).
__device__ __forceinline__ int members_below(const uint64_t *W, int wn, uint64_t k)
{
    int lo = 0;
#pragma unroll 1
    for (int s = 1 << ((31 - __clz(wn)) & ~1); s; s >>= 2) {
        int c = 0;
#pragma unroll
        for (int j = 1; j < 4; j++) {
            const int i = lo + j * s - 1;
            if (i < wn) c += W[i] < k;
        }
        lo += c * s;
    }
    return lo;
}

// Merges the nc candidates of a step (keys cand[0..nc), distinct, in any order; room for three
// more) into the sorted list W of wn keys in place, keeping the efp smallest; returns the new
// length and in *first_new the lowest place a candidate took.  A candidate's place is the number
// of candidates and of members below it (a count over the candidates, a search in W).  The
// places not taken hold the members in order, so from the last 32 places down every place finds
// its member from the number of candidates placed below it (one OR over the warp), and no member
// searches; members only move up, so the places below are still the old ones.  Up to 32
// candidates (nearly every step; always unless MANY) stay in registers; else place[] keeps their
// places.
template <bool MANY>
__device__ __forceinline__ int merge_step(uint64_t *W, int wn, int efp, uint64_t *cand, int nc, int32_t *place, int lane,
                                          int *first_new)
{
    const int wn2 = min(efp, wn + nc);
    if (lane < 3) cand[nc + lane] = ~0ull;               // the count below takes four at a time
    __syncwarp();
    const bool one = !MANY || nc <= 32;
    int at = 0x7fffffff, lowest = 0x7fffffff;
    uint64_t k = 0;
#pragma unroll 1
    for (int m0 = lane; m0 < nc; m0 += 32) {
        k = cand[m0];
        at = members_below(W, wn, k);
#pragma unroll 1
        for (int m = 0; m < nc; m += 4) {
            const ulonglong2 c0 = *reinterpret_cast<const ulonglong2 *>(cand + m);
            const ulonglong2 c1 = *reinterpret_cast<const ulonglong2 *>(cand + m + 2);
            at += (c0.x < k) + (c0.y < k) + (c1.x < k) + (c1.y < k);
        }
        if (!one) place[m0] = at;
        lowest = min(lowest, at);
    }
    lowest = (int)__reduce_min_sync(FULL, (unsigned)lowest);
    *first_new = lowest;
    int above = one ? __popc(__ballot_sync(FULL, at < wn2)) : 0;     // candidates placed before the end of the chunk
    if (!one) {
#pragma unroll 1
        for (int m0 = 0; m0 < nc; m0 += 32) above += __popc(__ballot_sync(FULL, m0 + lane < nc && place[m0 + lane] < wn2));
    }
#pragma unroll 1
    for (int c0 = (wn2 - 1) & ~31; c0 >= (lowest & ~31); c0 -= 32) {
        unsigned mine = 0;
        if (one) {
            if (at >= c0 && at < min(c0 + 32, wn2)) mine = 1u << (at - c0);
        } else {
#pragma unroll 1
            for (int m0 = lane; m0 < nc; m0 += 32) {
                const int o = place[m0] - c0;
                if (o >= 0 && o < min(32, wn2 - c0)) mine |= 1u << o;
            }
        }
        const unsigned mask = __reduce_or_sync(FULL, mine);
        const int t = c0 + lane, before = above - __popc(mask);
        const bool member = !((mask >> lane) & 1) && t < wn2;
        uint64_t key = 0;
        if (member) key = W[t - before - __popc(mask & ((1u << lane) - 1))];
        __syncwarp();
        if (member) W[t] = key;
        above = before;
        __syncwarp();
    }
    if (one) {
        if (at < wn2) W[at] = k;
    } else {
#pragma unroll 1
        for (int m0 = lane; m0 < nc; m0 += 32)
            if (place[m0] < wn2) W[place[m0]] = cand[m0];
    }
    return wn2;
}

// The codebooks of a walk or descent kernel into shared memory: the level-1 one and, for the full
// walk in FP16, the level-2 one behind it (FP32: read through the cache, returned as *C2).
template <int M1, int D1, typename CT, bool FQ, bool TAB>
__device__ __forceinline__ void load_codebooks(const WalkArgs &a, unsigned char *smem, const CT **C2)
{
    *C2 = nullptr;
    if constexpr (!TAB)
        copy_async(smem, sizeof(CT) == 4 ? (const void *)a.C1 : (const void *)a.C1h, walk_c1_bytes(a.d, M1, D1, sizeof(CT)));
    if constexpr (FQ && sizeof(CT) == 2) {
        unsigned char *c2 = smem + walk_c1_bytes(a.d, M1, D1, sizeof(CT));
        copy_async(c2, a.C2h, walk_c2_bytes(a.d, M1, D1));
        *C2 = reinterpret_cast<const CT *>(c2);
    } else if constexpr (FQ) {
        *C2 = reinterpret_cast<const CT *>(a.C2);
    }
    copy_wait();
    __syncthreads();
    pdl_wait();
    // only now may the next kernel start: what it reads without waiting for this one (the re-rank:
    // the list of ended walks, reset by the queue sort) has to be there
    pdl_launch();
}

// A team's share of scoring the n nodes in slot[0..n): blocks of slot_block nodes in turn, each
// staged and scored by one warp, totals into dist[0..n).  Block b takes the rows from b * SB mod STAGE_ROWS
// of the staging area; the team's size divides their number, so the rows of a warp are its own.
template <int M1, int D1, typename CT, bool FQ>
__device__ __forceinline__ void score_team(const CT *C1s, uint8_t *stage, const uint8_t *codes1, const uint8_t *codes2b, int M2P,
                                            const int32_t *slot, int n, int d, const LaneGeo<M1, D1> &g, int lane,
                                           int tw, int W, const CT *C2, float *dist)
{
    constexpr int SB = slot_block(M1), P1 = M1 / 16;
    const int s3 = slot_of_lane(lane, 3), node = M1 == 16 ? 2 * s3 + (lane >> 4) : s3;
#pragma unroll 1
    for (int b = tw; b * SB < n; b += W) {
        const int row0 = (b * SB) % STAGE_ROWS, r = lane / P1;
        uint8_t *st = stage + row0 * M1, *st2 = stage + STAGE_ROWS * M1 + row0 * M2P;
        if (r < SB && b * SB + r < n)
            copy16(st + lane * 16, codes1 + (int64_t)slot[b * SB + r] * M1 + (lane % P1) * 16);
        if constexpr (FQ)
            if (lane < SB && b * SB + lane < n)
                for (int u = 0; u < M2P; u += 16) copy16(st2 + lane * M2P + u, codes2b + (int64_t)slot[b * SB + lane] * M2P + u);
        copy_wait();
        __syncwarp();
        float v[8];
        if (FQ && D1 > 2 && !g.two) block_terms<M1, D1, CT, FQ, false, false>(C1s, st, st2, n - b * SB, d, g, lane, C2, M2P, v);
        else block_terms<M1, D1, CT, FQ, false, true>(C1s, st, st2, n - b * SB, d, g, lane, C2, M2P, v);
        const float t = reduce_block<M1>(v);
        if (lane_block<M1>(lane) == 0 && b * SB + node < n) dist[b * SB + node] = t;
        __syncwarp();
    }
}

// TEAM: a.team warps per query, for batches that leave most of an SM idle: the first walks, the
// others stage and score their share of each step's nodes (between two named barriers).  It
// shortens a step, which bounds a small batch (16 queries 247 -> 227 us, one 94 -> 84), and wastes
// issue slots in a large one.
// TAB (the table form, LC_LUT_TABLE): no codebook; each warp keeps its query's ADC table
// [256][M1] (FP16, built by table_kernel) in shared memory and scores nodes by table lookups.
// BATCH: beam > 1.  The plain walk is an instantiation of its own: it visits one row and merges at
// most 32 candidates a step, and the step's code has to stay small (the instruction cache bounds
// it: with the code for four rows beside its own the plain walk of 10k queries took 908 and not
// 853 us).
template <int M1, int D1, typename CT, bool FQ, bool TAB, bool BATCH, bool TEAM>
__global__ void __launch_bounds__(walk_threads(D1, FQ)) walk_kernel(const WalkArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, team = TEAM ? a.team : 1;
    const int warp = TEAM ? (threadIdx.x >> 5) / team : threadIdx.x >> 5, tw = TEAM ? (threadIdx.x >> 5) % team : 0;
    const int d = a.d;
    // the level-1 codebook, shared by every warp of the CTA
    CT *C1s = reinterpret_cast<CT *>(smem_raw);
    const CT *C2;
    load_codebooks<M1, D1, CT, FQ, TAB>(a, smem_raw, &C2);
    const WalkSmem L = walk_smem(M1, d, a.efcap, a.vt, a.beam, a.yq_in == nullptr, FQ ? a.M2P : 0);
    constexpr size_t TABB = TAB ? (size_t)256 * M1 * 2 : 0;            // the query's table
    unsigned char *base = smem_raw + (TAB ? 0 : walk_cb_bytes(d, M1, D1, sizeof(CT), FQ)) + (size_t)warp * (L.total + TABB);
    if constexpr (TAB) C1s = reinterpret_cast<CT *>(base + L.total);
    float *yq = reinterpret_cast<float *>(base + L.yq);
    uint8_t *stage = base + L.stage;
    uint64_t *W = reinterpret_cast<uint64_t *>(base + L.wkey);
    uint64_t *cand = reinterpret_cast<uint64_t *>(base + L.cand);
    int32_t *sel = reinterpret_cast<int32_t *>(base + L.sel);
    int32_t *slot = reinterpret_cast<int32_t *>(base + L.slot);
    volatile int32_t *ctl = reinterpret_cast<int32_t *>(base + L.ctl);
    float *dist = reinterpret_cast<float *>(cand) + 32 * a.beam;             // (read before candidates reach it)
    auto team_bar = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + warp), "r"(team * 32) : "memory"); };
    const int64_t gwarp = (int64_t)blockIdx.x * ((blockDim.x >> 5) / team) + warp;
    Visited V;
    V.tab = base + L.hash;
    V.tab_s = (uint32_t)__cvta_generic_to_shared(V.tab);
    V.stash = reinterpret_cast<int32_t *>(base + L.hash + a.vt.bytes);
    V.own_s = (uint32_t)__cvta_generic_to_shared(base + L.stage);
    const int H = 1 << a.hash_log;
    const int my_slot = TEAM ? lane : chunk_slot<M1>(lane);
    const unsigned lt_mask = (1u << lane) - 1;

    for (;;) {
        int64_t qi = 0;
        if (lane == 0 && tw == 0) qi = atomicAdd(a.counter, 1ull);
        qi = __shfl_sync(FULL, qi, 0);
        if constexpr (TEAM) {
            if (tw == 0 && lane == 0) ctl[0] = (int32_t)min(qi, (int64_t)0x7fffffff);
            team_bar();
            qi = ctl[0];
        }
        if (qi >= a.nq) break;
        const int64_t q = a.order ? (int64_t)a.order[qi] : qi;
        V.spill = a.spill + ((a.spill_tables >= a.nq ? qi : gwarp) << a.spill_log);
        // this query's ef' = max(ef, k)
        const int efp = a.efq ? max(min(max(__ldg(a.efq + q), 1), a.efp), a.k) : a.efp;
        if constexpr (TAB) {
            const uint4 *src = reinterpret_cast<const uint4 *>(a.tab + q * 256 * M1);
            uint4 *dst = reinterpret_cast<uint4 *>(C1s);
#pragma unroll 4
            for (int i = lane; i < 256 * M1 * 2 / 16; i += 32) dst[i] = __ldg(src + i);
            __syncwarp();
        }
        // rotation y' = R y (fixed order u = 0..d-1); uint8 queries convert exactly to FP32
        const float *yrot = a.yq_in ? a.yq_in + q * d : yq;
        if (a.yq_in) {
            // computed by rotate_kernel
        } else if (a.Q8) {
            const uint8_t *y = a.Q8 + q * d;
#pragma unroll 1
            for (int t = lane; t < d; t += 32) {
                float s = 0.f;
#pragma unroll 4
                for (int u = 0; u < d; u++) s = fmaf(__ldg(a.Rt + (int64_t)u * d + t), (float)__ldg(y + u), s);
                yq[t] = s;
            }
        } else {
            const float *y = a.Q + q * d;
#pragma unroll 1
            for (int t = lane; t < d; t += 32) {
                float s = 0.f;
#pragma unroll 4
                for (int u = 0; u < d; u++) s = fmaf(__ldg(a.Rt + (int64_t)u * d + t), __ldg(y + u), s);
                yq[t] = s;
            }
        }
        if (tw == 0) V.clear(a.vt, lane);
        __syncwarp();
        LaneGeo<M1, D1> g;
        g.init(a.s1, yrot, FQ ? a.sub2 : nullptr, d, lane);
        if constexpr (TEAM) {
            if (tw > 0) {
                for (;;) {
                    team_bar();
                    const int n = ctl[1];
                    if (n == 0) break;                   // the walk has ended
                    score_team<M1, D1, CT, FQ>(C1s, stage, a.codes1, a.codes2b, a.M2P, slot, n, d, g, lane, tw, team, C2, dist);
                    team_bar();
                }
                continue;
            }
        }
        // One loop runs the greedy descent of the upper levels (Section 2) and then the level-0
        // best-first search.  Each iteration gathers the nodes to score in slot[] and scores
        // them at a single call site, so the kernel holds one copy of the scoring code.
        int32_t n_up = 0, n_dist = 0, n_expand = 0;
        int32_t cur = a.ep;
        float dcur = 0.f;
        int lvl = a.max_level;             // upper level being descended
        int phase = 0;                     // 0: entry point, 1: upper levels, 2: level 0
        int wn = 1;
        bool failed = false;
        int scan_from = 0;                 // every member of W before it is expanded
        const int B = BATCH ? a.beam : 1;  // level-0 expansions per step
        if (a.mode == 2) {
            // level 0 from the entry node the descent launch recorded (as at its end below)
            cur = a.seed[q];
            dcur = a.seed_d[q];
            n_up = a.seed_up[q];
            phase = 2;
            if (lane == 0) W[0] = walk_key(dcur, cur);
            V.first(a.vt, cur, lane);
            n_dist = 1;
            __syncwarp();
        }
        for (;;) {
            int ns = 0;
            if (phase == 0) {
                if (lane == 0) slot[0] = cur;
                ns = 1;
            } else if (phase == 1) {
                // the current node's row at this level
                const int32_t e = a.upper_adj[((int64_t)a.upper_off[cur] + lvl - 1) * DEG + lane];
                const unsigned vm = __ballot_sync(FULL, e >= 0);
                ns = __popc(vm);
                if (e >= 0) slot[__popc(vm & lt_mask)] = e;
                n_up += ns;
            } else {
                if (a.tcap > 0 && n_dist >= a.tcap) break;     // search-time cap T (Section 3.1)
                // the B best unexpanded members of W, marked expanded, their ids in sel[]
                int nb = 0;
#pragma unroll 1
                for (int b0 = scan_from; b0 < wn && nb < B; b0 += 32) {
                    const int p = b0 + lane;
                    const uint64_t key = p < wn ? W[p] : 1;
                    const bool open = !(key & 1);
                    const unsigned m = __ballot_sync(FULL, open);
                    const int i = nb + __popc(m & lt_mask);
                    if (open && i < B) {
                        sel[i] = walk_id(key);
                        W[p] = key | 1;
                    }
                    if (nb == 0 && m) scan_from = b0;
                    nb += __popc(m);
                }
                nb = min(nb, B);
                if (nb == 0) break;
                n_expand += nb;
                __syncwarp();
                if (BATCH && nb > 4 && lane >= 4 && lane < nb)
                    prefetch_l1(a.adj0 + (int64_t)sel[lane] * DEG);
                // their adjacency rows through the visited test, four rows at a time while the
                // limits leave room for all of them, else row by row; fresh nodes are appended
                const int half = (1 << a.spill_log) / 2;
#pragma unroll 1
                for (int r0 = 0; r0 < nb;) {
                    int cnt = BATCH ? min(4, nb - r0) : 1;
                    if (V.spilled ? V.scount + 32 * cnt > half : V.hcount + 32 * cnt > shared_visited_cap(H)) {
                        cnt = 1;
                        if (!V.spilled && V.hcount + 32 > shared_visited_cap(H)) {
                            V.spilled = true;            // from here on counted to the global limit
                            if (!a.vt.tag) clear_spill(V.spill, a.spill_log, lane);
                        }
                        if (V.spilled && V.scount + 32 > half) {
                            failed = true;
                            break;
                        }
                    }
                    int nf;
                    if (!a.vt.tag) {
                        nf = visit_rows_ids(V.tab_s, V.own_s, a.vt.bb, V.spill, a.spill_log, V.spilled, a.adj0, sel + r0,
                                            cnt, slot, ns, lane);
                    } else if constexpr (!BATCH) {
                        nf = visit_ids<true>(V, a.vt, a.spill_log, __ldg(a.adj0 + (int64_t)sel[r0] * DEG + lane), slot, ns, lane);
                    } else {
                        int32_t ev[4];
#pragma unroll
                        for (int u = 0; u < 4; u++) ev[u] = u < cnt ? __ldg(a.adj0 + (int64_t)sel[r0 + u] * DEG + lane) : -1;
                        nf = visit_rows<true>(V, a.vt, a.spill_log, ev, cnt, slot, ns, lane);
                    }
                    ns += nf;
                    n_dist += nf;
                    if (V.spilled) V.scount += nf; else V.hcount += nf;
                    r0 += cnt;
                }
                if (failed) break;
                if (ns == 0) {
                    __syncwarp();
                    continue;
                }
            }
            // score the gathered nodes 32 at a time: the upper levels keep the best, level 0
            // collects those that can enter W and merges them into it
            uint32_t bd = ~0u, bi = ~0u;
            const uint64_t wmax = phase == 2 && wn == efp ? W[wn - 1] : ~0ull;
            int nc = 0;
            if (TEAM && ns > 0) {                          // (0 would tell the team that the walk has ended)
                if (lane == 0) ctl[1] = ns;
                team_bar();
                score_team<M1, D1, CT, FQ>(C1s, stage, a.codes1, a.codes2b, a.M2P, slot, ns, d, g, lane, 0, team, C2, dist);
                team_bar();
            }
#pragma unroll 1
            for (int ch = 0; ch < ns; ch += 32) {          // (once unless BATCH)
                const int nf = min(32, ns - ch);
                if (!TEAM) stage_codes<M1, FQ>(stage, a.codes1, a.codes2b, a.M2P, slot + ch, nf, lane);
                float de;
                if constexpr (TEAM) de = lane < nf ? dist[ch + lane] : 0.f;
                else de = score_staged<M1, D1, CT, FQ, TAB, BATCH && !FQ && (D1 > 0)>(C1s, stage, stage + STAGE_ROWS * M1, nf, d, g, lane, C2, a.M2P);
                const int32_t id = my_slot < nf ? slot[ch + my_slot] : -1;
                if (phase < 2) {                         // at most 32 nodes here
                    warp_best(id >= 0 ? __float_as_uint(de) : ~0u, (uint32_t)id, &bd, &bi);
                } else {
                    const uint64_t k = id >= 0 ? walk_key(de, id) : ~0ull;
                    const unsigned km = __ballot_sync(FULL, k < wmax);
                    if (k < wmax) cand[nc + __popc(km & lt_mask)] = k;
                    nc += __popc(km);
                }
            }
            __syncwarp();
            if (phase < 2) {
                bool enter0 = false;
                if (phase == 0) {
                    dcur = __uint_as_float(bd);
                    if (lvl >= 1) {
                        n_up = 1;                           // the entry point's evaluation
                        phase = 1;
                    } else {
                        enter0 = true;
                    }
                } else if (ns > 0 && (bd < __float_as_uint(dcur) || (bd == __float_as_uint(dcur) && (int32_t)bi < cur))) {
                    cur = (int32_t)bi;                      // greedy move at this level
                    dcur = __uint_as_float(bd);
                } else if (--lvl == 0) {
                    enter0 = true;
                }
                if (enter0) {
                    // level 0: best-first search with the result list W (sorted keys)
                    phase = 2;
                    if (lane == 0) W[0] = walk_key(dcur, cur);
                    V.first(a.vt, cur, lane);
                    n_dist = 1;
                    __syncwarp();
                }
            } else if (nc > 0) {
                int first_new;
                wn = merge_step<BATCH>(W, wn, efp, cand, nc, slot, lane, &first_new);
                scan_from = min(scan_from, first_new & ~31);
                __syncwarp();
            }
        }

        if constexpr (TEAM) {
            if (lane == 0) ctl[1] = 0;
            team_bar();
        }
        // outputs
        if (a.refine) {
            if (!a.yq_in)
#pragma unroll 1
                for (int t = lane; t < d; t += 32) a.yq_out[q * d + t] = yq[t];
#pragma unroll 1
            for (int i = lane; i < a.R; i += 32)
                a.short_out[q * a.R + i] = (!failed && i < wn) ? walk_id(W[i]) : -1;
        } else {
#pragma unroll 1
            for (int i = lane; i < a.R; i += 32) {
                bool ok = !failed && i < wn;
                a.ids_out[q * a.R + i] = ok ? walk_id(W[i]) : -1;
                a.dists_out[q * a.R + i] = ok ? key_dist(W[i]) : __int_as_float(0x7f800000);
            }
        }
        if (lane == 0) {
            if (a.stats_out) {
                a.stats_out[q * 3 + 0] = failed ? -1 : n_dist;
                a.stats_out[q * 3 + 1] = n_expand;
                a.stats_out[q * 3 + 2] = n_up;
            }
            if (failed) atomicOr(a.status, 1);
        }
        __syncwarp();
        if (a.done_list && lane == 0) {
            __threadfence();                             // the shortlist (every lane's part) before the entry
            asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(a.done_list + atomicAdd(a.done_tail, 1)), "r"((int32_t)q)
                         : "memory");
        }
    }
}


// ------------------------------------------------------------------------------------------
// Upper-level descent alone (the first launch of an ordered search): the greedy descent of
// Section 2 from the entry point down to level 1, exactly as walk_kernel runs it before level
// 0, writing each query's level-0 entry node, its walk distance and the upper-level
// evaluations.  It needs none of the level-0 state (result list, visited tables, merge
// buffers), so a warp holds only its staged code rows and node list: more warps fit per SM
// (up to 32), and more descents are in flight at once.
constexpr int MAX_DESCENT_WARPS = 32;

__host__ __device__ inline size_t descent_smem_per_warp(int M1, int m2p)
{
    return align_up((size_t)32 * (M1 + m2p), 16) + 32 * 4;
}

// threads per CTA the instantiation is compiled for: the full-decode walk keeps more per-lane
// state (the level-2 sub-space of every coordinate), so it gets registers for 16 warps
__host__ __device__ constexpr int descent_threads(bool fq) { return fq ? 16 * 32 : MAX_DESCENT_WARPS * 32; }

template <int M1, int D1, typename CT, bool FQ, bool TAB = false>
__global__ void __launch_bounds__(descent_threads(FQ)) descent_kernel(const WalkArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = a.d;
    CT *C1s = reinterpret_cast<CT *>(smem_raw);
    const CT *C2;
    load_codebooks<M1, D1, CT, FQ, TAB>(a, smem_raw, &C2);
    const int m2p = FQ ? a.M2P : 0;
    unsigned char *base = smem_raw + (TAB ? 0 : walk_cb_bytes(d, M1, D1, sizeof(CT), FQ)) +
                          (size_t)warp * descent_smem_per_warp(M1, m2p);
    uint8_t *stage = base;
    int32_t *slot = reinterpret_cast<int32_t *>(base + align_up((size_t)32 * (M1 + m2p), 16));
    const int my_slot = chunk_slot<M1>(lane);
    const unsigned lt_mask = (1u << lane) - 1;

    for (;;) {
        int64_t qi = 0;
        if (lane == 0) qi = atomicAdd(a.counter, 1ull);
        qi = __shfl_sync(FULL, qi, 0);
        if (qi >= a.nq) break;
        const int64_t q = qi;
        const float *yrot = a.yq_in + q * d;       // y' = R y from the rotation kernel
        // TAB: the query's ADC table [256][M1], read through L1 (a descent scores few nodes)
        const CT *T1 = TAB ? reinterpret_cast<const CT *>(a.tab + q * 256 * M1) : C1s;
        LaneGeo<M1, D1> g;
        g.init(a.s1, yrot, FQ ? a.sub2 : nullptr, d, lane);
        // the entry point's evaluation, then steepest moves level by level (as walk_kernel)
        int32_t cur = a.ep, n_up = 0;
        float dcur = 0.f;
        int lvl = a.max_level;
        bool first = true;
        for (;;) {
            int ns;
            if (first) {
                if (lane == 0) slot[0] = cur;
                ns = 1;
            } else {
                const int32_t e = a.upper_adj[((int64_t)a.upper_off[cur] + lvl - 1) * DEG + lane];
                const unsigned vm = __ballot_sync(FULL, e >= 0);
                ns = __popc(vm);
                if (e >= 0) slot[__popc(vm & lt_mask)] = e;
                n_up += ns;
            }
            uint32_t bd = ~0u, bi = ~0u;
            if (ns > 0) {
                stage_codes<M1, FQ>(stage, a.codes1, a.codes2b, a.M2P, slot, ns, lane);
                const float de = score_staged<M1, D1, CT, FQ, TAB, !FQ && (D1 > 0)>(T1, stage, stage + 32 * M1, ns, d, g, lane, C2, a.M2P);
                const int32_t id = my_slot < ns ? slot[my_slot] : -1;
                warp_best(id >= 0 ? __float_as_uint(de) : ~0u, (uint32_t)id, &bd, &bi);
            }
            __syncwarp();
            if (first) {
                first = false;
                dcur = __uint_as_float(bd);
                if (lvl < 1) break;
                n_up = 1;                                   // the entry point's evaluation
            } else if (ns > 0 && (bd < __float_as_uint(dcur) || (bd == __float_as_uint(dcur) && (int32_t)bi < cur))) {
                cur = (int32_t)bi;                          // greedy move at this level
                dcur = __uint_as_float(bd);
            } else if (--lvl == 0) {
                break;
            }
        }
        if (lane == 0) {
            a.seed[q] = cur;
            a.seed_d[q] = dcur;
            a.seed_up[q] = n_up;
        }
        __syncwarp();
    }
}

constexpr size_t MAX_SMEM_PER_BLOCK = 227 * 1024;

// Warps per query of a batch of nq: four while no SM has more than four queries (two for M1 = 16,
// whose staging area holds two blocks), else one: with six queries an SM two warps each took 183
// us where one took 179.
inline int walk_team(int64_t nq, int sms, int M1)
{
    return nq > 4 * (int64_t)sms ? 1 : M1 == 16 ? 2 : 4;
}

// Launch shape of the descent: as many warps as fit next to the codebook, at most 32.
template <int M1, int D1, typename CT, bool FQ, bool TAB = false>
static cudaError_t launch_descent(const WalkArgs &wa, int sms, int *wpc_out, int *grid_out, size_t *smem_out)
{
    const size_t c1 = TAB ? 0 : walk_cb_bytes(wa.d, M1, D1, sizeof(CT), FQ);
    const size_t per = descent_smem_per_warp(M1, FQ ? wa.M2P : 0);
    if (c1 + per > MAX_SMEM_PER_BLOCK) return cudaErrorInvalidConfiguration;
    int wpc = (int)std::min<size_t>(MAX_DESCENT_WARPS, (MAX_SMEM_PER_BLOCK - c1) / per);
    wpc = (int)std::min<int64_t>(wpc, std::max<int64_t>(1, (wa.nq + sms - 1) / sms));
    cudaError_t e = cudaFuncSetAttribute(descent_kernel<M1, D1, CT, FQ, TAB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)MAX_SMEM_PER_BLOCK);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, descent_kernel<M1, D1, CT, FQ, TAB>);
    if (e != cudaSuccess) return e;
    wpc = std::min(wpc, fa.maxThreadsPerBlock / 32);
    const size_t smem = c1 + per * wpc;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, descent_kernel<M1, D1, CT, FQ, TAB>, wpc * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int64_t need = (wa.nq + wpc - 1) / wpc;
    *grid_out = (int)std::min<int64_t>(need, (int64_t)per_sm * sms);
    *wpc_out = wpc;
    *smem_out = smem;
    return cudaSuccess;
}

// Compile-time shape of an instantiation (level-1 sub-quantisers, sub-space width, full walk),
// for dispatching a generic launcher over the instantiations.
template <int A, int B, bool C>
struct WalkShape {
    static constexpr int M1 = A, D1 = B;
    static constexpr bool FQ = C;
};

template <int M1, int D1, typename CT, bool FQ, bool TAB = false>
static cudaError_t run_descent(const WalkArgs &wa, size_t smem, int wpc, int grid, cudaStream_t st, bool pdl)
{
    return launch(descent_kernel<M1, D1, CT, FQ, TAB>, grid, wpc * 32, smem, st, pdl, wa);
}

// Warps per CTA: as many as fit next to the codebook (at most MAX_WALK_WARPS, and at most
// want if want > 0).
template <int M1, int D1, typename CT, bool FQ, bool TAB, bool BATCH, bool TEAM>
static cudaError_t launch_walk(const WalkArgs &wa, size_t smem_per_warp, int num_sms, int want, int *wpc_out,
                               int *grid_out, size_t *smem_out)
{
    size_t c1 = TAB ? 0 : walk_cb_bytes(wa.d, M1, D1, sizeof(CT), FQ);
    if (c1 + smem_per_warp > MAX_SMEM_PER_BLOCK) return cudaErrorInvalidConfiguration;
    int wpc = (int)std::min<size_t>(walk_threads(D1, FQ) / 32, (MAX_SMEM_PER_BLOCK - c1) / smem_per_warp);
    if (want > 0) wpc = std::min(wpc, want);
    if (TEAM) wpc = std::min(wpc, std::min(15, walk_threads(D1, FQ) / 32 / wa.team));      // (a named barrier each)
    // a batch that does not fill the GPU spreads over all SMs, evenly: one CTA on each (777 queries
    // run as 152 CTAs of 6 warps, and not as 130)
    const int64_t even = std::max<int64_t>(1, (wa.nq + num_sms - 1) / num_sms);
    const bool small = even < wpc;
    wpc = (int)std::min<int64_t>(wpc, even);
    size_t smem = c1 + smem_per_warp * wpc;
    // the attribute is an upper bound: set to the maximum, so plans made in any order (the
    // server plans at submission and launches later) all remain launchable
    cudaError_t e = cudaFuncSetAttribute(walk_kernel<M1, D1, CT, FQ, TAB, BATCH, TEAM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)MAX_SMEM_PER_BLOCK);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, walk_kernel<M1, D1, CT, FQ, TAB, BATCH, TEAM>,
                                                      wpc * (TEAM ? wa.team : 1) * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int64_t need = small ? std::min<int64_t>(wa.nq, num_sms) : (wa.nq + wpc - 1) / wpc;
    *grid_out = (int)std::min<int64_t>(need, (int64_t)per_sm * num_sms);
    *wpc_out = wpc;
    *smem_out = smem;
    return cudaSuccess;
}

template <int M1, int D1, typename CT, bool FQ, bool TAB, bool BATCH, bool TEAM>
static cudaError_t run_walk(const WalkArgs &wa, size_t smem, int wpc, int grid, cudaStream_t st, bool pdl)
{
    return launch(walk_kernel<M1, D1, CT, FQ, TAB, BATCH, TEAM>, grid, wpc * (TEAM ? wa.team : 1) * 32, smem, st, pdl, wa);
}

// Runs f(WalkShape<M1, D1, FQ>) for the instantiation of a sub-space width variant, M1 and the
// full-decode flag.  The full walk exists for the uniform splits and, in FP32, for any split.
template <typename CT, typename F>
static auto by_shape(int variant, int M1, bool fq, F &&f) -> decltype(f(WalkShape<16, 6, false>{}))
{
    if (fq) {
        switch (variant) {
        case 1: return f(WalkShape<16, 6, true>{});
        case 2: return f(WalkShape<32, 3, true>{});
        case 3: return f(WalkShape<64, 2, true>{});
        default:
            if constexpr (sizeof(CT) == 4)
                return M1 == 16 ? f(WalkShape<16, 0, true>{}) : M1 == 32 ? f(WalkShape<32, 0, true>{})
                                                               : f(WalkShape<64, 0, true>{});
            else
                return decltype(f(WalkShape<16, 6, false>{}))(cudaErrorInvalidValue);
        }
    }
    switch (variant) {
    case 1: return f(WalkShape<16, 6, false>{});
    case 2: return f(WalkShape<32, 3, false>{});
    case 3: return f(WalkShape<64, 2, false>{});
    default: return M1 == 16 ? f(WalkShape<16, 0, false>{}) : M1 == 32 ? f(WalkShape<32, 0, false>{})
                                                             : f(WalkShape<64, 0, false>{});
    }
}

// Launch shape, launch and kernel address of the walk, launch shape and launch of the descent, per
// codebook element type (lc_walk_f32.cu, lc_walk_f16.cu) and for the table form (LC_LUT_TABLE;
// M1 = 32 at d = 96).  Which walk instantiation also depends on wa.beam and wa.team (walk_fn:
// batch, team).
#define WALK_ENTRIES(NAME)                                                                                                  \
    cudaError_t walk_config_##NAME(int variant, int M1, bool fq, const WalkArgs &wa, size_t per_warp, int sms, int want,    \
                                   int *wpc, int *grid, size_t *smem);                                                      \
    cudaError_t walk_run_##NAME(int variant, int M1, bool fq, const WalkArgs &wa, size_t smem, int wpc, int grid,           \
                                cudaStream_t st, bool pdl);                                                                 \
    const void *walk_fn_##NAME(int variant, int M1, bool fq, bool batch, bool team);                                        \
    cudaError_t descent_config_##NAME(int variant, int M1, bool fq, const WalkArgs &wa, int sms, int *wpc, int *grid,       \
                                      size_t *smem);                                                                        \
    cudaError_t descent_run_##NAME(int variant, int M1, bool fq, const WalkArgs &wa, size_t smem, int wpc, int grid,        \
                                   cudaStream_t st, bool pdl);
WALK_ENTRIES(f32)
WALK_ENTRIES(f16)
WALK_ENTRIES(tab)
#undef WALK_ENTRIES

// The same for the form of a search.
inline cudaError_t walk_config(WalkForm f, int variant, int M1, bool fq, const WalkArgs &wa, size_t per_warp, int sms,
                               int want, int *wpc, int *grid, size_t *smem)
{
    return (f == WALK_F32 ? walk_config_f32 : f == WALK_F16 ? walk_config_f16 : walk_config_tab)(variant, M1, fq, wa, per_warp,
                                                                                              sms, want, wpc, grid, smem);
}
inline cudaError_t walk_run(WalkForm f, int variant, int M1, bool fq, const WalkArgs &wa, size_t smem, int wpc, int grid,
                            cudaStream_t st, bool pdl)
{
    return (f == WALK_F32 ? walk_run_f32 : f == WALK_F16 ? walk_run_f16 : walk_run_tab)(variant, M1, fq, wa, smem, wpc, grid, st,
                                                                                        pdl);
}
inline const void *walk_fn(WalkForm f, int variant, int M1, bool fq, bool batch, bool team)
{
    return (f == WALK_F32 ? walk_fn_f32 : f == WALK_F16 ? walk_fn_f16 : walk_fn_tab)(variant, M1, fq, batch, team);
}
inline cudaError_t descent_config(WalkForm f, int variant, int M1, bool fq, const WalkArgs &wa, int sms, int *wpc, int *grid,
                                  size_t *smem)
{
    return (f == WALK_F32 ? descent_config_f32 : f == WALK_F16 ? descent_config_f16 : descent_config_tab)(variant, M1, fq, wa,
                                                                                                       sms, wpc, grid, smem);
}
inline cudaError_t descent_run(WalkForm f, int variant, int M1, bool fq, const WalkArgs &wa, size_t smem, int wpc, int grid,
                               cudaStream_t st, bool pdl)
{
    return (f == WALK_F32 ? descent_run_f32 : f == WALK_F16 ? descent_run_f16 : descent_run_tab)(variant, M1, fq, wa, smem, wpc,
                                                                                              grid, st, pdl);
}

}  // namespace lc

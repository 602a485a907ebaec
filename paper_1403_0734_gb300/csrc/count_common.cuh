// count_common.cuh -- device helpers shared by the counting kernels (the
// ordered DFS in count.cu and the pivoting counter in sct.cu): launch
// context, the colour hash of cFFF_k, 128-bit total accumulation, and the
// G+(u) bitmap builders.
#pragma once

#include <climits>
#include <type_traits>

#include "kc_internal.cuh"

namespace kc {
namespace cc {

// One oriented graph as the kernels see it (device pointers).
struct GraphDesc {
    const int64_t* offp;
    const int32_t* adjp;
    const int32_t* queue;
    const int32_t* perm;
    const uint32_t* core;
    int32_t core_lo, core_tw;
};

inline GraphDesc desc_of(const kc_graph* g)
{
    return {g->offp, g->adjp, g->queue, g->perm, g->core, g->core_lo, g->core_tw};
}

// Launch context of one owner class.  Single-graph mode (ng == 0): item i is
// the owner at queue position q0 + qoff + i * qstride (qoff/qstride select a
// part of the owners).  Batch mode (ng > 0): item i belongs to graph g with
// gpre[g] <= i < gpre[g+1] and is the owner at position gq0[g] + i - gpre[g]
// of that graph's queue; totals are per graph.
struct Ctx {
    const int64_t* __restrict__ offp;
    const int32_t* __restrict__ adjp;
    const int32_t* __restrict__ queue;
    const int32_t* __restrict__ perm;
    const uint32_t* __restrict__ core;  // adjacency bitmap of the ranks from core_lo on
    int32_t core_lo, core_tw;
    int64_t q0, q1;
    int64_t nitems;
    int64_t qoff, qstride;
    const GraphDesc* gd;
    const int64_t* gq0;
    const int64_t* gpre;
    int ng;
    int k;
    uint32_t colours;
    uint64_t seed;
    int pair;        // plain pair sampling instead of colours (Sec. 6)
    uint64_t pthr;   // pair kept iff its hash < pthr
    unsigned long long* total;
    unsigned long long* pv;
    unsigned long long* po;
    unsigned long long* cursor;
    unsigned long long* work;  // nullable: bitmap word-operations executed
    float density;             // for the host's dispatch: edges / pairs of vertices (density_of)
};

inline float density_of(const kc_graph* g)
{
    return g->n > 1 ? (float)(2.0 * (double)g->m / ((double)g->n * (g->n - 1.0))) : 0.0f;
}

inline void set_graph(Ctx& c, const kc_graph* g)
{
    c.offp = g->offp;
    c.adjp = g->adjp;
    c.queue = g->queue;
    c.perm = g->perm;
    c.core = g->core;
    c.core_lo = g->core_lo;
    c.core_tw = g->core_tw;
    c.density = density_of(g);
}

// The context of one owner: a launch context with that owner's graph and total.
// Only resolve fills it.  A variable that already holds a copy of the launch's
// context, or takes it on another path, keeps the launch's offp after a resolve
// compiled by nvcc 13.0 (32 of 32 lanes of a kernel that only compared the
// pointers, with __restrict__ on Ctx's members and without); it is null in a batch.
struct OwnerCtx : Ctx {
    OwnerCtx() = default;
    OwnerCtx(const Ctx&) = delete;
    OwnerCtx(const OwnerCtx&) = delete;
    OwnerCtx& operator=(const Ctx&) = delete;
    OwnerCtx& operator=(const OwnerCtx&) = delete;
};
static_assert(!std::is_constructible<OwnerCtx, const Ctx&>::value && !std::is_assignable<OwnerCtx&, const Ctx&>::value &&
                  !std::is_copy_constructible<OwnerCtx>::value && !std::is_copy_assignable<OwnerCtx>::value,
              "an owner's context comes from resolve alone");

// The owner (rank r) of class item `item`, with a context whose graph
// pointers and total are that owner's graph's.  False past the last item.
__device__ __forceinline__ bool resolve(const Ctx& b, int64_t item, OwnerCtx& c, int32_t& r)
{
    if (item >= b.nitems) return false;
    static_cast<Ctx&>(c) = b;
    if (b.ng == 0) {
        r = b.queue[b.q0 + b.qoff + item * b.qstride];
        return true;
    }
    int lo = 0, hi = b.ng;  // largest g with gpre[g] <= item
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (b.gpre[mid] <= item) lo = mid; else hi = mid;
    }
    const GraphDesc gd = b.gd[lo];
    c.offp = gd.offp;
    c.adjp = gd.adjp;
    c.queue = gd.queue;
    c.perm = gd.perm;
    c.core = gd.core;
    c.core_lo = gd.core_lo;
    c.core_tw = gd.core_tw;
    c.total = b.total + 2 * lo;
    r = gd.queue[b.gq0[lo] + (item - b.gpre[lo])];
    return true;
}

// colour(u, x): splitmix64 output function over seed ^ (G * (u<<32 | x)),
// reduced to [0, c) by a 64x64 multiply-high (Sec. 6; spec in kc.h).
__device__ __forceinline__ uint32_t colour_of(uint64_t seed, int32_t u, int32_t x, uint32_t c)
{
    uint64_t key = ((uint64_t)(uint32_t)u << 32) | (uint64_t)(uint32_t)x;
    uint64_t z = seed ^ (0x9E3779B97F4A7C15ull * key);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (uint32_t)__umul64hi(z, (uint64_t)c);
}

// Pair sampling (Sec. 6, plain pair sampling): the pair {x, y} of Gamma+(u)
// is kept iff h < thr, h = F(F(seed ^ G (u<<32 | a)) ^ G b) with a < b the
// two original ids and F the splitmix64 output function (spec in kc.h).
__device__ __forceinline__ bool pair_kept(uint64_t seed, int32_t u, uint32_t x, uint32_t y, uint64_t thr)
{
    const uint32_t a = x < y ? x : y, b = x < y ? y : x;
    uint64_t z = seed ^ (0x9E3779B97F4A7C15ull * (((uint64_t)(uint32_t)u << 32) | (uint64_t)a));
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    z ^= 0x9E3779B97F4A7C15ull * (uint64_t)b;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return z < thr;
}

// The per-node label a sampling filter keeps for x_j of Gamma+(u) (ur, xid:
// original ids): its colour under cFFF_k, its id under pair sampling.
__device__ __forceinline__ uint32_t sample_label(const Ctx& c, int32_t ur, int32_t xid)
{
    return c.pair ? (uint32_t)xid : colour_of(c.seed, ur, xid, c.colours);
}

// Whether the pair with labels li, lj survives the sampling filter.
__device__ __forceinline__ bool sample_keep(const Ctx& c, int32_t ur, uint32_t li, uint32_t lj)
{
    return c.pair ? pair_kept(c.seed, ur, li, lj, c.pthr) : li == lj;
}

// cFFF_k: a sampled (k-1)-clique of G+(u) lies inside one colour class
// (Map 2 emits monochromatic pairs only), so a vertex whose class in Gamma+(u)
// has fewer than k-1 members lies in none, and its Gamma+ list need not be
// read at all (Round 2 shrinks with the sampling).  Such a vertex's label
// gets kSkipLabel; the flag is the same for its whole class, so labels still
// compare equal exactly within a class, and the builders skip its row.
// Colours are below c <= 2^31 (the flag bit is no colour); plain pair
// sampling (labels are ids) is not filtered.
constexpr uint32_t kSkipLabel = 0x80000000u;

__device__ __forceinline__ bool class_filter_on(const Ctx& c) { return !c.pair && c.colours <= kSkipLabel; }

// Lane j holds the label of x_j (j < d): flags small classes (match_any).
__device__ __forceinline__ uint32_t class_flag_w1(const Ctx& c, uint32_t col, int d, int need, int lane)
{
    if (!class_filter_on(c)) return col;
    const uint32_t key = lane < d ? col : kSkipLabel + (uint32_t)lane;
    const uint32_t peers = __match_any_sync(kFull, key);
    return (lane < d && __popc(peers) < need) ? (col | kSkipLabel) : col;
}

// Labels sCol[0..d) in shared memory, threads t0, t0+nt, ... of the caller
// (d <= 32 nt): flags small classes.  CTA: every thread of the block calls
// it (two __syncthreads), else the lanes of one warp (two __syncwarp).
template <bool CTA>
__device__ __forceinline__ void class_flags_smem(const Ctx& c, uint32_t* sCol, int d, int need, int t0, int nt)
{
    if (!class_filter_on(c)) return;
    uint32_t small = 0;  // bit q: element t0 + q nt is in a class smaller than need
    for (int q = 0; q < 32; ++q) {
        const int j = t0 + q * nt;
        if (j >= d) break;
        const uint32_t cj = sCol[j];
        int cnt = 0;
        for (int i = 0; i < d && cnt < need; ++i) cnt += sCol[i] == cj;
        if (cnt < need) small |= 1u << q;
    }
    if (CTA) __syncthreads(); else __syncwarp();
    for (int q = 0; q < 32; ++q) {
        const int j = t0 + q * nt;
        if (j >= d) break;
        if ((small >> q) & 1u) sCol[j] |= kSkipLabel;
    }
    if (CTA) __syncthreads(); else __syncwarp();
}

// 128-bit total as (lo, hi) words.
__device__ __forceinline__ void add_total(unsigned long long* t, unsigned long long v)
{
    if (v == 0) return;
    unsigned long long old = atomicAdd(&t[0], v);
    if (old + v < old) atomicAdd(&t[1], 1ull);
}

// A warp's running total: sent when the graph changes (batches) and at the
// end, not once per owner -- all owners of a graph share one address, which
// takes one addition every few nanoseconds.
struct TotalSum {
    unsigned long long* at;
    unsigned long long lo = 0, hi = 0;
    __device__ __forceinline__ explicit TotalSum(unsigned long long* t) : at(t) {}
    __device__ __forceinline__ void add(unsigned long long* t, unsigned long long v, int lane)
    {
        if (t != at) {
            flush(lane);
            at = t;
            lo = hi = 0;
        }
        lo += v;
        if (lo < v) ++hi;
    }
    __device__ __forceinline__ void flush(int lane)
    {
        if (lane != 0) return;
        add_total(at, lo);
        if (hi) atomicAdd(&at[1], hi);
    }
};

// One owner's graph, for the one-warp kernels (sampling labels need the
// caller's ids, Ctx::perm: single graphs only).
struct Gr {
    const int64_t* offp;
    const int32_t* adjp;
    const uint32_t* core;
    int32_t core_lo, core_tw;
    unsigned long long* total;
};

// Owners for one-warp kernels, `take` (at most 32) per cursor step: their
// graphs, ranks, offsets and sizes are fetched together, a lane each.
struct Owners {
    int take_n;
    __device__ __forceinline__ explicit Owners(int n) : take_n(n) {}
    int have = 0, at = 0;
    int32_t rank = 0;
    int graph = 0, deg = 0;
    int64_t off = 0;
    // Whether there is another owner; the same in every lane.
    __device__ __forceinline__ bool next(const Ctx& cb, int lane)
    {
        if (at < have) return true;
        unsigned long long pos = 0;
        if (lane == 0) pos = atomicAdd(cb.cursor, (unsigned long long)take_n);
        pos = __shfl_sync(kFull, pos, 0);
        if ((int64_t)pos >= cb.nitems) return false;
        at = 0;
        have = (int)min((int64_t)take_n, cb.nitems - (int64_t)pos);
        if (lane < have) {
            const int64_t item = (int64_t)pos + lane;
            const int64_t* offp;
            if (cb.ng == 0) {
                rank = cb.queue[cb.q0 + cb.qoff + item * cb.qstride];
                offp = cb.offp;
            } else {
                int lo = 0, hi = cb.ng;  // largest g with gpre[g] <= item
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (cb.gpre[mid] <= item) lo = mid; else hi = mid;
                }
                graph = lo;
                rank = cb.gd[lo].queue[cb.gq0[lo] + (item - cb.gpre[lo])];
                offp = cb.gd[lo].offp;
            }
            off = offp[rank];
            deg = (int)(offp[rank + 1] - off);
        }
        return true;
    }
    __device__ __forceinline__ void take(const Ctx& cb, Gr& g, int32_t& r, int64_t& b, int& d)
    {
        r = __shfl_sync(kFull, rank, at);
        b = __shfl_sync(kFull, off, at);
        d = __shfl_sync(kFull, deg, at);
        const int gi = __shfl_sync(kFull, graph, at);
        const GraphDesc* p = cb.gd + gi;
        g.offp = cb.ng ? p->offp : cb.offp;
        g.adjp = cb.ng ? p->adjp : cb.adjp;
        g.core = cb.ng ? p->core : cb.core;
        g.core_lo = cb.ng ? p->core_lo : cb.core_lo;
        g.core_tw = cb.ng ? p->core_tw : cb.core_tw;
        g.total = cb.total + 2 * gi;
        ++at;
    }
};

__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ uint32_t mask_above(int b) { return b >= 31 ? 0u : (kFull << (b + 1)); }
__device__ __forceinline__ uint32_t mask_below(int b) { return (1u << b) - 1u; }


// Rows of G+(u) for an owner with d <= 32 W (W = 1, 2), by one warp (Map 2
// pairs kept by Reduce 2): lane j holds x_j and x_{j+32} (ranks, INT_MAX past
// d) and gets the upper rows of both (up[h][w]: word w of element lane + 32 h;
// bit j set iff x_j is in Gamma+(x_i), j > i).
//
// The lists Gamma+(x_i) are read eight at a time, four lanes and one aligned
// 128-bit load per lane to a list, and every entry is looked up in a hash
// table of Gamma+(u): a byte with the index, checked against x itself, so the
// table needs neither clearing nor an empty mark.  Elements that collide under
// every multiplier tried (none, as a rule) are searched in the lists one by
// one.  A lookup is six instructions for each entry and a 16-entry step serves
// eight short lists; one list at a time, searched by shuffles, took some forty
// instructions for 32 entries of a single list.
template <int W>
struct SmallBuf {
    int32_t x[32 * W];
    uint8_t slot[1024 * W];
};

constexpr int kHashTries = 8;

template <int W, bool COL>
__device__ __forceinline__ void build_rows_small(const Ctx& c, const Gr& g, const int32_t (&x)[W], int d, const uint32_t (&col)[W],
                                                 int32_t ur, SmallBuf<W>& sb, int lane, uint32_t (&up)[W][W])
{
    constexpr int kShift = W == 1 ? 22 : 21;
    int32_t maxL = 0;
    int64_t s0[W];
    int len[W];
    uint32_t inside[W];  // elements of the core
#pragma unroll
    for (int h = 0; h < W; ++h) {
        const int j = lane + 32 * h;
        sb.x[j] = x[h];
        inside[h] = __ballot_sync(kFull, j < d && x[h] >= g.core_lo);
        const bool need = j < d - 1 && x[h] < g.core_lo && !(COL && class_filter_on(c) && (col[h] & kSkipLabel));  // (small colour class)
        s0[h] = need ? g.offp[x[h]] : 0;
        len[h] = need ? (int)(g.offp[x[h] + 1] - s0[h]) : 0;
        if (d > 32 * h) maxL = __shfl_sync(kFull, x[h], (d - 1 - 32 * h) & 31);
#pragma unroll
        for (int w = 0; w < W; ++w) up[h][w] = 0u;
    }
    int nlist = d;  // elements before the core
#pragma unroll
    for (int h = 0; h < W; ++h) nlist -= __popc(inside[h]);
    // the table; lost: elements without a slot of their own
    uint32_t lost[W] = {}, mul = 0x9E3779B1u;
#pragma unroll 1
    for (int t = 0; nlist > 0; ++t) {
#pragma unroll
        for (int h = 0; h < W; ++h)
            if (lane + 32 * h < d) sb.slot[((uint32_t)x[h] * mul) >> kShift] = (uint8_t)(lane + 32 * h);
        __syncwarp();
        uint32_t any = 0;
#pragma unroll
        for (int h = 0; h < W; ++h) {
            const bool ok = lane + 32 * h >= d || sb.slot[((uint32_t)x[h] * mul) >> kShift] == lane + 32 * h;
            lost[h] = __ballot_sync(kFull, !ok);
            any |= lost[h];
        }
        if (any == 0u || t == kHashTries - 1) break;
        mul = mul * 0x2C1B3C6Du + 2u;  // odd again
    }
    const int sub = lane & 3;
#pragma unroll 1
    for (int g0 = 0; g0 < min(nlist, d - 1); g0 += 8) {
        const int src = (g0 & 31) + (lane >> 2);
        int64_t b = __shfl_sync(kFull, s0[0], src);
        int n = __shfl_sync(kFull, len[0], src);
        if (W == 2 && g0 >= 32) {
            b = __shfl_sync(kFull, s0[W - 1], src);
            n = __shfl_sync(kFull, len[W - 1], src);
        }
        uint32_t m[W];
#pragma unroll
        for (int w = 0; w < W; ++w) m[w] = 0u;
        // rel: this lane's first entry of the step, relative to the list's start
        const int32_t* list = g.adjp + b;
        for (int rel = 4 * sub - (int)(b & 3); rel < n; rel += 16) {
            const int4 y = *(const int4*)(list + rel);
            const int32_t ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t idx = sb.slot[((uint32_t)ys[q] * mul) >> kShift] & (32u * W - 1u);
                if (sb.x[idx] == ys[q] && (unsigned)(rel + q) < (unsigned)n) {
                    if (W == 1 || idx < 32u) m[0] |= 1u << (idx & 31u);
                    else m[W - 1] |= 1u << (idx & 31u);
                }
            }
            if (y.w >= maxL) break;  // ascending: nothing further on for this lane
        }
        const int row = 4 * (lane & 7);
        const bool mine = (lane >> 3) == ((g0 & 31) >> 3);
#pragma unroll
        for (int w = 0; w < W; ++w) {
            m[w] |= __shfl_xor_sync(kFull, m[w], 1);
            m[w] |= __shfl_xor_sync(kFull, m[w], 2);
            const uint32_t v = __shfl_sync(kFull, m[w], row);
            if (mine) {
                if (W == 1 || g0 < 32) up[0][w] = v;
                else up[W - 1][w] = v;
            }
        }
    }
    if (lost[0] | lost[W - 1])
#pragma unroll 1
    for (int e = 0; e < d; ++e) {
        if (!((lost[W == 1 || e < 32 ? 0 : W - 1] >> (e & 31)) & 1u)) continue;
        const int32_t xe = sb.x[e];
#pragma unroll
        for (int h = 0; h < W; ++h) {
            if (lane + 32 * h >= e) continue;
            int lo = 0, hi = len[h];
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (g.adjp[s0[h] + mid] < xe) lo = mid + 1; else hi = mid;
            }
            if (lo < len[h] && g.adjp[s0[h] + lo] == xe) {
                if (W == 1 || e < 32) up[h][0] |= 1u << (e & 31);
                else up[h][W - 1] |= 1u << (e & 31);
            }
        }
    }
    // rows of the core's elements, four at a time: every lane reads its own
    // elements' words of the row (lanes without one read word 0 and mask it), and
    // four lanes keep the ballots; what does not belong to an upper row of the
    // core is masked once at the end
    if (nlist < d - 1) {
        uint32_t word[W], bit[W], val[W][W];
        int off[W];
#pragma unroll
        for (int h = 0; h < W; ++h) {
            const bool in = (inside[h] >> lane) & 1u;
            off[h] = in ? x[h] - g.core_lo : 0;
            word[h] = (uint32_t)off[h] >> 5;
            bit[h] = in ? 1u << (off[h] & 31) : 0u;
#pragma unroll
            for (int w = 0; w < W; ++w) val[h][w] = 0u;
        }
#pragma unroll 1
        for (int i0 = nlist & ~3; i0 < d - 1; i0 += 4) {
            uint32_t v[4][W];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                int xi = __shfl_sync(kFull, off[0], (i0 + t) & 31);
                if (W == 2 && i0 >= 32) xi = __shfl_sync(kFull, off[W - 1], (i0 + t) & 31);
                const uint32_t* row = g.core + (int64_t)xi * g.core_tw;
#pragma unroll
                for (int h = 0; h < W; ++h) v[t][h] = row[word[h]];
            }
            const bool mine = (unsigned)(lane ^ (i0 & 31)) < 4u;
#pragma unroll
            for (int h = 0; h < W; ++h) {
                const uint32_t b0 = __ballot_sync(kFull, v[0][h] & bit[h]), b1 = __ballot_sync(kFull, v[1][h] & bit[h]);
                const uint32_t b2 = __ballot_sync(kFull, v[2][h] & bit[h]), b3 = __ballot_sync(kFull, v[3][h] & bit[h]);
                const uint32_t w = lane & 2 ? (lane & 1 ? b3 : b2) : (lane & 1 ? b1 : b0);
                if (mine) {
                    if (W == 1 || i0 < 32) val[0][h] = w;
                    else val[W - 1][h] = w;
                }
            }
        }
#pragma unroll
        for (int h = 0; h < W; ++h) {
            const int j = lane + 32 * h;
            if (j < nlist || j >= d) continue;
#pragma unroll
            for (int w = h; w < W; ++w) up[h][w] = w == h ? val[h][w] & mask_above(lane) : val[h][w];
        }
    }
    if (COL) {  // (rows with an edge: random graph n = 5e5, m = 3e7, pairs at k = 4, 7.7 -> 6.7 ms)
#pragma unroll
        for (int h = 0; h < W; ++h) {
            uint32_t rows = __ballot_sync(kFull, (up[h][0] | up[h][W - 1]) != 0u);
#pragma unroll 1
            for (; rows; rows &= rows - 1u) {
                const int i = __ffs(rows) - 1;
                const uint32_t ci = __shfl_sync(kFull, col[h], i);
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const uint32_t keep = __ballot_sync(kFull, sample_keep(c, ur, ci, col[w]));
                    if (lane == i) up[h][w] &= keep;
                }
            }
        }
    }
    __syncwarp();  // sb is free again
}

// Lower half of the symmetric G+(u) bitmap from the upper rows (bit i of
// row j for every i < j with bit j in row i).
__device__ __forceinline__ uint32_t lower_rows_w1(uint32_t up, int d, int lane)
{
    uint32_t low = 0;
    for (int j = 1; j < d; ++j) {
        const uint32_t colj = __ballot_sync(kFull, (up >> j) & 1u);
        if (lane == j) low = colj;
    }
    return low;
}

// Direct-address table over the rank span [lo, lo + 32 words) of Gamma+(u):
// bit (y - lo) set iff y is in Gamma+(u), pre[w] = number of elements below
// lo + 32 w, so y's local index is pre[w] + popc(bits[w] below y's bit).
// words == 0: no table (the span is too wide); searches fall back to binary
// search in sL.
struct SpanTable {
    uint32_t* bits;
    uint16_t* pre;
    int32_t lo;
    int words;
};

// Fill T for sL[0..d) (ascending) by the threads of the CTA when the span
// fits maxw words; ends with __syncthreads().  Every thread must call it.
__device__ __forceinline__ void span_table_build(SpanTable& T, const int32_t* sL, int d, int maxw)
{
    const int64_t span = (int64_t)sL[d - 1] - sL[0] + 1;
    T.lo = sL[0];
    T.words = span <= 32LL * maxw ? (int)((span + 31) >> 5) : 0;
    if (T.words == 0) return;
    for (int w = threadIdx.x; w < T.words; w += blockDim.x) T.bits[w] = 0u;
    __syncthreads();
    for (int j = threadIdx.x; j < d; j += blockDim.x) {
        const int off = sL[j] - T.lo;
        atomicOr(&T.bits[off >> 5], 1u << (off & 31));
    }
    for (int w = threadIdx.x; w < T.words; w += blockDim.x) {
        const int32_t key = T.lo + 32 * w;
        int a = 0, z = d;
        while (a < z) {
            const int mid = (a + z) >> 1;
            if (sL[mid] < key) a = mid + 1; else z = mid;
        }
        T.pre[w] = (uint16_t)a;
    }
    __syncthreads();
}

// First j with s[j] >= v in the ascending s[0..d).
__device__ __forceinline__ int first_at_least(const int32_t* s, int d, int32_t v)
{
    int lo = 0, hi = d;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (s[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Rows of G+(u) into a bitmap A (row stride RS words, zeroed beforehand) by
// warps w0, w0+nw, ... of the caller; sL holds Gamma+(u) (ranks, ascending),
// sCol their sampling labels (COL; ur: u's original id).  With SYM the
// bitmap is made symmetric.
template <bool SYM, bool COL>
__device__ __forceinline__ void build_rows(const Ctx& c, const int32_t* sL, const uint32_t* sCol, int d,
                                           uint32_t* A, int RS, int w0, int nw, int lane, int32_t ur = 0,
                                           const SpanTable* T = nullptr)
{
    const int32_t maxL = sL[d - 1];
    const bool direct = T && T->words > 0;
    // the core's elements (a suffix): bits gathered from the core bitmap, a
    // ballot for each word.  Words that hold no element before the core are
    // written by their ballot alone.  (Chung-Lu n = 1e6, k = 4 with memberships:
    // 4-word class 2.14 -> 1.14 ms, 8 words 1.82 -> 1.15 ms, 16 words 1.76 -> 1.36
    // ms: a gather is 8 instructions for 32 pairs, a list chunk some 30, and
    // lists of hubs are longer than the owners' rows.)
    const int nlist = maxL >= c.core_lo ? first_at_least(sL, d, c.core_lo) : d;
    for (int jb = nlist >> 5; jb * 32 < d; ++jb) {
        const int j = jb * 32 + lane;
        const bool in = j >= nlist && j < d;
        const int off = in ? sL[j] - c.core_lo : 0;
        const uint32_t cj = COL && in ? sCol[j] : 0u;
        const int iend = SYM ? d : min(d, jb * 32 + 32);
        for (int i0 = nlist + w0; i0 < iend; i0 += 4 * nw) {
            uint32_t v[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int i = i0 + t * nw;
                v[t] = 0u;
                if (i < iend && in && (SYM || j > i))
                    v[t] = c.core[(int64_t)(sL[i] - c.core_lo) * c.core_tw + (off >> 5)];
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int i = i0 + t * nw;
                if (i >= iend) break;
                bool hit = (v[t] >> (off & 31)) & 1u;
                if (COL) {
                    const uint32_t ci = sCol[i];
                    hit = hit && !(class_filter_on(c) && (ci & kSkipLabel)) && sample_keep(c, ur, ci, cj);
                }
                const uint32_t w = __ballot_sync(kFull, hit);
                if (lane == 0 && w) {
                    if (SYM && jb == (nlist >> 5)) atomicOr(&A[(int64_t)i * RS + jb], w);
                    else A[(int64_t)i * RS + jb] = w;
                }
            }
        }
    }
    for (int i = w0; i < min(nlist, d - 1); i += nw) {
        const uint32_t ci = COL ? sCol[i] : 0u;
        if (COL && class_filter_on(c) && (ci & kSkipLabel)) continue;  // too small a colour class: no sampled clique
        const int32_t xi = sL[i];
        const int64_t s0 = c.offp[xi], s1 = c.offp[xi + 1];
        for (int64_t p0 = s0; p0 < s1; p0 += 32) {
            const int64_t pp = p0 + lane;
            const int32_t y = pp < s1 ? c.adjp[pp] : INT_MAX;
            if (y <= maxL) {
                int lo = i + 1;
                bool hit;
                if (direct) {  // y > x_i >= lo: inside the span
                    const int off = y - T->lo;
                    const uint32_t wv = T->bits[off >> 5];
                    hit = (wv >> (off & 31)) & 1u;
                    lo = (int)T->pre[off >> 5] + __popc(wv & mask_below(off & 31));
                } else {
                    int hi = d;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (sL[mid] < y) lo = mid + 1; else hi = mid;
                    }
                    hit = lo < d && sL[lo] == y;
                }
                if (hit && (!COL || sample_keep(c, ur, ci, sCol[lo]))) {
                    atomicOr(&A[(int64_t)i * RS + (lo >> 5)], 1u << (lo & 31));
                    if (SYM) atomicOr(&A[(int64_t)lo * RS + (i >> 5)], 1u << (i & 31));
                }
            }
            if (__shfl_sync(kFull, y, 31) >= maxL) break;
        }
    }
}

// Row widths (words) the closing kernels (close.cu) are built for: 1..6, 8,
// 12, 16; the number of the narrowest one that holds a set of n elements.
constexpr int kCloseBins = 9;
__host__ __device__ __forceinline__ int close_bin(int n)
{
    const int w = (n + 31) >> 5;
    return w <= 6 ? w - 1 : (w <= 8 ? 6 : (w <= 12 ? 7 : 8));
}

// Opt a kernel in to `smem` bytes of dynamic shared memory.  The default
// limit (48 KB) covers static and dynamic shared memory together, so the
// attribute is set whenever the dynamic part alone comes near it.
template <typename K>
inline cudaError_t allow_smem(K kernel, size_t smem)
{
    if (smem <= 32 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// Owners a warp takes per cursor step and the CTAs (of `warps` warps) to
// launch, at most `room`: up to `most` where every warp of a full GPU still
// gets several steps, one where there are too few owners for that (taken four
// at a time, a class of 700 owners ran on a quarter of the warps: 135 -> 229
// us for a whole count of a 20,000-vertex graph).
struct OwnerSteps {
    int take, grid;
};
inline OwnerSteps owner_steps(int64_t nitems, int warps, int64_t room, int most)
{
    const int64_t per = nitems / (4 * room * warps);
    const int take = (int)std::min<int64_t>(std::max<int64_t>(per, 1), most);
    return {take, (int)std::min<int64_t>((nitems + (int64_t)warps * take - 1) / ((int64_t)warps * take), room)};
}

template <typename K>
inline int blocks_per_sm(K kernel, int threads, size_t smem)
{
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, threads, smem) != cudaSuccess || nb < 1)
        nb = 1;
    return nb;
}

}  // namespace cc
}  // namespace kc

// list.cu -- k-clique listing: every k-clique of G once, as k caller ids in
// the order < (owner first), streamed through a caller buffer in chunks.
//
// The exact algorithm lists as well as counts (Sec. 1; Reduce 3 of Sec. 3
// enumerates the (k-1)-cliques of each G+(u)); the output can be far larger
// than device memory (Table 1's counts), so it is produced in chunks:
//   1. per-owner counts q_{u,k-1} by the counting kernels;
//   2. on the host, the owner queue is cut into consecutive runs whose counts
//      fit the caller's buffer, and each owner gets its offset in the run;
//   3. per run, one CTA per owner rebuilds G+(u) (upper bitmap rows), counts
//      the cliques under each first-level vertex x_i1, scans those counts and
//      writes every clique at its owner's offset plus its sub-tree's offset
//      -- a deterministic layout, so the warps of a CTA write without any
//      global atomics;
//   4. the run is handed to the caller's callback, then the buffer is reused.
// Inside a sub-tree one warp walks the ordered chains x_i1 < x_i2 < ... with
// its candidate sets in a per-warp stack (lanes over words) and writes the
// last level's elements by rank selection, 32 cliques at a time.
#include <algorithm>
#include <climits>
#include <vector>

#include "count_common.cuh"

namespace kc {

int num_sms();

namespace {

using cc::Ctx;

constexpr int kListWarps = 8;

// Lowest element of the W-word set S at or above word `low`, removed from S;
// -1 when none is left.  `low` advances to the word of the element.
__device__ int set_pop(uint32_t* S, int& low, int W, int lane)
{
    while (low < W) {
        const int w = low + lane;
        const uint32_t v = w < W ? S[w] : 0u;
        const uint32_t nz = __ballot_sync(kFull, v != 0u);
        if (nz) {
            const int f = __ffs(nz) - 1;
            const uint32_t vf = __shfl_sync(kFull, v, f);
            __syncwarp();
            if (lane == f) S[w] = vf & (vf - 1u);
            __syncwarp();
            low += f;
            return low * 32 + __ffs(vf) - 1;
        }
        low += 32;
    }
    return -1;
}

// Elements of S (words low..W-1) as the last clique member: counts them and,
// with WRITE, stores clique number pos + j for the j-th element.  Lanes
// 0..t-1 hold the ids of the chain's levels in `chid`.
template <bool WRITE>
__device__ uint64_t leaves(const uint32_t* S, int low, int W, const int32_t* sL, int32_t uid, int32_t e1id, int t,
                           int32_t chid, int32_t* out, int kk, int64_t pos, int64_t lim, int lane)
{
    uint64_t run = 0;
    for (int g0 = low; g0 < W; g0 += 32) {
        const int w = g0 + lane;
        const uint32_t v = w < W ? S[w] : 0u;
        const uint32_t pc = (uint32_t)__popc(v);
        uint32_t pre = pc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(kFull, pre, o);
            if (lane >= o) pre += x;
        }
        const uint32_t gt = __shfl_sync(kFull, pre, 31);
        if (WRITE) {
            const uint32_t excl = pre - pc;
            for (uint32_t b = 0; b < gt; b += 32) {
                const uint32_t j = b + (uint32_t)lane;
                int ww = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const uint32_t p = __shfl_sync(kFull, pre, ww + step - 1);
                    if (p <= j) ww += step;
                }
                const uint32_t vw = __shfl_sync(kFull, v, ww);
                const uint32_t ex = __shfl_sync(kFull, excl, ww);
                const int64_t row = pos + (int64_t)run + (int64_t)j;
                const bool ok = j < gt && row < lim;  // rows past the run's buffer are never written
                int32_t* o = out + row * kk;
                for (int c = 0; c < t; ++c) {
                    const int32_t id = __shfl_sync(kFull, chid, c);
                    if (ok) o[2 + c] = id;
                }
                if (ok) {
                    const int leaf = (g0 + ww) * 32 + (int)__fns(vw, 0, (int)(j - ex) + 1);
                    o[0] = uid;
                    o[1] = e1id;
                    o[kk - 1] = sL[leaf];
                }
            }
        }
        run += gt;
    }
    return run;
}

// Cliques of `need` more vertices inside the set in stk[0..W) (words from
// low0 on), each completed by the chain; stk holds `need` levels of W words.
template <bool WRITE>
__device__ uint64_t warp_enum(uint32_t* stk, int W, int need, int low0, const uint32_t* A, int RS,
                              const int32_t* sL, int32_t uid, int32_t e1id, int32_t* out,
                              int kk, int64_t pos, int64_t lim, int lane)
{
    uint64_t total = 0;
    int t = 0, low = low0;
    int lowr = low0;
    int32_t chid = 0;
    for (;;) {
        uint32_t* S = stk + (int64_t)t * W;
        if (need - t == 1) {
            total += leaves<WRITE>(S, low, W, sL, uid, e1id, t, chid, out, kk, pos + (int64_t)total, lim,
                                   lane);
            if (t == 0) break;
            --t;
            low = __shfl_sync(kFull, lowr, t);
            continue;
        }
        const int e = set_pop(S, low, W, lane);
        if (e < 0) {
            if (t == 0) break;
            --t;
            low = __shfl_sync(kFull, lowr, t);
            continue;
        }
        uint32_t* D = S + W;
        const int lc = e >> 5;  // upper rows: the child set lies above e
        const uint32_t* Ae = A + (int64_t)e * RS;
        int cnt = 0;
        for (int w = lc + lane; w < W; w += 32) {
            const uint32_t v = S[w] & Ae[w];
            D[w] = v;
            cnt += __popc(v);
        }
        cnt = (int)__reduce_add_sync(kFull, (unsigned)cnt);
        __syncwarp();
        if (cnt < need - t - 1) continue;
        if (lane == t) {
            lowr = low;
            chid = sL[e];
        }
        ++t;
        low = lc;
    }
    return total;
}

struct LLayout {
    int64_t L, cnt, A, stk, total;
};

__host__ __device__ inline LLayout make_llayout(int W, int RS, int NW, int levels)
{
    const int64_t D = 32LL * W;
    LLayout l;
    l.L = 0;
    l.cnt = D;                 // uint64 per first-level vertex
    l.A = l.cnt + 2 * D;
    l.stk = l.A + D * RS;
    l.total = l.stk + (int64_t)NW * levels * W;
    return l;
}

// Exclusive scan of cnt1[0..d), by one warp.
__device__ void scan_counts(unsigned long long* cnt1, int d, int lane)
{
    unsigned long long carry = 0;
    for (int b0 = 0; b0 < d; b0 += 32) {
        const int j = b0 + lane;
        const unsigned long long v = j < d ? cnt1[j] : 0ull;
        unsigned long long incl = v;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const unsigned long long x = __shfl_up_sync(kFull, incl, s);
            if (lane >= s) incl += x;
        }
        if (j < d) cnt1[j] = carry + incl - v;
        carry += __shfl_sync(kFull, incl, 31);
    }
}

// One CTA per owner of the run: G+(u), per-x_i1 counts, their scan, writes.
template <bool HEAVY>
__global__ void __launch_bounds__(256) k_list(Ctx cb, int W, int levels, const unsigned long long* ooff,
                                              int32_t* out, int64_t lim, uint32_t* gscratch, int64_t tile_words)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, NW = blockDim.x >> 5;
    const int RS = HEAVY ? W : W + 1;
    const LLayout lay = make_llayout(W, RS, NW, levels);
    uint32_t* base = HEAVY ? gscratch + (int64_t)blockIdx.x * tile_words : smem;
    int32_t* sL = (int32_t*)(base + lay.L);
    unsigned long long* cnt1 = (unsigned long long*)(base + lay.cnt);
    uint32_t* A = base + lay.A;
    uint32_t* stk = base + lay.stk + (int64_t)wid * levels * W;
    __shared__ long long s_item;
    const int kk = cb.k, need = kk - 2;

    for (;;) {
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(cb.cursor, 1ull);
        __syncthreads();
        const long long item = s_item;
        cc::OwnerCtx c;
        int32_t r;
        if (!cc::resolve(cb, (int64_t)item, c, r)) break;
        const int64_t b = c.offp[r];
        const int d = (int)(c.offp[r + 1] - b);
        const int32_t uid = c.perm[r];
        const int64_t o = (int64_t)ooff[item];
        for (int j = threadIdx.x; j < d; j += blockDim.x) sL[j] = c.adjp[b + j];
        for (int64_t j = threadIdx.x; j < (int64_t)d * RS; j += blockDim.x) A[j] = 0u;
        __syncthreads();
        cc::build_rows<false, false>(c, sL, nullptr, d, A, RS, wid, NW, lane);
        __syncthreads();
        // from here on sL holds the caller's ids: one load per element of the
        // owner instead of one, waited for, per clique
        for (int j = threadIdx.x; j < d; j += blockDim.x) sL[j] = c.perm[sL[j]];
        __syncthreads();

        // pass 1: cliques under each first-level vertex
        for (int e1 = wid; e1 < d; e1 += NW) {
            const int lo = e1 >> 5;
            int pc = 0;
            for (int w = lo + lane; w < W; w += 32) {
                const uint32_t v = A[(int64_t)e1 * RS + w];
                stk[w] = v;
                pc += __popc(v);
            }
            pc = (int)__reduce_add_sync(kFull, (unsigned)pc);
            __syncwarp();
            const unsigned long long n1 =
                pc < need ? 0ull
                          : warp_enum<false>(stk, W, need, lo, A, RS, sL, uid, 0, out, kk, 0, 0, lane);
            if (lane == 0) cnt1[e1] = n1;
        }
        __syncthreads();
        if (wid == 0) scan_counts(cnt1, d, lane);
        __syncthreads();

        // pass 2: write each sub-tree at its offset
        for (int e1 = wid; e1 < d; e1 += NW) {
            const int lo = e1 >> 5;
            int pc = 0;
            for (int w = lo + lane; w < W; w += 32) {
                const uint32_t v = A[(int64_t)e1 * RS + w];
                stk[w] = v;
                pc += __popc(v);
            }
            pc = (int)__reduce_add_sync(kFull, (unsigned)pc);
            __syncwarp();
            if (pc < need) continue;
            warp_enum<true>(stk, W, need, lo, A, RS, sL, uid, sL[e1], out, kk,
                            o + (int64_t)cnt1[e1], lim, lane);
        }
        __syncthreads();
    }
}

template <int WM>
__device__ __forceinline__ void load_row(const uint32_t* A, int e, uint32_t (&x)[WM])
{
    if (WM == 2) {
        const uint2 v = ((const uint2*)A)[e];
        x[0] = v.x;
        x[1] = v.y;
        return;
    }
#pragma unroll
    for (int q = 0; q < WM / 4; ++q) {
        const uint4 v = ((const uint4*)A)[e * (WM / 4) + q];
        x[4 * q] = v.x;
        x[4 * q + 1] = v.y;
        x[4 * q + 2] = v.z;
        x[4 * q + 3] = v.w;
    }
}

// The cliques made of u, x_e1 and `need` vertices of row e1, in the order of
// their chains: counted, or with WRITE stored from clique number pos on.  A
// warp; every lane holds the whole candidate set, lane t the state of level t,
// and lane j the caller's ids ids[q] of the elements 32 q + j.
template <int WM, bool WRITE>
__device__ unsigned long long walk(const uint32_t* A, const int32_t* sL, const int32_t (&ids)[WM], int e1, int need,
                                   int32_t uid, int32_t* out, int kk, int64_t pos, int64_t lim, int lane)
{
    const bool quads = kk == 4 && ((uintptr_t)out & 15) == 0;  // a clique is one 128-bit store
    const uint32_t lt = cc::mask_below(lane);
    uint32_t C[WM], it[WM], st_C[WM], st_it[WM];
    load_row<WM>(A, e1, C);
    unsigned long long total = 0;
    int32_t chid = sL[e1];  // lane t: id of the chain's t-th vertex
    int t = 0;              // levels below x_e1
#pragma unroll
    for (int q = 0; q < WM; ++q) st_C[q] = st_it[q] = it[q] = 0u;

    // elements of S as the last vertex
    auto leaves = [&](const uint32_t (&S)[WM], int chain) {
#pragma unroll
        for (int q = 0; q < WM; ++q) {
            if (S[q] == 0u) continue;
            const int64_t row = pos + __popc(S[q] & lt);
            const bool ok = ((S[q] >> lane) & 1u) && row < lim;  // rows past the run's buffer are never written
            int32_t* o = out + row * kk;
            if (quads) {
                const int4 v = make_int4(uid, __shfl_sync(kFull, chid, 0), __shfl_sync(kFull, chid, 1), ids[q]);
                if (ok) *(int4*)o = v;
            } else {
                for (int i = 0; i < chain; ++i) {
                    const int32_t id = __shfl_sync(kFull, chid, i);
                    if (ok) o[1 + i] = id;
                }
                if (ok) {
                    o[0] = uid;
                    o[kk - 1] = ids[q];
                }
            }
            pos += __popc(S[q]);
        }
    };

    if (need == 1) {
        if (WRITE) {
            leaves(C, 1);
        } else {
#pragma unroll
            for (int q = 0; q < WM; ++q) total += (unsigned long long)__popc(C[q]);
        }
        return total;
    }
    bool enter = true;
    for (;;) {
        if (enter) {  // a new set: its elements that have enough neighbours above them in it
            uint32_t sum = 0;
#pragma unroll
            for (int q = 0; q < WM; ++q) {
                uint32_t n = 0;
                if ((C[q] >> lane) & 1u) {
                    uint32_t x[WM];
                    load_row<WM>(A, q * 32 + lane, x);
#pragma unroll
                    for (int w = 0; w < WM; ++w) n += (uint32_t)__popc(C[w] & x[w]);
                }
                if (!WRITE) sum += n;
                it[q] = __ballot_sync(kFull, n >= (uint32_t)(need - 1));
            }
            if (!WRITE && need == 2) {  // two vertices missing: the edges inside
                total += (unsigned long long)__reduce_add_sync(kFull, sum);
#pragma unroll
                for (int q = 0; q < WM; ++q) it[q] = 0u;
            }
            enter = false;
        }
        int e = -1;
#pragma unroll
        for (int q = 0; q < WM; ++q)
            if (e < 0 && it[q]) {
                e = q * 32 + __ffs(it[q]) - 1;
                it[q] &= it[q] - 1u;
            }
        if (e < 0) {
            if (t == 0) break;
            --t;
            ++need;
#pragma unroll
            for (int q = 0; q < WM; ++q) {
                C[q] = __shfl_sync(kFull, st_C[q], t);
                it[q] = __shfl_sync(kFull, st_it[q], t);
            }
            continue;
        }
        uint32_t Cn[WM];
        load_row<WM>(A, e, Cn);
#pragma unroll
        for (int q = 0; q < WM; ++q) Cn[q] &= C[q];
        if (WRITE) {
            const int32_t id = sL[e];
            if (lane == t + 1) chid = id;
            if (need == 2) {
                leaves(Cn, t + 2);
                continue;
            }
        }
        if (lane == t) {
#pragma unroll
            for (int q = 0; q < WM; ++q) {
                st_C[q] = C[q];
                st_it[q] = it[q];
            }
        }
        ++t;
        --need;
#pragma unroll
        for (int q = 0; q < WM; ++q) C[q] = Cn[q];
        enter = true;
    }
    return total;
}

// Owners of 33..32 WM elements, a CTA each: as k_list, with the sets and the
// chain in registers (walk), the counts of pass 1 closed two levels early and a
// clique of four ids stored at once.  Bound: the latency of an owner's chains,
// a few hundred owners to a run.  k = 4, against k_list: a run of 325 owners of
// two words 207 -> 59 us, of 3 owners of four words 263 -> 89 us; a listing of
// 6.7e6 cliques with owners of eight words 1.49 -> 0.89 ms.  Wider owners stay
// with k_list: sets in registers gained nothing there (0.357 against 0.362 ms
// at k = 3, 16 words).
template <int WM>
__global__ void __launch_bounds__(256) k_list_reg(Ctx cb, const unsigned long long* ooff, int32_t* out, int64_t lim)
{
    constexpr int D = 32 * WM;
    __shared__ __align__(16) uint32_t A[D * WM];
    __shared__ int32_t sL[D];
    __shared__ unsigned long long cnt1[D];
    __shared__ long long s_item;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, NW = blockDim.x >> 5;
    const int kk = cb.k, need = kk - 2;
    for (;;) {
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(cb.cursor, 1ull);
        __syncthreads();
        const long long item = s_item;
        cc::OwnerCtx c;
        int32_t r;
        if (!cc::resolve(cb, (int64_t)item, c, r)) break;
        const int64_t b = c.offp[r];
        const int d = (int)(c.offp[r + 1] - b);
        const int32_t uid = c.perm[r];
        const int64_t o = (int64_t)ooff[item];
        for (int j = threadIdx.x; j < d; j += blockDim.x) sL[j] = c.adjp[b + j];
        for (int j = threadIdx.x; j < d * WM; j += blockDim.x) A[j] = 0u;
        __syncthreads();
        cc::build_rows<false, false>(c, sL, nullptr, d, A, WM, wid, NW, lane);
        __syncthreads();
        for (int j = threadIdx.x; j < d; j += blockDim.x) sL[j] = c.perm[sL[j]];
        __syncthreads();
        int32_t ids[WM];
#pragma unroll
        for (int q = 0; q < WM; ++q) ids[q] = q * 32 + lane < d ? sL[q * 32 + lane] : 0;
        for (int e1 = wid; e1 < d; e1 += NW) {
            const unsigned long long n1 = walk<WM, false>(A, sL, ids, e1, need, uid, out, kk, 0, 0, lane);
            if (lane == 0) cnt1[e1] = n1;
        }
        __syncthreads();
        if (wid == 0) scan_counts(cnt1, d, lane);
        __syncthreads();
        for (int e1 = wid; e1 < d; e1 += NW)
            walk<WM, true>(A, sL, ids, e1, need, uid, out, kk, o + (int64_t)cnt1[e1], lim, lane);
        __syncthreads();
    }
}

// Owners of at most 32 elements, a warp each, rows and chain in registers: the
// cliques are met in the order the layout wants (x_i1, then the chains below it,
// ascending), so one pass writes them from the owner's offset on.  k_list
// counted every sub-tree first, with a CTA of one warp per owner: 754 us for
// the 17,000 owners of a 20,000-vertex power-law graph at k = 4; here 108 us, 67
// with a clique of four ids stored at once.
__global__ void __launch_bounds__(256) k_list_w1(Ctx cb, const unsigned long long* ooff, int32_t* out, int64_t lim)
{
    __shared__ cc::SmallBuf<1> s_buf[8];
    const int lane = threadIdx.x & 31;
    const uint32_t lt = cc::mask_below(lane);
    const int kk = cb.k, r0 = kk - 1;
    const bool quads = kk == 4 && ((uintptr_t)out & 15) == 0;  // a clique is one 128-bit store
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(cb.cursor, 1ull);
        item = __shfl_sync(kFull, item, 0);
        cc::OwnerCtx c;
        int32_t r;
        if (!cc::resolve(cb, (int64_t)item, c, r)) break;
        const int64_t b = c.offp[r];
        const int d = (int)(c.offp[r + 1] - b);
        const int32_t xs[1] = {lane < d ? c.adjp[b + lane] : INT_MAX};
        const uint32_t cols[1] = {0u};
        uint32_t rows[1][1];
        const cc::Gr g{c.offp, c.adjp, c.core, c.core_lo, c.core_tw, c.total};
        cc::build_rows_small<1, false>(c, g, xs, d, cols, 0, s_buf[threadIdx.x >> 5], lane, rows);
        const uint32_t up = rows[0][0];
        const int32_t id = lane < d ? c.perm[xs[0]] : 0, uid = c.perm[r];
        int64_t pos = (int64_t)ooff[item];
        // level t's state in lane t: candidate set, elements left to visit, element
        uint32_t st_C = 0, st_it = 0;
        int st_e = 0, t = 0;
        uint32_t C = d >= 32 ? kFull : ((1u << d) - 1u);
        uint32_t it = __ballot_sync(kFull, ((C >> lane) & 1u) && __popc(C & up) >= r0 - 1);
        for (;;) {
            if (it == 0u) {
                if (t == 0) break;
                --t;
                C = __shfl_sync(kFull, st_C, t);
                it = __shfl_sync(kFull, st_it, t);
                continue;
            }
            const int e = __ffs(it) - 1;
            it &= it - 1u;
            const uint32_t Cn = C & __shfl_sync(kFull, up, e);
            if (lane == t) {
                st_C = C;
                st_it = it;
                st_e = e;
            }
            ++t;
            const int need = r0 - t;  // vertices to choose in Cn
            if (need > 1) {
                C = Cn;
                it = __ballot_sync(kFull, ((C >> lane) & 1u) && __popc(C & up) >= need - 1);
                continue;
            }
            const int64_t row = pos + __popc(Cn & lt);
            const bool ok = ((Cn >> lane) & 1u) && row < lim;  // rows past the run's buffer are never written
            int32_t* o = out + row * kk;
            if (quads) {
                const int32_t i1 = __shfl_sync(kFull, id, __shfl_sync(kFull, st_e, 0));
                const int32_t i2 = __shfl_sync(kFull, id, __shfl_sync(kFull, st_e, 1));
                if (ok) *(int4*)o = make_int4(uid, i1, i2, id);
                pos += __popc(Cn);
                --t;
                continue;
            }
            for (int q = 0; q < t; ++q) {
                const int32_t cid = __shfl_sync(kFull, id, __shfl_sync(kFull, st_e, q));
                if (ok) o[1 + q] = cid;
            }
            if (ok) {
                o[0] = uid;
                o[kk - 1] = id;
            }
            pos += __popc(Cn);
            --t;  // C and it are still this level's
        }
    }
}

// k = 1 (every vertex) and k = 2 (every edge u < x, x in Gamma+(u)).
__global__ void k_list_small(Ctx cb, const unsigned long long* ooff, int32_t* out, int64_t lim)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t item = warp; item < cb.nitems; item += nwarps) {
        cc::OwnerCtx c;
        int32_t r;
        if (!cc::resolve(cb, item, c, r)) break;
        const int64_t o = (int64_t)ooff[item];
        const int32_t uid = c.perm[r];
        if (cb.k == 1) {
            if (lane == 0 && o < lim) out[o] = uid;
            continue;
        }
        const int64_t b = c.offp[r];
        const int d = (int)(c.offp[r + 1] - b);
        for (int j = lane; j < d && o + j < lim; j += 32) {
            out[(o + j) * 2] = uid;
            out[(o + j) * 2 + 1] = c.perm[c.adjp[b + j]];
        }
    }
}

}  // namespace

kc_status list_run(const kc_graph* g, int k, unsigned flags, int32_t* buf, int64_t cap, kc_list_fn fn, void* user,
                   uint64_t* listed, cudaStream_t s)
{
    const bool dev = (flags & KC_DEVICE_PTRS) != 0;
    const int32_t n = g->n;
    *listed = 0;
    if (n == 0) return KC_OK;
    Scratch sc(s);
    unsigned long long* small = nullptr;  // [0..1] total, [2..15] cursors
    KC_TRY(sc.get(&small, 24));
    KC_CK(cudaMemsetAsync(small, 0, 24 * sizeof(unsigned long long), s));

    // queue (owners by d+ descending) and per-owner counts, on the host
    std::vector<int32_t> hq(n);
    KC_CK(cudaMemcpyAsync(hq.data(), g->queue, (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    std::vector<unsigned long long> cnt(n, 0ull);  // rank space
    int64_t qend = n;
    if (k == 1) {
        std::fill(cnt.begin(), cnt.end(), 1ull);
    } else if (k == 2) {
        std::vector<int32_t> dp(n);
        KC_CK(cudaMemcpyAsync(dp.data(), g->dplus, (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        KC_CK(cudaStreamSynchronize(s));
        for (int32_t r = 0; r < n; ++r) cnt[r] = (unsigned long long)dp[r];
        qend = ge_at(g, 1);
    } else {
        qend = ge_at(g, k - 1);
        unsigned long long* po = nullptr;
        KC_TRY(sc.get(&po, n));
        KC_CK(cudaMemsetAsync(po, 0, (size_t)n * sizeof(unsigned long long), s));
        Plan plan;
        const bool planned = find_plan(g, k, false, &plan);
        int64_t slot_words = 0;
        const int64_t hw = heavy_scratch_words(g, k, &slot_words, planned ? &plan : nullptr);
        uint32_t* heavy = nullptr;
        if (hw > 0) KC_TRY(sc.get(&heavy, hw));
        CountArgs a;
        a.plan = planned ? &plan : nullptr;
        a.k = k;
        a.colours = 0;
        a.seed = 0;
        a.per_vertex = false;
        a.total = small;
        a.pv = nullptr;
        a.po = po;
        a.work = nullptr;
        a.sc = &sc;
        KC_TRY(count_launch(g, a, small + 2, heavy, hw, s));
        KC_CK(cudaMemcpyAsync(cnt.data(), po, (size_t)n * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    }
    KC_CK(cudaStreamSynchronize(s));
    if (qend <= 0) return KC_OK;

    // device buffers for one run
    unsigned long long* doff = nullptr;
    KC_TRY(sc.get(&doff, qend));
    int32_t* dbuf = buf;
    if (!dev) KC_TRY(sc.get(&dbuf, cap * (int64_t)k));
    unsigned long long* cursors = small + 2;

    // widest-owner tiles for the listing kernel
    const int Wh = std::max(1, (g->max_dplus + 31) / 32);
    const int levels = std::max(1, k - 2);
    const LLayout hl = make_llayout(Wh, Wh, kListWarps, levels);
    const int64_t tile_words = (hl.total + 3) & ~3LL;  // keeps every tile 16-byte aligned
    int64_t h0 = 0, h1 = 0;
    class_range(g, k, 0, &h0, &h1);
    const int sms = num_sms();
    const int64_t htiles = k >= 3 ? std::min<int64_t>(std::max<int64_t>(h1 - h0, 0), sms) : 0;
    uint32_t* htile = nullptr;
    if (htiles > 0) KC_TRY(sc.get(&htile, tile_words * htiles));

    std::vector<unsigned long long> hoff;
    uint64_t delivered = 0;
    int64_t a0 = 0;
    while (a0 < qend) {
        unsigned long long T = 0;
        int64_t b0 = a0;
        while (b0 < qend) {
            const unsigned long long cu = cnt[hq[b0]];
            if (cu > (unsigned long long)cap) return KC_ENOMEM;  // one owner's cliques exceed the buffer
            if (T + cu > (unsigned long long)cap) break;
            T += cu;
            ++b0;
        }
        if (T == 0) {  // only owners without cliques remain in this run
            a0 = b0;
            continue;
        }
        hoff.assign((size_t)(b0 - a0), 0ull);
        unsigned long long acc = 0;
        for (int64_t i = a0; i < b0; ++i) {
            hoff[(size_t)(i - a0)] = acc;
            acc += cnt[hq[i]];
        }
        KC_CK(cudaMemcpyAsync(doff, hoff.data(), hoff.size() * sizeof(unsigned long long), cudaMemcpyHostToDevice,
                              s));
        KC_CK(cudaMemsetAsync(cursors, 0, kCursorWords * sizeof(unsigned long long), s));
        Ctx base;
        cc::set_graph(base, g);
        base.qoff = 0;
        base.qstride = 1;
        base.gd = nullptr;
        base.gq0 = nullptr;
        base.gpre = nullptr;
        base.ng = 0;
        base.k = k;
        base.colours = 0;
        base.seed = 0;
        base.pair = 0;
        base.pthr = 0;
        base.total = small;
        base.pv = nullptr;
        base.po = nullptr;
        base.work = nullptr;
        if (k <= 2) {
            Ctx c = base;
            c.q0 = a0;
            c.q1 = b0;
            c.nitems = b0 - a0;
            c.cursor = cursors;
            const int grid = (int)std::min<int64_t>((c.nitems + 7) / 8, (int64_t)sms * 16);
            k_list_small<<<grid, 256, 0, s>>>(c, doff, dbuf, (int64_t)T);
            KC_LAUNCHED();
        } else {
            for (int slot = 0; slot < kOwnerSlots; ++slot) {
                int64_t q0 = 0, q1 = 0;
                class_range(g, k, slot, &q0, &q1);
                const int64_t lo = std::max(q0, a0), hi = std::min(q1, b0);
                if (hi <= lo) continue;
                Ctx c = base;
                c.q0 = lo;
                c.q1 = hi;
                c.nitems = hi - lo;
                c.cursor = cursors + slot;
                const unsigned long long* off = doff + (lo - a0);
                if (slot == 0) {
                    const int grid = (int)std::min<int64_t>(c.nitems, htiles);
                    k_list<true><<<grid, kListWarps * 32, 0, s>>>(c, Wh, levels, off, dbuf, (int64_t)T, htile,
                                                                   tile_words);
                    KC_LAUNCHED();
                    continue;
                }
                const int W = slot_words(slot);
                if (W == 1) {
                    const int grid = (int)std::min<int64_t>((c.nitems + 7) / 8,
                                                            (int64_t)sms * cc::blocks_per_sm(k_list_w1, 256, 0));
                    k_list_w1<<<grid, 256, 0, s>>>(c, off, dbuf, (int64_t)T);
                    KC_LAUNCHED();
                    continue;
                }
                if (W <= 8) {
                    auto kern = W == 2 ? k_list_reg<2> : (W == 4 ? k_list_reg<4> : k_list_reg<8>);
                    const int grid = (int)std::min<int64_t>(c.nitems, (int64_t)sms * cc::blocks_per_sm(kern, 256, 0));
                    kern<<<grid, 256, 0, s>>>(c, off, dbuf, (int64_t)T);
                    KC_LAUNCHED();
                    continue;
                }
                const int NW = kListWarps;
                const LLayout l = make_llayout(W, W + 1, NW, levels);
                const size_t smem = (size_t)l.total * 4;
                auto kern = k_list<false>;
                KC_CK(cc::allow_smem(kern, smem));
                const int grid =
                    (int)std::min<int64_t>(c.nitems, (int64_t)sms * cc::blocks_per_sm(kern, NW * 32, smem));
                kern<<<grid, NW * 32, smem, s>>>(c, W, levels, off, dbuf, (int64_t)T, nullptr, 0);
                KC_LAUNCHED();
            }
        }
        if (!dev)
            KC_CK(cudaMemcpyAsync(buf, dbuf, (size_t)T * k * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        KC_CK(cudaStreamSynchronize(s));
        delivered += T;
        *listed = delivered;
        if (fn(user, buf, (int64_t)T) != 0) return KC_ECANCELED;
        a0 = b0;
    }
    return KC_OK;
}

}  // namespace kc

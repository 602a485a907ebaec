// close.cu -- candidate sets closed on a compact copy of their subgraph
// (Reduce 3, Alg. 1; Sec. 3), for the 4-, 8- and 16-word owner classes.
//
// The ordered search of dfs.cu walks the chains x_i1 < x_i2 < ... until three
// vertices are missing.  Here the chain stops one level earlier: a candidate
// set C (the elements of G+(u) above the chain that are adjacent to all of
// it) that still needs four vertices is closed at once, with the number of
// 4-cliques of G[C] through every v of C.
//
//   1. Compact copy.  The elements of C are renumbered 0..c-1 and the rows of
//      G[C] rebuilt by ballots: c rows of ceil(c/32) words instead of c rows
//      of the owner's 9..16 words (the candidate sets of a power-law graph's
//      hub cores hold a third of Gamma+(u), and every later step is a pass
//      over rows).  Row a is then one or two 128-bit shared loads.
//   2. If at least half of the pairs of C are edges, the rows are flipped:
//      B is the complement of G[C], else B = G[C].  X_v is v's row of B.
//   3. One thread per v.  With nb_v = |X_v|, co(v,a) = |X_v & X_a|, M the
//      edges of B, t_v the triangles of B through v, T all triangles of B,
//      d = c - 1 - nb_v, and N(v) the neighbours of v in G[C]: the complement
//      edges inside N(v) are  M_v = M - nb_v - sum_{a in X_v} (nb_a - 1) + t_v,
//      the complement 2-paths inside N(v)  P_v = sum_{a in N(v)}
//      C(nb_a - co(v,a), 2), the complement triangles inside N(v)
//      T_v = T - sum_{a in X_v} t_a + sum_{edges ab of B in X_v} co(a,b) - k_v
//      with k_v the 4-cliques of B through v, and by inclusion-exclusion over
//      the complement edges of a triple the 4-cliques through v number
//        C(d,3) - (d-2) M_v + P_v - T_v.
//      P_v and t_v come from one pass over all rows a of C, the same row for
//      every thread (a broadcast load).
//   4. The two sums over edges ab of B inside X_v come from a walk over the
//      triangles of B, each visited once (v < a < b) and credited to its
//      three corners: m = |X_v & X_a & X_b| sums to 3 k_v over the triangles
//      through v.  With B = G[C] this walk alone is the answer.
// All terms fit 32 bits: c <= 511, C(511,3) < 2^25, 512 C(511,2) < 2^27, and
// three times the sum of t_a over a row is below 2^28.
//
// Bound: population counts (16 lanes per SM and clock) and instruction issue.
// Step 3 needs c ceil(c/32) counts per element; adding words bitwise first
// (full adders, three-input logic) brings 5 or 8 words down to 3 or 4 counts.
//
// Layout: one launch per row width WC of the copy, so that a launch runs one
// short body (all widths in one kernel were 300 KB of code and waited for
// instructions more than for anything else) with shared memory for its own
// sets.  A team is one warp up to 128 elements (no barrier but the warp's),
// two warps up to 256 and four above; when the elements do not fill the last
// round of threads, several threads share an element and split the rows.
#include <algorithm>

#include "count_common.cuh"

namespace kc {

int num_sms();

namespace {

using cc::Ctx;
using cc::add_total;
using cc::close_bin;
using cc::kCloseBins;
using cc::mask_above;
using cc::mask_below;


constexpr int kPush = 7;       // entries a lane queues at a time
constexpr int kQueue = 256;    // entries of a queue: 31 + 32 * kPush at most

template <int NT>
__device__ __forceinline__ void sync()
{
    if (NT == 32) __syncwarp(); else __syncthreads();
}

// Sum over the NT cooperating threads; ends with their barrier (values
// written to shared memory before the call are visible after it).
template <int NT>
__device__ __forceinline__ uint32_t team_sum(uint32_t v, uint32_t* red, int lane, int wid)
{
    v = __reduce_add_sync(kFull, v);
    if (NT == 32) {
        __syncwarp();
        return v;
    }
    if (lane == 0) red[wid] = v;
    __syncthreads();
    uint32_t s = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) s += red[w];
    return s;
}

// Shared working set of one team for sets of up to D elements.
struct Team {
    uint32_t* B;      // rows of the compact copy
    uint16_t* pos;    // [D] element of G+(u) behind compact index j
    uint16_t* nb;     // [D] c - 1 - degree
    int32_t* tt;      // [D] triangles of B through j
    int32_t* acc;     // [D] sums credited to j
    uint32_t* red;    // [32] partial sums of the team's warps
    uint32_t* queue;  // [warps][2][kQueue] edges and triangles found and not yet used
};

// Words a compact row takes (stride), by row width WC: vector loads need 2 or
// a multiple of 4; 12 instead of 8 spreads random rows over all banks.
__host__ __device__ constexpr int row_words(int WC) { return WC <= 2 ? WC : (WC <= 4 ? 4 : (WC <= 12 ? 12 : 16)); }

template <int WC>
__device__ __forceinline__ void load_row(const uint32_t* B, int j, uint32_t (&x)[WC])
{
    constexpr int SW = row_words(WC);
    const uint32_t* p = B + j * SW;
    if (SW >= 4) {
#pragma unroll
        for (int q = 0; q < WC / 4; ++q) {
            const uint4 a = ((const uint4*)p)[q];
            x[4 * q] = a.x;
            x[4 * q + 1] = a.y;
            x[4 * q + 2] = a.z;
            x[4 * q + 3] = a.w;
        }
        constexpr int T = WC & ~3;
        if ((WC & 3) == 1) x[T] = p[T];
        if ((WC & 3) >= 2) {
            const uint2 a = *(const uint2*)(p + T);
            x[T] = a.x;
            x[WC & 2 ? T + 1 : T] = a.y;
        }
        if ((WC & 3) == 3) x[WC - 1] = p[WC - 1];
    } else if (SW == 2) {
        const uint2 a = *(const uint2*)p;
        x[0] = a.x;
        x[WC - 1] = a.y;
    } else {
        x[0] = p[0];
    }
}

__device__ __forceinline__ uint32_t maj(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a ^ b)); }

// Population count of words x[I..N): groups of seven (three counts) or three
// (two counts) are added bitwise first.
template <int N, int I = 0>
__device__ __forceinline__ uint32_t popc_words(const uint32_t (&x)[N])
{
    if constexpr (N - I >= 7) {
        const uint32_t s1 = x[I] ^ x[I + 1] ^ x[I + 2], c1 = maj(x[I], x[I + 1], x[I + 2]);
        const uint32_t s2 = x[I + 3] ^ x[I + 4] ^ x[I + 5], c2 = maj(x[I + 3], x[I + 4], x[I + 5]);
        const uint32_t s = s1 ^ s2 ^ x[I + 6], c3 = maj(s1, s2, x[I + 6]);
        const uint32_t t = c1 ^ c2 ^ c3, f = maj(c1, c2, c3);
        return (uint32_t)__popc(s) + 2u * (uint32_t)__popc(t) + 4u * (uint32_t)__popc(f) + popc_words<N, I + 7>(x);
    } else if constexpr (N - I >= 5) {
        const uint32_t s1 = x[I] ^ x[I + 1] ^ x[I + 2], c1 = maj(x[I], x[I + 1], x[I + 2]);
        const uint32_t s = s1 ^ x[I + 3] ^ x[I + 4], c2 = maj(s1, x[I + 3], x[I + 4]);
        return (uint32_t)__popc(s) + 2u * ((uint32_t)__popc(c1) + (uint32_t)__popc(c2)) + popc_words<N, I + 5>(x);
    } else if constexpr (N - I >= 3) {
        const uint32_t s = x[I] ^ x[I + 1] ^ x[I + 2], c = maj(x[I], x[I + 1], x[I + 2]);
        return (uint32_t)__popc(s) + 2u * (uint32_t)__popc(c) + popc_words<N, I + 3>(x);
    } else if constexpr (N - I >= 1) {
        return (uint32_t)__popc(x[I]) + popc_words<N, I + 1>(x);
    } else {
        return 0u;
    }
}

template <int WC>
__device__ __forceinline__ uint32_t co_count(const uint32_t (&a)[WC], const uint32_t (&b)[WC])
{
    uint32_t z[WC];
#pragma unroll
    for (int w = 0; w < WC; ++w) z[w] = a[w] & b[w];
    return popc_words<WC>(z);
}

// Threads that share one element in a round whose first element is `base`:
// the largest power of two S with S * (elements left) <= NT, at most 32.
template <int NT>
__device__ __forceinline__ int share_log(int c, int base)
{
    const int left = c - base;
    int lg = 0;
#pragma unroll 1
    while (lg < 5 && (left << (lg + 1)) <= NT) ++lg;
    return lg;
}

// Sum over the S = 1 << lg adjacent lanes that share an element.
__device__ __forceinline__ uint32_t share_sum(uint32_t v, int lg)
{
#pragma unroll 1
    for (int o = 0; o < lg; ++o) v += __shfl_xor_sync(kFull, v, 1 << o);
    return v;
}

// One triangle v < a < b of B (step 4).
template <int WC>
__device__ __forceinline__ void credit_triangle(const Team& t, bool dense, int v, int a, int b)
{
    uint32_t X[WC], Xa[WC], Xb[WC], Y[WC];
    load_row<WC>(t.B, v, X);
    load_row<WC>(t.B, a, Xa);
    load_row<WC>(t.B, b, Xb);
#pragma unroll
    for (int w = 0; w < WC; ++w) Y[w] = X[w] & Xa[w];
    const int m = (int)co_count<WC>(Y, Xb);
    if (dense) {
        atomicAdd(&t.acc[v], 3 * (int)co_count<WC>(Xa, Xb) - m);
        atomicAdd(&t.acc[a], 3 * (int)co_count<WC>(X, Xb) - m);
        atomicAdd(&t.acc[b], 3 * (int)popc_words<WC>(Y) - m);
    } else if (m) {
        atomicAdd(&t.acc[v], m);
        atomicAdd(&t.acc[a], m);
        atomicAdd(&t.acc[b], m);
    }
}

// Queues the set bits of `bits` (n of them in this lane) at q[qn..], as
// tag | (32 w + bit) << shift, at most kPush per lane and call: the lanes'
// shares are laid out by a warp scan.  Removes them from bits and n; returns
// the new length, the same in every lane.
template <int N>
__device__ __forceinline__ int push_bits(uint32_t* q, int qn, uint32_t (&bits)[N], uint32_t& n, uint32_t tag, int shift,
                                         int base, int lane)
{
    uint32_t k = min(n, (uint32_t)kPush), inc = k;
    n -= k;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += x;
    }
    uint32_t* at = q + qn + (inc - k);
#pragma unroll
    for (int w = 0; w < N; ++w)
#pragma unroll 1
        while (bits[w] && k) {
            *at++ = tag | ((uint32_t)(base + w * 32 + __ffs(bits[w]) - 1) << shift);
            bits[w] &= bits[w] - 1u;
            --k;
        }
    __syncwarp();
    return qn + (int)__shfl_sync(kFull, inc, 31);
}

// Step 4 by a team: every warp takes the elements v of its rounds (or its
// share of their bits) and queues their edges v < a of B; 32 edges at a time,
// one per lane, find their common elements b > a and queue the triangles; 32
// triangles at a time are credited.  The two queues keep the warps full
// however unevenly edges and triangles fall (lanes that walked their own v's
// edges and triangles were a third busy).  At most 31 entries wait and 32
// kPush join them, so a queue never overflows.
template <int WC, int NT>
__device__ __forceinline__ uint32_t walk4(const Team& t, bool dense, int c, int wc, int lane, int wid)
{
    constexpr int SW = row_words(WC);
    uint32_t* eq = t.queue + 2 * wid * kQueue;
    uint32_t* tq = eq + kQueue;
    const int tid = wid * 32 + lane;
    uint32_t ntri = 0, n = 0, bits[1] = {0u}, every = 0u;
    int en = 0, tn = 0;             // waiting edges and triangles
    int base = 0, step = 0, v = 0;  // the round: first element, elements, own element
    int q = wc;                     // word of the round's rows
#pragma unroll 1
    for (;;) {
        // the next word with edges of some lane
        while (!__any_sync(kFull, n != 0u)) {
            if (++q >= wc) {
                base += step;
                if (base >= c) break;
                const int lg = share_log<NT>(c, base);
                const int sub = tid & ((1 << lg) - 1);
                step = NT >> lg;
                v = base + (tid >> lg);
                q = (base + ((wid * 32) >> lg)) >> 5;
                // the bits of a word that fall to this lane: every S-th
                every = (lg == 0 ? kFull : (lg == 1 ? 0x55555555u : (lg == 2 ? 0x11111111u : (lg == 3 ? 0x01010101u : (lg == 4 ? 0x00010001u : 1u))))) << sub;
                if (q >= wc) continue;  // this warp has no element in the round
            }
            bits[0] = (v < c && q >= (v >> 5)) ? t.B[v * SW + q] & every & (q == (v >> 5) ? mask_above(v & 31) : kFull) : 0u;
            n = (uint32_t)__popc(bits[0]);
        }
        const bool last = base >= c;
        if (!last) en = push_bits<1>(eq, en, bits, n, (uint32_t)v, 10, q * 32, lane);
#pragma unroll 1
        while (last ? en + tn > 0 : en >= 32) {
            const int k = min(en, 32);
            en -= k;
            uint32_t Y[WC], ny = 0, e = 0;
#pragma unroll
            for (int w = 0; w < WC; ++w) Y[w] = 0u;
            if (lane < k) {
                e = eq[en + lane];
                const int u = (int)(e & 1023u), a = (int)(e >> 10), qa = a >> 5;
                const uint32_t above = mask_above(a & 31);
                uint32_t X[WC], Xa[WC];
                load_row<WC>(t.B, u, X);
                load_row<WC>(t.B, a, Xa);
#pragma unroll
                for (int w = 0; w < WC; ++w) Y[w] = X[w] & Xa[w] & (w > qa ? kFull : (w == qa ? above : 0u));
                ny = popc_words<WC>(Y);
                if (dense) {
                    atomicAdd(&t.acc[u], -3 * t.tt[a]);
                    atomicAdd(&t.acc[a], -3 * t.tt[u]);
                }
            }
            ntri += ny;
            bool more = __any_sync(kFull, ny != 0u);
#pragma unroll 1
            do {
                if (more) {
                    tn = push_bits<WC>(tq, tn, Y, ny, e, 20, 0, lane);
                    more = __any_sync(kFull, ny != 0u);
                }
                const int keep = last && en == 0 && !more ? 0 : 31;
#pragma unroll 1
                while (tn > keep) {
                    const int kt = min(tn, 32);
                    tn -= kt;
                    if (lane < kt) {
                        const uint32_t x = tq[tn + lane];
                        credit_triangle<WC>(t, dense, (int)(x & 1023u), (int)((x >> 10) & 1023u), (int)(x >> 20));
                    }
                    __syncwarp();
                }
            } while (more);
        }
        if (last) break;
    }
    return ntri;
}

// The 4-cliques of G[C] through every element of C, by a team of NT threads:
// credit(j, K) is called once per element j with a non-zero K.  t.pos holds C
// (c >= 4 elements, visible to the team), T its owner's symmetric rows
// (stride RS).  Returns the number of 4-cliques (every thread); ends with the
// team's barrier.
template <int WC, int NT, typename Credit>
__device__ __forceinline__ unsigned long long close_set(const Team& t, int c, const uint32_t* __restrict__ T, int RS,
                                                        int lane, int wid, unsigned long long* wk, Credit credit)
{
    constexpr int SW = row_words(WC), NW = NT / 32;
    const int wc = (c + 31) >> 5;
    const int tid = wid * 32 + lane;
    // 1. rows: ballot jw of row i holds the adjacency of pos[i] to elements
    // 32 jw .. 32 jw + 31; four rows at a time, stored by four lanes
#pragma unroll 1
    for (int jw = 0; jw < WC; ++jw) {
        const int j = jw * 32 + lane;
        const bool ok = j < c;
        const int p = ok ? (int)t.pos[j] : 0;
        const uint32_t* Tp = T + (p >> 5);
        const uint32_t bit = ok ? 1u << (p & 31) : 0u;
#pragma unroll 1
        for (int i0 = 4 * wid; i0 < c; i0 += 4 * NW) {
            const uint2 pp = *(const uint2*)(t.pos + i0);  // rows past c - 1 read as row 0
            const int p0 = (int)(pp.x & 0xffffu), p1 = i0 + 1 < c ? (int)(pp.x >> 16) : 0;
            const int p2 = i0 + 2 < c ? (int)(pp.y & 0xffffu) : 0, p3 = i0 + 3 < c ? (int)(pp.y >> 16) : 0;
            const uint32_t v0 = Tp[p0 * RS], v1 = Tp[p1 * RS], v2 = Tp[p2 * RS], v3 = Tp[p3 * RS];
            const uint32_t b0 = __ballot_sync(kFull, v0 & bit), b1 = __ballot_sync(kFull, v1 & bit);
            const uint32_t b2 = __ballot_sync(kFull, v2 & bit), b3 = __ballot_sync(kFull, v3 & bit);
            const uint32_t mine = lane & 2 ? (lane & 1 ? b3 : b2) : (lane & 1 ? b1 : b0);
            if (lane < 4 && i0 + lane < c) t.B[(i0 + lane) * SW + jw] = mine;
        }
    }
    sync<NT>();
    // 2. degrees; flip to the complement when it is the sparser side
    uint32_t loc = 0;
#pragma unroll 1
    for (int v = tid; v < c; v += NT) {
        uint32_t X[WC];
        load_row<WC>(t.B, v, X);
        const uint32_t nbv = (uint32_t)(c - 1) - popc_words<WC>(X);
        t.nb[v] = (uint16_t)nbv;
        t.acc[v] = 0;
        loc += nbv;
    }
    const uint32_t nbsum = team_sum<NT>(loc, t.red, lane, wid);
    const bool dense = 2u * nbsum <= (uint32_t)c * (uint32_t)(c - 1);
    int Tall = 0;
    if (dense) {
    #pragma unroll 1
    for (int v = tid; v < c; v += NT) {
#pragma unroll
            for (int w = 0; w < WC; ++w) {
                const int left = c - 32 * w;
                uint32_t m = left >= 32 ? kFull : (left > 0 ? mask_below(left) : 0u);
                if (w == (v >> 5)) m &= ~(1u << (v & 31));
                t.B[v * SW + w] = ~t.B[v * SW + w] & m;
            }
        }
        sync<NT>();
        // 3. one pass over all rows a: co(v,a) against every v
        const int M = (int)(nbsum >> 1);
        uint32_t tl = 0;
    #pragma unroll 1
    for (int base = 0; base < c;) {
            const int lg = share_log<NT>(c, base), S = 1 << lg;
            const int sub = tid & (S - 1), v = base + (tid >> lg);
            const bool on = v < c;
            uint32_t X[WC];
            load_row<WC>(t.B, on ? v : 0, X);
            uint32_t t2 = 0, s1 = 0, P2 = 0;
            const uint32_t* own = t.B + (on ? v : 0) * SW;
#pragma unroll 1
            for (int q = 0; q < wc; ++q) {
                uint32_t xw = own[q] >> sub;
                const int lim = min(32, c - q * 32);
#pragma unroll 4
                for (int b = sub; b < lim; b += S) {
                    const int a = q * 32 + b;
                    uint32_t Xa[WC];
                    load_row<WC>(t.B, a, Xa);
                    const uint32_t co = co_count<WC>(X, Xa), nba = t.nb[a], rest = nba - co;
                    if (xw & 1u) {
                        t2 += co;
                        s1 += nba;
                    } else {
                        P2 += rest * (rest - 1u);
                    }
                    xw >>= S & 31;
                }
            }
            if (lg) {
                t2 = share_sum(t2, lg);
                s1 = share_sum(s1, lg);
                P2 = share_sum(P2, lg);
            }
            if (on && sub == 0) {
                const int nbv = t.nb[v], d = c - 1 - nbv, tv = (int)(t2 >> 1);
                const int Mv = M - nbv - ((int)s1 - nbv) + tv;
                t.tt[v] = tv;
                t.acc[v] = -3 * (d * (d - 1) * (d - 2) / 6 - Mv * (d - 2) + (int)(P2 >> 1));
                tl += (uint32_t)tv;
            }
            base += NT >> lg;
        }
        Tall = (int)(team_sum<NT>(tl, t.red + 8, lane, wid) / 3u);
    }
    // 4. triangles of B
    const uint32_t steps = walk4<WC, NT>(t, dense, c, wc, lane, wid);
    sync<NT>();
    unsigned long long sum = 0;
#pragma unroll 1
    for (int v = tid; v < c; v += NT) {
        const int K = dense ? -Tall - t.acc[v] / 3 : t.acc[v] / 3;
        sum += (unsigned long long)K;
        if (K) credit(v, (uint32_t)K);
    }
    if (wk) {
        *wk += (unsigned long long)steps * (unsigned)(WC * (dense ? 4 : 2));
#pragma unroll 1
        for (int v = tid; v < c; v += NT) *wk += (unsigned long long)((dense ? c + 1 : 1) * WC);
    }
    // an element's 4-cliques are below 2^25, their sum below 2^34
    sum = cc::warp_sum64(sum);
    if (NT == 32) {
        __syncwarp();
        return sum / 4u;
    }
    uint32_t* r = t.red + 16;  // [NW][2]
    if (lane == 0) {
        r[2 * wid] = (uint32_t)sum;
        r[2 * wid + 1] = (uint32_t)(sum >> 32);
    }
    __syncthreads();
    unsigned long long all = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) all += ((unsigned long long)r[2 * w + 1] << 32) | r[2 * w];
    return all / 4u;
}

// Lists the elements of the word set held by a warp's lanes (lane w: word w,
// Wd words) into t.pos, the warps of the team sharing the words.  The caller
// synchronises the team.
template <int NT>
__device__ __forceinline__ void list_set(const Team& t, uint32_t u, int Wd, int lane, int wid)
{
    const int pc = __popc(u);
    int inc = pc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += x;
    }
#pragma unroll 1
    for (int w = wid; w < Wd; w += NT / 32) {
        const uint32_t uw = __shfl_sync(kFull, u, w);
        const int ex = __shfl_sync(kFull, inc - pc, w);
        if ((uw >> lane) & 1u) t.pos[ex + __popc(uw & mask_below(lane))] = (uint16_t)(w * 32 + lane);
    }
}

__device__ __forceinline__ uint32_t upper_word(const uint32_t* __restrict__ T, int RS, int e, int Wd, int lane)
{
    const int we = e >> 5;
    uint32_t v = (lane >= we && lane < Wd) ? T[e * RS + lane] : 0u;
    if (lane == we) v &= mask_above(e & 31);
    return v;
}

struct TeamLayout {
    int B, pos, nb, tt, acc, red, queue, total;  // byte offsets
};

// Working set of a team of NW warps for rows of WC words.
__host__ __device__ constexpr TeamLayout team_layout(int WC, int NW)
{
    const int D = 32 * WC;
    TeamLayout l{};
    l.B = 0;
    l.tt = l.B + D * row_words(WC) * 4;
    l.acc = l.tt + D * 4;
    l.pos = l.acc + D * 4;
    l.nb = l.pos + D * 2;
    l.red = l.nb + D * 2;
    l.queue = l.red + 32 * 4;
    l.total = l.queue + NW * 2 * kQueue * 4;
    return l;
}

constexpr int team_threads(int WC) { return WC <= 4 ? 32 : (WC <= 8 ? 64 : 128); }
constexpr int cta_threads(int WC) { return WC <= 4 ? 128 : team_threads(WC); }
constexpr int ctas_per_sm(int WC) { return WC <= 1 ? 8 : (WC <= 4 ? 6 : (WC <= 8 ? 8 : 3)); }

// Chung-Lu n = 1e6, m = 2e7, k = 6 with memberships, against the pair search of
// dfs.cu: 16-word class 325 -> 53 ms, 8-word class 49 -> 7 ms; 70-77 % of the
// issue slots busy, shared-memory wavefronts 66-70 %.
//
// The launches of one class read their sets from lists, one per row width:
// entry i of the lists, in the order of the widths, lives in the spare word
// W + 1 of row i % rows of tile i / rows (no memory of its own), as
// owner << 10 | e1.
struct Lists {
    uint32_t* tiles;
    int64_t tile_words;
    int RS, W, rows;
    unsigned int* count;  // [16] sets of every width, filled by the tile build
    __device__ __forceinline__ uint32_t& entry(unsigned int i) const
    {
        const unsigned int o = i / (unsigned)rows;
        return tiles[(int64_t)o * tile_words + (int64_t)(i - o * (unsigned)rows) * RS + W + 1];
    }
};

// Fills the lists: a warp takes 32 rows of an owner, reads the sizes that the
// tile build left in word W, and places each set in its width's list.
__global__ void __launch_bounds__(256) k_close_list(Ctx cb, Lists L, int chunks, unsigned int* fill)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t it = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < cb.nitems * chunks; it += nw) {
        const int64_t oi = it / chunks;
        const int e = (int)(it - oi * chunks) * 32 + lane;
        Ctx c;
        int32_t r;
        if (!cc::resolve(cb, oi, c, r)) break;
        const int d = (int)(c.offp[r + 1] - c.offp[r]);
        const int size = e < d ? (int)L.tiles[oi * L.tile_words + (int64_t)e * L.RS + L.W] : 0;
        const int bin = size >= 4 ? close_bin(size) : kCloseBins;
        const uint32_t peers = __match_any_sync(kFull, bin);
        const int lead = __ffs(peers) - 1;
        unsigned int at = 0;
        if (bin < kCloseBins && lane == lead) at = atomicAdd(&fill[bin], (unsigned)__popc(peers));
        at = __shfl_sync(kFull, at, lead);
        if (bin < kCloseBins) {
            for (int b = 0; b < bin; ++b) at += L.count[b];
            L.entry(at + (unsigned)__popc(peers & mask_below(lane))) = (uint32_t)oi << 10 | (uint32_t)e;
        }
    }
}

// The sets of one width: a team takes a list entry from the cursor, lists the
// set, and closes it.  Memberships go to global memory at once (a few per
// cent of a set's work, and it leaves the shared memory to the sets).
template <int WC>
__global__ void __launch_bounds__(cta_threads(WC), ctas_per_sm(WC)) k_close(Ctx cb, Lists L, int bin, unsigned int* cursor)
{
    constexpr int NT = team_threads(WC), NW = NT / 32;
    constexpr TeamLayout l = team_layout(WC, NW);
    extern __shared__ __align__(16) char smem_close[];
    __shared__ unsigned int s_item;
    const int lane = threadIdx.x & 31, wid = NT == 32 ? 0 : (int)threadIdx.x >> 5;
    char* base = smem_close + (NT == 32 ? (int)(threadIdx.x >> 5) * l.total : 0);
    const Team t{(uint32_t*)(base + l.B), (uint16_t*)(base + l.pos), (uint16_t*)(base + l.nb), (int32_t*)(base + l.tt),
                 (int32_t*)(base + l.acc), (uint32_t*)(base + l.red), (uint32_t*)(base + l.queue)};
    const unsigned int sets = L.count[bin];
    unsigned int first = 0;
    for (int b = 0; b < bin; ++b) first += L.count[b];
    for (;;) {
        unsigned int item = 0;
        if (NT == 32) {
            if (lane == 0) item = atomicAdd(cursor, 1u);
            item = __shfl_sync(kFull, item, 0);
        } else {
            if (threadIdx.x == 0) s_item = atomicAdd(cursor, 1u);
            __syncthreads();
            item = s_item;
            __syncthreads();
        }
        if (item >= sets) break;
        const uint32_t ent = L.entry(first + item);
        const int64_t oi = ent >> 10;
        const int e1 = (int)(ent & 1023u);
        Ctx c;
        int32_t r;
        if (!cc::resolve(cb, oi, c, r)) break;
        const uint32_t* __restrict__ T = L.tiles + oi * L.tile_words;
        const int n = (int)T[e1 * L.RS + L.W];
        list_set<NT>(t, upper_word(T, L.RS, e1, L.W, lane), L.W, lane, wid);
        sync<NT>();
        unsigned long long wk = 0;
        const int32_t* mem = c.pv ? c.adjp + c.offp[r] : nullptr;
        const unsigned long long sub =
            close_set<WC, NT>(t, n, T, L.RS, lane, wid, c.work ? &wk : nullptr, [&](int j, uint32_t K) {
                if (mem) atomicAdd(&c.pv[mem[t.pos[j]]], (unsigned long long)K);
            });
        if (c.work) {
            wk = cc::warp_sum64(wk);
            if (lane == 0 && wk) atomicAdd(c.work, wk);
        }
        if (sub && lane == 0 && wid == 0) {
            add_total(c.total, sub);
            if (c.po) atomicAdd(&c.po[r], sub);
            if (mem) {
                atomicAdd(&c.pv[r], sub);
                atomicAdd(&c.pv[mem[e1]], sub);
            }
        }
    }
}

template <int WC>
kc_status launch_bin(const Ctx& c, const Lists& L, int bin, unsigned int* cursor, cudaStream_t s)
{
    constexpr int teams = cta_threads(WC) / team_threads(WC);
    const size_t smem = (size_t)team_layout(WC, team_threads(WC) / 32).total * teams;
    auto kern = k_close<WC>;
    KC_CK(cc::allow_smem(kern, smem));
    const int64_t room = (int64_t)num_sms() * cc::blocks_per_sm(kern, cta_threads(WC), smem);
    const int grid = (int)std::min<int64_t>((c.nitems * L.rows + teams - 1) / teams, room);
    kern<<<grid, cta_threads(WC), smem, s>>>(c, L, bin, cursor);
    KC_LAUNCHED();
    return KC_OK;
}

}  // namespace

// Whether the closing kernels count k in the class of W words with `items`
// owners (a list entry holds 22 bits of the owner's number).
bool close_supported(int W, int k, int64_t items) { return (W == 8 || W == 16) && k == 6 && items < (1 << 22); }

// Search pass of a split class over finished tiles (symmetric rows of RS = W
// + 4 words, the candidate-set sizes in word W and their numbers by width in
// ctr[0..15]; ctr[16..47]: zeroed).  dmax: no |Gamma+| in the class is larger.
kc_status close_launch(const Ctx& c, int W, int dmax, uint32_t* tiles, int64_t tile_words, int RS, unsigned int* ctr,
                       cudaStream_t s)
{
    const int chunks = (std::min(dmax, 32 * W) + 31) / 32;
    const Lists L{tiles, tile_words, RS, W, 32 * W, ctr};
    const int64_t warps = c.nitems * chunks;
    k_close_list<<<(int)std::min<int64_t>((warps + 7) / 8, (int64_t)num_sms() * 8), 256, 0, s>>>(c, L, chunks, ctr + 16);
    KC_LAUNCHED();
    unsigned int* cur = ctr + 32;
    KC_TRY(launch_bin<1>(c, L, 0, cur, s));
    KC_TRY(launch_bin<2>(c, L, 1, cur + 1, s));
    if (chunks > 2) KC_TRY(launch_bin<3>(c, L, 2, cur + 2, s));
    if (chunks > 3) KC_TRY(launch_bin<4>(c, L, 3, cur + 3, s));
    if (chunks > 4) KC_TRY(launch_bin<5>(c, L, 4, cur + 4, s));
    if (chunks > 5) KC_TRY(launch_bin<6>(c, L, 5, cur + 5, s));
    if (chunks > 6) KC_TRY(launch_bin<8>(c, L, 6, cur + 6, s));
    if (chunks > 8) KC_TRY(launch_bin<12>(c, L, 7, cur + 7, s));
    if (chunks > 12) KC_TRY(launch_bin<16>(c, L, 8, cur + 8, s));
    return KC_OK;
}

}  // namespace kc

// close.cuh -- candidate sets closed on a compact copy of their subgraph
// (Reduce 3, Alg. 1; Sec. 3), for the 2-, 4-, 8- and 16-word owner classes.
//
// The ordered search of dfs.cu walks the chains x_i1 < x_i2 < ... until three
// vertices are missing.  Here a candidate set C (the elements of G+(u) above
// the chain that are adjacent to all of it) that still needs three or four
// vertices is closed at once, with the number of triangles or 4-cliques of
// G[C] through every v of C: one level earlier than the ordered search.
//
//   1. Compact copy.  The elements of C are renumbered 0..c-1 and the rows of
//      G[C] squeezed to them: c rows of ceil(c/32) words instead of c rows of
//      the owner's 9..16 words (the candidate sets of a power-law graph's hub
//      cores hold a third of Gamma+(u), and every later step is a pass over
//      rows).  A lane squeezes one row, word by word, with the parallel-suffix
//      moves of "compress" (Warren, Hacker's Delight, 7-4); the moves depend on
//      C alone and are worked out once per set.
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
//      the complement edges of a pair or a triple, through v go
//        C(d,2) - M_v triangles and C(d,3) - (d-2) M_v + P_v - T_v 4-cliques.
//      P_v and t_v come from one pass over all rows a of C, the same row for
//      every thread (a broadcast load).
//   4. The sums over edges ab of B inside X_v come from a walk over the
//      triangles of B, each visited once (v < a < b) and credited to its
//      three corners: m = |X_v & X_a & X_b| sums to 3 k_v over the triangles
//      through v.  With B = G[C] this walk alone is the answer.  Triangles
//      (three vertices missing) need no pass 3: M_v = M - sum_{a in X_v}
//      (nb_a - co(v,a) / 2), a walk over the edges of B.
// All terms fit 32 bits: c <= 511, C(511,3) < 2^25, 512 C(511,2) < 2^27, and
// three times the sum of t_a over a row is below 2^28.
//
// Bound: population counts (16 lanes per SM and clock) and instruction issue.
// Step 3 needs c ceil(c/32) counts per element; adding words bitwise first
// (full adders, three-input logic) brings 5 or 8 words down to 3 or 4 counts.
//
// A team is one warp up to 256 elements (no barrier but the warp's) and four
// above; when the elements do not fill the last round of
// threads, several threads share an element and split the rows.  Edges and
// triangles of B go through queues, so that the warps stay full however
// unevenly they fall.
#pragma once

#include "count_common.cuh"

namespace kc {
namespace cl {

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
    uint32_t* moves;  // [words of the owner's rows][8] compress moves, mask, size
};

// Words a compact row takes (stride), by row width WC: vector loads need 2 or
// a multiple of 4.
__host__ __device__ constexpr int row_words(int WC) { return WC <= 2 ? WC : (WC + 3) & ~3; }

// Place of word q of row j.  Rows of 8 words have their two 128-bit halves
// swapped in every second group of four rows, so that the same half of random
// rows falls on all banks.
template <int WC>
__device__ __forceinline__ int word_at(int j, int q)
{
    constexpr int SW = row_words(WC);
    return SW == 8 ? j * 8 + (((q ^ j) & 4) | (q & 3)) : j * SW + q;
}

template <int WC>
__device__ __forceinline__ void load_row(const uint32_t* B, int j, uint32_t (&x)[WC])
{
    constexpr int SW = row_words(WC);
    const uint32_t* p = B + j * SW;
    if (SW >= 4) {
        const int flip = SW == 8 ? j & 4 : 0;
#pragma unroll
        for (int q = 0; q < WC / 4; ++q) {
            const uint4 a = *(const uint4*)(p + ((4 * q) ^ flip));
            x[4 * q] = a.x;
            x[4 * q + 1] = a.y;
            x[4 * q + 2] = a.z;
            x[4 * q + 3] = a.w;
        }
        constexpr int T = WC & ~3;
        const uint32_t* e = p + (T ^ flip);
        if ((WC & 3) == 1) x[T] = e[0];
        if ((WC & 3) >= 2) {
            const uint2 a = *(const uint2*)e;
            x[T] = a.x;
            x[WC & 2 ? T + 1 : T] = a.y;
        }
        if ((WC & 3) == 3) x[WC - 1] = e[2];
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

// The edges v < a of B, 32 at a time: body(k, e, final) with edge e = v | a <<
// 10 in lanes below k; the last call has final set (k may be 0 there).  Every
// warp of the team takes the elements v of its rounds (or its share of their
// bits).  At most 31 entries wait and 32 kPush join them, so the queue never
// overflows.
template <int WC, int NT, typename Body>
__device__ __forceinline__ void for_edges(const Team& t, int c, int wc, int lane, int wid, Body body)
{
    uint32_t* eq = t.queue + 2 * wid * kQueue;
    const int tid = wid * 32 + lane;
    uint32_t n = 0, bits[1] = {0u}, every = 0u;
    int en = 0;                     // waiting edges
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
            bits[0] = (v < c && q >= (v >> 5)) ? t.B[word_at<WC>(v, q)] & every & (q == (v >> 5) ? mask_above(v & 31) : kFull) : 0u;
            n = (uint32_t)__popc(bits[0]);
        }
        const bool last = base >= c;
        if (!last) en = push_bits<1>(eq, en, bits, n, (uint32_t)v, 10, q * 32, lane);
        bool once = last;
#pragma unroll 1
        while (once || en >= 32) {
            const int k = min(en, 32);
            en -= k;
            body(k, lane < k ? eq[en + lane] : 0u, last && en == 0);
            once = last && en > 0;
        }
        if (last) break;
    }
}

// Step 4, four vertices missing: the edges find their common elements b > a
// and queue the triangles; 32 triangles at a time are credited.  Returns the
// lane's triangles.
template <int WC, int NT>
__device__ __forceinline__ uint32_t walk4(const Team& t, bool dense, int c, int wc, int lane, int wid)
{
    uint32_t* tq = t.queue + (2 * wid + 1) * kQueue;
    uint32_t ntri = 0;
    int tn = 0;
    for_edges<WC, NT>(t, c, wc, lane, wid, [&](int k, uint32_t e, bool final) {
        uint32_t Y[WC], ny = 0;
#pragma unroll
        for (int w = 0; w < WC; ++w) Y[w] = 0u;
        if (lane < k) {
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
            const int keep = final && !more ? 0 : 31;
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
    });
    return ntri;
}

// Step 4, three vertices missing: acc of both ends of an edge va gets twice
// its share of M_v's sum (dense), or co(v,a).
template <int WC, int NT>
__device__ __forceinline__ uint32_t walk3(const Team& t, bool dense, int c, int wc, int lane, int wid)
{
    uint32_t nedge = 0;
    for_edges<WC, NT>(t, c, wc, lane, wid, [&](int k, uint32_t e, bool) {
        if (lane < k) {
            const int u = (int)(e & 1023u), a = (int)(e >> 10);
            uint32_t X[WC], Xa[WC];
            load_row<WC>(t.B, u, X);
            load_row<WC>(t.B, a, Xa);
            const int co = (int)co_count<WC>(X, Xa);
            atomicAdd(&t.acc[u], dense ? 2 * (int)t.nb[a] - co : co);
            atomicAdd(&t.acc[a], dense ? 2 * (int)t.nb[u] - co : co);
            ++nedge;
        }
        __syncwarp();
    });
    return nedge;
}

// Lists the elements of the word set held by a warp's lanes (lane w: word w,
// zero from Wd on) into t.pos, the warps of the team sharing the words, and
// the moves that compress a row to them (more than one word: WC).  The caller
// synchronises the team.
template <int WC, int NT>
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
    if (WC > 1 && wid == 0 && lane < ((Wd + 3) & ~3)) {
        uint32_t m = u, mk = ~m << 1, mv[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            uint32_t mp = mk ^ (mk << 1);
            mp ^= mp << 2;
            mp ^= mp << 4;
            mp ^= mp << 8;
            mp ^= mp << 16;
            mv[i] = mp & m;
            m = (m ^ mv[i]) | (mv[i] >> (1 << i));
            mk &= ~mp;
        }
        uint4* o = (uint4*)(t.moves + 8 * lane);
        o[0] = make_uint4(u, mv[0], mv[1], mv[2]);
        o[1] = make_uint4(mv[3], mv[4], (uint32_t)pc, 0u);
    }
}

// The NEED-cliques (3 or 4) of G[C] through every element of C, by a team of
// NT threads: credit(j, K) is called once per element j with a non-zero K.
// list_set has prepared C (c >= NEED elements, visible to the team); T: its
// owner's symmetric rows (Wd words in use, stride RS a multiple of 4 words,
// 16-byte aligned).  Returns the number of NEED-cliques (every thread); ends
// with the team's barrier.
template <int WC, int NEED, int NT, typename Credit>
__device__ __forceinline__ unsigned long long close_set(const Team& t, int c, const uint32_t* __restrict__ T, int RS,
                                                        int Wd, int lane, int wid, unsigned long long* wk, Credit credit)
{
    constexpr int NW = NT / 32;
    static_assert(WC <= 16 && (NEED == 3 || NEED == 4), "32-bit sums hold up to 511 elements");
    const int wc = (c + 31) >> 5;
    const int tid = wid * 32 + lane;
    // 1. rows, and their degrees
    uint32_t loc = 0;
    if (WC == 1) {
        // one word: a ballot gives a whole row, four rows at a time
        const int p = lane < c ? (int)t.pos[lane] : 0;
        const uint32_t* Tp = T + (p >> 5);
        const uint32_t bit = lane < c ? 1u << (p & 31) : 0u;
        uint32_t mine = 0;
#pragma unroll 1
        for (int i0 = 0; i0 < c; i0 += 4) {
            const uint2 pp = *(const uint2*)(t.pos + i0);  // rows past c - 1 read as row 0
            const int p0 = (int)(pp.x & 0xffffu), p1 = i0 + 1 < c ? (int)(pp.x >> 16) : 0;
            const int p2 = i0 + 2 < c ? (int)(pp.y & 0xffffu) : 0, p3 = i0 + 3 < c ? (int)(pp.y >> 16) : 0;
            const uint32_t v0 = Tp[p0 * RS], v1 = Tp[p1 * RS], v2 = Tp[p2 * RS], v3 = Tp[p3 * RS];
            const uint32_t b0 = __ballot_sync(kFull, v0 & bit), b1 = __ballot_sync(kFull, v1 & bit);
            const uint32_t b2 = __ballot_sync(kFull, v2 & bit), b3 = __ballot_sync(kFull, v3 & bit);
            if ((lane ^ i0) < 4) mine = lane & 2 ? (lane & 1 ? b3 : b2) : (lane & 1 ? b1 : b0);
        }
        if (lane < c) {
            t.B[lane] = mine;
            const uint32_t nbv = (uint32_t)(c - 1 - __popc(mine));
            t.nb[lane] = (uint16_t)nbv;
            t.acc[lane] = 0;
            loc = nbv;
        }
    } else {
#pragma unroll 1
        for (int v0 = wid * 32; v0 < c; v0 += NT) {
            const int v = v0 + lane;
            const bool on = v < c;
            const uint32_t* row = T + (int)t.pos[on ? v : 0] * RS;
            uint32_t cur = 0, dg = 0;
            int off = 0, k = 0;
#pragma unroll 1
            for (int w4 = 0; w4 < Wd; w4 += 4) {
                const uint4 r4 = *(const uint4*)(row + w4);
                const uint32_t r[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 ma = ((const uint4*)(t.moves + 8 * (w4 + i)))[0], mb = ((const uint4*)(t.moves + 8 * (w4 + i)))[1];
                    if (mb.z == 0u) continue;
                    uint32_t x = r[i] & ma.x, z;
                    dg += (uint32_t)__popc(x);
                    z = x & ma.y;
                    x = (x ^ z) | (z >> 1);
                    z = x & ma.z;
                    x = (x ^ z) | (z >> 2);
                    z = x & ma.w;
                    x = (x ^ z) | (z >> 4);
                    z = x & mb.x;
                    x = (x ^ z) | (z >> 8);
                    z = x & mb.y;
                    x = (x ^ z) | (z >> 16);
                    cur |= x << off;
                    const int end = off + (int)mb.z;
                    if (end >= 32) {
                        if (on) t.B[word_at<WC>(v, k)] = cur;
                        ++k;
                        cur = off ? x >> (32 - off) : 0u;
                    }
                    off = end & 31;
                }
            }
            if (on) {
                if (off) t.B[word_at<WC>(v, k++)] = cur;
#pragma unroll 1
                for (; k < WC; ++k) t.B[word_at<WC>(v, k)] = 0u;
                const uint32_t nbv = (uint32_t)(c - 1) - dg;
                t.nb[v] = (uint16_t)nbv;
                t.acc[v] = 0;
                loc += nbv;
            }
        }
    }
    // 2. flip to the complement when it is the sparser side
    const uint32_t nbsum = team_sum<NT>(loc, t.red, lane, wid);
    const bool dense = 2u * nbsum <= (uint32_t)c * (uint32_t)(c - 1);
    const int M = (int)(nbsum >> 1);
    int Tall = 0;
    if (dense) {
#pragma unroll 1
        for (int v = tid; v < c; v += NT) {
#pragma unroll
            for (int w = 0; w < WC; ++w) {
                const int left = c - 32 * w;
                uint32_t m = left >= 32 ? kFull : (left > 0 ? mask_below(left) : 0u);
                if (w == (v >> 5)) m &= ~(1u << (v & 31));
                uint32_t& x = t.B[word_at<WC>(v, w)];
                x = ~x & m;
            }
        }
        sync<NT>();
    }
    if (NEED == 4 && dense) {
        // 3. one pass over all rows a: co(v,a) against every v
        uint32_t tl = 0;
#pragma unroll 1
        for (int base = 0; base < c;) {
            const int lg = share_log<NT>(c, base), S = 1 << lg;
            const int sub = tid & (S - 1), v = base + (tid >> lg);
            const bool on = v < c;
            uint32_t X[WC];
            load_row<WC>(t.B, on ? v : 0, X);
            uint32_t t2 = 0, s1 = 0, P2 = 0;
#pragma unroll 1
            for (int q = 0; q < wc; ++q) {
                uint32_t xw = t.B[word_at<WC>(on ? v : 0, q)] >> sub;
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
                const int Mv = M - (int)s1 + tv;
                t.tt[v] = tv;
                t.acc[v] = -3 * (d * (d - 1) * (d - 2) / 6 - Mv * (d - 2) + (int)(P2 >> 1));
                tl += (uint32_t)tv;
            }
            base += NT >> lg;
        }
        Tall = (int)(team_sum<NT>(tl, t.red + 8, lane, wid) / 3u);
    }
    const uint32_t steps = NEED == 4 ? walk4<WC, NT>(t, dense, c, wc, lane, wid) : walk3<WC, NT>(t, dense, c, wc, lane, wid);
    sync<NT>();
    unsigned long long sum = 0;
#pragma unroll 1
    for (int v = tid; v < c; v += NT) {
        int K = t.acc[v] / (NEED == 4 ? 3 : 2);
        if (dense) {
            const int d = c - 1 - (int)t.nb[v];
            K = NEED == 4 ? -Tall - K : d * (d - 1) / 2 - M + K;
        }
        sum += (unsigned long long)K;
        if (K) credit(v, (uint32_t)K);
    }
    if (wk) {
        // the edges of B, met once each by walk4 to find their triangles
        if (NEED == 4 && tid == 0) *wk += (unsigned long long)(dense ? M : c * (c - 1) / 2 - M) * WC;
        *wk += (unsigned long long)steps * (unsigned)(WC * (NEED == 4 ? (dense ? 4 : 2) : 1));
#pragma unroll 1
        for (int v = tid; v < c; v += NT) *wk += (unsigned long long)(Wd + (NEED == 4 && dense ? c * WC : 0));
    }
    // an element's cliques are below 2^25, their sum below 2^34
    sum = cc::warp_sum64(sum);
    if (NT == 32) {
        __syncwarp();
        return sum / (unsigned)NEED;
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
    return all / (unsigned)NEED;
}

// Row e above e, one word per lane (lane w: word w).
__device__ __forceinline__ uint32_t upper_word(const uint32_t* __restrict__ T, int RS, int e, int Wd, int lane)
{
    const int we = e >> 5;
    uint32_t v = (lane >= we && lane < Wd) ? T[e * RS + lane] : 0u;
    if (lane == we) v &= mask_above(e & 31);
    return v;
}

struct TeamLayout {
    int B, pos, nb, tt, acc, red, queue, moves, total;  // byte offsets
};

// Working set of a team of NW warps for rows of WC words out of owners' rows
// of W words.
__host__ __device__ constexpr TeamLayout team_layout(int WC, int W, int NW)
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
    l.moves = l.queue + NW * 2 * kQueue * 4;
    l.total = l.moves + ((W + 3) & ~3) * 32;
    return l;
}

__device__ __forceinline__ Team team_at(char* base, const TeamLayout& l)
{
    return Team{(uint32_t*)(base + l.B), (uint16_t*)(base + l.pos), (uint16_t*)(base + l.nb), (int32_t*)(base + l.tt),
                (int32_t*)(base + l.acc), (uint32_t*)(base + l.red), (uint32_t*)(base + l.queue), (uint32_t*)(base + l.moves)};
}

}  // namespace cl
}  // namespace kc

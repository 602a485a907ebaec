// quad.cu -- k = 4 for owners of more than 64 elements (rows of 4..32 words),
// and k = 5 in the 4-word class.
//
// k = 5: q_{u,4} is the number of 4-cliques of G+(u); each edge v < a counts the
// edges inside C = row v & row a, one row load for each b of C.  Totals only.
// (Lists of the search's few elements per set cost more than these loops while
// rows are 128 bits; 8 words stay with the search, 16 words close sets, close.cu.)
// Chung-Lu n = 1e6, total: 1.43 -> 1.30 ms.
//
// k = 4:
// q_{u,3} is the number of triangles of G+(u).  One CTA per owner builds the
// bitmap rows in shared memory and walks the edges of G+(u), v < a, once: with
// co = popc(row v & row a) over upper rows (no memberships) their sum is the
// count; over whole rows (memberships) co is the number of triangles on the
// edge, and the sum at each end is twice the triangles through it.
//
// Four lanes hold a row v in registers and take its words in turn; each edge
// costs one row load and one AND and count per word.  Bound: instruction
// issue and shared-memory loads, about 40 instructions for 32 edges of a 16-word
// row.  The general search (dfs.cu) spent 130 there: it listed each candidate
// set's elements by rank before it read their rows.  Chung-Lu n = 1e6, m = 2e7,
// with memberships, builds included: 16 words 1.36 -> 0.94 ms, 8 words 1.15 ->
// 0.63 ms, 4 words 1.14 -> 0.48 ms.
#include <algorithm>

#include "close.cuh"

namespace kc {

int num_sms();

namespace {

using cc::add_total;
using cc::Ctx;
using cc::mask_above;

constexpr int kSpanWords = 1024;

struct QLayout {
    int L, col, acc, A, bits, pre, total;  // 32-bit words
};

// D: elements at most; rows of WM words, stride WM + 4 (128-bit loads, and
// consecutive rows on different banks).
__host__ __device__ inline QLayout quad_layout(int D, int WM, bool pv, bool col)
{
    QLayout l;
    l.L = 0;
    l.col = l.L + D;
    l.acc = l.col + (col ? D : 0);
    l.A = l.acc + (pv ? D : 0);
    l.bits = l.A + D * (WM + 4);
    l.pre = l.bits + kSpanWords;
    l.total = l.pre + kSpanWords / 2;
    return l;
}

template <bool PV, bool COL, int WM, int K>  // K = 5: !PV, WM = 4
__global__ void __launch_bounds__(WM <= 4 ? 128 : 256, WM <= 4 ? 8 : (WM <= 16 ? 4 : 1)) k_quad(Ctx cb, int D)
{
    extern __shared__ __align__(16) uint32_t smem[];
    constexpr int RS = WM + 4;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, NW = blockDim.x >> 5;
    const QLayout lay = quad_layout(D, WM, PV, COL);
    int32_t* sL = (int32_t*)(smem + lay.L);
    uint32_t* sCol = smem + lay.col;
    uint32_t* acc = smem + lay.acc;
    uint32_t* sA = smem + lay.A;
    __shared__ unsigned int s_next;
    __shared__ unsigned long long s_tot, s_wk;
    __shared__ long long s_item;
    for (;;) {
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(cb.cursor, 1ull);
        __syncthreads();
        cc::OwnerCtx c;
        int32_t r;
        if (!cc::resolve(cb, (int64_t)s_item, c, r)) break;
        const int64_t b = c.offp[r];
        const int d = (int)(c.offp[r + 1] - b);
        const int Wd = (d + 31) >> 5, nq = (Wd + 3) >> 2;
        const int32_t ur = COL ? c.perm[r] : 0;
        for (int j = threadIdx.x; j < d; j += blockDim.x) {
            const int32_t x = c.adjp[b + j];
            sL[j] = x;
            if (COL) sCol[j] = cc::sample_label(c, ur, c.perm[x]);
            if (PV) acc[j] = 0u;
        }
        for (int j = threadIdx.x; j < d * RS / 4; j += blockDim.x) ((uint4*)sA)[j] = make_uint4(0u, 0u, 0u, 0u);
        if (threadIdx.x == 0) {
            s_next = 0u;
            s_tot = 0ull;
            s_wk = 0ull;
        }
        __syncthreads();
        if (COL) cc::class_flags_smem<true>(c, sCol, d, K - 1, threadIdx.x, blockDim.x);
        cc::SpanTable T{smem + lay.bits, (uint16_t*)(smem + lay.pre), 0, 0};
        if (sL[0] < c.core_lo) cc::span_table_build(T, sL, d, kSpanWords);  // (lists are read)
        cc::build_rows<PV, COL>(c, sL, sCol, d, sA, RS, wid, NW, lane, ur, &T);
        __syncthreads();

        unsigned long long tot = 0, wk = 0;
        for (;;) {
            unsigned int t = 0;
            if (lane == 0) t = atomicAdd(&s_next, 8u);
            const int v = (int)__shfl_sync(kFull, t, 0) + (lane >> 2);
            if (v - (lane >> 2) >= d) break;
            uint32_t sum = 0;
            if (v < d) {
                uint32_t X[WM];
#pragma unroll
                for (int q = 0; q < WM / 4; ++q) {
                    const uint4 x = q < nq ? ((const uint4*)(sA + v * RS))[q] : make_uint4(0u, 0u, 0u, 0u);
                    X[4 * q] = x.x;
                    X[4 * q + 1] = x.y;
                    X[4 * q + 2] = x.z;
                    X[4 * q + 3] = x.w;
                }
                const int vw = v >> 5;
                for (int w = vw + ((lane - vw) & 3); w < Wd; w += 4) {
                    uint32_t bits = sA[v * RS + w];
                    if (w == vw) bits &= mask_above(v & 31);
                    while (bits) {
                        const int a = w * 32 + __ffs(bits) - 1;
                        bits &= bits - 1u;
                        const uint4* Ra = (const uint4*)(sA + a * RS);
                        uint32_t co = 0;
                        if (K == 4) {
#pragma unroll
                            for (int q = 0; q < WM / 4; ++q) {
                                if (q >= nq) continue;
                                const uint4 x = Ra[q];
                                const uint32_t z[4] = {X[4 * q] & x.x, X[4 * q + 1] & x.y, X[4 * q + 2] & x.z,
                                                       X[4 * q + 3] & x.w};
                                co += cl::popc_words<4>(z);
                            }
                        } else {  // WM == 4
                            const uint4 x = Ra[0];
                            const uint32_t C[4] = {X[0] & x.x, X[1] & x.y, X[2] & x.z, X[3] & x.w};
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                uint32_t left = C[q];
#pragma unroll 1
                                while (left) {
                                    const int e = q * 32 + __ffs(left) - 1;
                                    left &= left - 1u;
                                    const uint4 y = *(const uint4*)(sA + e * RS);
                                    const uint32_t z[4] = {C[0] & y.x, C[1] & y.y, C[2] & y.z, C[3] & y.w};
                                    co += cl::popc_words<4>(z);
                                    if (c.work) wk += 4u;
                                }
                            }
                        }
                        sum += co;
                        if (PV && co) atomicAdd(&acc[a], co);
                        if (c.work) wk += (unsigned)(4 * nq);
                    }
                }
                if (PV && sum) atomicAdd(&acc[v], sum);
            }
            tot += sum;
        }
        tot = cc::warp_sum64(tot);
        if (lane == 0 && tot) atomicAdd(&s_tot, tot);
        if (c.work) {
            wk = cc::warp_sum64(wk);
            if (lane == 0 && wk) atomicAdd(&s_wk, wk);
        }
        __syncthreads();
        // whole rows: every triangle was met on its three edges, a vertex has two of them
        const unsigned long long q = PV ? s_tot / 3ull : s_tot;
        if (threadIdx.x == 0) {
            add_total(c.total, q);
            if (c.po) c.po[r] = q;
            if (PV && q) atomicAdd(&c.pv[r], q);
            if (c.work && s_wk) atomicAdd(c.work, s_wk);
        }
        if (PV)
            for (int j = threadIdx.x; j < d; j += blockDim.x)
                if (acc[j]) atomicAdd(&c.pv[sL[j]], (unsigned long long)(acc[j] / 2u));
        __syncthreads();
    }
}

template <bool PV, bool COL, int WM, int K>
kc_status go(const Ctx& c, int D, cudaStream_t s)
{
    auto kern = k_quad<PV, COL, WM, K>;
    const size_t smem = (size_t)quad_layout(D, WM, PV, COL).total * 4;
    const int threads = WM <= 4 ? 128 : 256;
    KC_CK(cc::allow_smem(kern, smem));
    const int grid = (int)std::min<int64_t>(c.nitems, (int64_t)num_sms() * cc::blocks_per_sm(kern, threads, smem));
    kern<<<grid, threads, smem, s>>>(c, D);
    KC_LAUNCHED();
    return KC_OK;
}

template <bool PV, bool COL>
kc_status by_width(const Ctx& c, int W, int D, cudaStream_t s)
{
    if constexpr (!PV)
        if (c.k == 5) return go<PV, COL, 4, 5>(c, D, s);
    switch (W) {
    case 4: return go<PV, COL, 4, 4>(c, D, s);
    case 8: return go<PV, COL, 8, 4>(c, D, s);
    case 16: return go<PV, COL, 16, 4>(c, D, s);
    case 32: return go<PV, COL, 32, 4>(c, D, s);
    }
    return KC_ENOTSUP;
}

}  // namespace

// The class of W = 4, 8, 16 or 32 words at k = 4, of 4 words at k = 5 without
// memberships; dmax: no |Gamma+| is larger.
kc_status quad_launch(const Ctx& c, int W, int dmax, bool pv, bool col, cudaStream_t s)
{
    const int D = 32 * ((std::min(dmax, 32 * W) + 31) / 32);
    if (pv) return col ? KC_ENOTSUP : by_width<true, false>(c, W, D, s);
    return col ? by_width<false, true>(c, W, D, s) : by_width<false, false>(c, W, D, s);
}

}  // namespace kc

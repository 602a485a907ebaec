// close.cu -- the counting kernels of the 4-, 8- and 16-word owner classes
// that close candidate sets on compact copies (close.cuh); the 2-word class
// closes its own in dfs.cu.
//
// 8 and 16 words (split classes): the owners' rows are in global tiles
// (k_tile_build), the sets of all owners are listed by the row width of their
// copies, and one launch per width closes them -- a launch runs one short
// body (all widths in one kernel were 300 KB of code and waited for
// instructions more than for anything else), has shared memory for its own
// sets only, and balances single sets instead of owners.
// 4 words: an owner per CTA, rows in shared memory, a set per warp.
// Chung-Lu n = 1e6, m = 2e7, against the pair search of dfs.cu, tiles included:
// k = 6 with memberships, 16-word class 325 -> 43 ms, 8-word 49 -> 6.7 ms,
// 4-word 17.4 -> 2.5 ms (issue slots 60-75 % busy); k = 5 total, 16-word class
// 11.9 -> 8.0 ms; colour estimate (c = 8, k = 6), 16-word
// class 9.0 -> 2.1 ms, 8-word 3.3 -> 1.4 ms.
// Tried and not kept: the counts |X_v & X_a| over all a kept as binary digits
// (bitwise row additions along X_v) instead of c intersections: widths 5, 6, 8
// 3-9 % faster, widths 3 and 4 3-7 % slower, the whole k = 6 count 54.3 -> 52.8 ms.
#include <algorithm>

#include "close.cuh"

namespace kc {

int num_sms();

namespace {

using namespace cl;
using cc::add_total;
using cc::close_bin;
using cc::Ctx;
using cc::kCloseBins;

constexpr int team_threads(int WC) { return WC <= 8 ? 32 : 128; }
constexpr int cta_threads(int WC) { return WC <= 4 ? 128 : (WC <= 8 ? 64 : 128); }
constexpr int ctas_per_sm(int WC) { return WC <= 1 ? 8 : (WC <= 4 ? 6 : (WC <= 8 ? 10 : 3)); }

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
        cc::OwnerCtx c;
        int32_t r;
        if (!cc::resolve(cb, oi, c, r)) break;
        const int d = (int)(c.offp[r + 1] - c.offp[r]);
        const int size = e < d ? (int)L.tiles[oi * L.tile_words + (int64_t)e * L.RS + L.W] : 0;
        const int bin = size >= cb.k - 2 ? close_bin(size) : kCloseBins;
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

// Sets a team takes per cursor step at most (1 for teams of several warps).
constexpr int sets_taken(int WC) { return WC == 1 ? 8 : (WC == 2 ? 4 : 1); }

// The sets of one width: a team takes list entries from the cursor (several
// where a set is so small that the chain of loads that leads to it would
// outlast it: a lane each fetches their owners, offsets and sizes), lists
// each set, and closes it.  Memberships go to global memory at once (a few per
// cent of a set's work, and it leaves the shared memory to the sets).
template <int WC, int NEED>
__global__ void __launch_bounds__(cta_threads(WC), ctas_per_sm(WC)) k_close(Ctx cb, Lists L, int bin, int take, unsigned int* cursor)
{
    constexpr int NT = team_threads(WC), NW = NT / 32;
    constexpr TeamLayout l = team_layout(WC, 16, NW);
    extern __shared__ __align__(16) char smem_close[];
    __shared__ unsigned int s_item;
    const int lane = threadIdx.x & 31, wid = NT == 32 ? 0 : (int)threadIdx.x >> 5;
    const Team t = team_at(smem_close + (NT == 32 ? (int)(threadIdx.x >> 5) * l.total : 0), l);
    const unsigned int sets = L.count[bin];
    unsigned int first = 0;
    for (int b = 0; b < bin; ++b) first += L.count[b];
    // one total for all teams: a team adds its own up and sends it once (one
    // addition per set had 1e6 sets wait 3 ns each at that one address)
    unsigned long long tot = 0;
    unsigned long long* total = cb.total;
    for (;;) {
        unsigned int item = 0;
        if (NT == 32) {
            if (lane == 0) item = atomicAdd(cursor, (unsigned)take);
            item = __shfl_sync(kFull, item, 0);
        } else {
            if (threadIdx.x == 0) s_item = atomicAdd(cursor, 1u);
            __syncthreads();
            item = s_item;
            __syncthreads();
        }
        if (item >= sets) break;
        const int have = (int)min((unsigned)take, sets - item);
        uint32_t ent = 0;
        int64_t at = 0;
        int deg = 0, size = 0;
        if (lane < have) {
            ent = L.entry(first + item + (unsigned)lane);
            cc::OwnerCtx cl;
            int32_t own;
            cc::resolve(cb, ent >> 10, cl, own);
            at = cl.offp[own];
            deg = (int)(cl.offp[own + 1] - at);
            size = (int)L.tiles[(int64_t)(ent >> 10) * L.tile_words + (int64_t)(ent & 1023u) * L.RS + L.W];
        }
#pragma unroll 1
        for (int i = 0; i < have; ++i) {
            const uint32_t e = __shfl_sync(kFull, ent, i);
            const int64_t b = __shfl_sync(kFull, at, i);
            const int Wd = (__shfl_sync(kFull, deg, i) + 31) >> 5, n = __shfl_sync(kFull, size, i), e1 = (int)(e & 1023u);
            cc::OwnerCtx c;
            int32_t r;
            cc::resolve(cb, e >> 10, c, r);  // (always an item)
            const uint32_t* __restrict__ T = L.tiles + (int64_t)(e >> 10) * L.tile_words;
            list_set<WC, NT>(t, upper_word(T, L.RS, e1, Wd, lane), Wd, lane, wid);
            sync<NT>();
            unsigned long long wk = 0;
            const int32_t* mem = c.pv ? c.adjp + b : nullptr;
            const unsigned long long sub =
                close_set<WC, NEED, NT>(t, n, T, L.RS, Wd, lane, wid, c.work ? &wk : nullptr, [&](int j, uint32_t K) {
                    if (mem) atomicAdd(&c.pv[mem[t.pos[j]]], (unsigned long long)K);
                });
            if (c.work) {
                wk = cc::warp_sum64(wk);
                if (lane == 0 && wk) atomicAdd(c.work, wk);
            }
            if (c.total != total) {  // another graph of a batch
                if (lane == 0 && wid == 0) add_total(total, tot);
                total = c.total;
                tot = 0;
            }
            tot += sub;
            if (sub && lane == 0 && wid == 0) {
                if (c.po) atomicAdd(&c.po[r], sub);
                if (mem) {
                    atomicAdd(&c.pv[r], sub);
                    atomicAdd(&c.pv[mem[e1]], sub);
                }
            }
        }
    }
    if (lane == 0 && wid == 0) add_total(total, tot);
}

template <int WC, int NEED>
kc_status launch_bin(const Ctx& c, const Lists& L, int bin, unsigned int* cursor, cudaStream_t s)
{
    constexpr int teams = cta_threads(WC) / team_threads(WC);
    const size_t smem = (size_t)team_layout(WC, 16, team_threads(WC) / 32).total * teams;
    auto kern = k_close<WC, NEED>;
    KC_CK(cc::allow_smem(kern, smem));
    const int64_t room = (int64_t)num_sms() * cc::blocks_per_sm(kern, cta_threads(WC), smem);
    // sets per cursor step: one for classes too small to give every team several
    const int grid = (int)std::min<int64_t>((c.nitems * L.rows + teams - 1) / teams, room);
    const int take = c.nitems * L.rows > 64 * room * teams ? sets_taken(WC) : 1;
    kern<<<grid, cta_threads(WC), smem, s>>>(c, L, bin, take, cursor);
    KC_LAUNCHED();
    return KC_OK;
}

constexpr int kOwnWarps = 4;
constexpr int kOwnRS = 8;  // row stride of the 4-word rows in shared memory
constexpr int kSpanWords = 1024;

struct OwnLayout {
    int A, L, col, lo, hi, total;  // byte offsets; the teams (and, while the rows are built, the span table) come first
};

__host__ __device__ constexpr OwnLayout own_layout()
{
    OwnLayout o{};
    o.A = kOwnWarps * team_layout(4, 4, 1).total;
    o.L = o.A + 128 * kOwnRS * 4;
    o.col = o.L + 128 * 4;
    o.lo = o.col + 128 * 4;
    o.hi = o.lo + 128 * 4;
    o.total = o.hi + 128 * 4;
    return o;
}

// The 4-word class: an owner per CTA of four warps, rows and memberships in
// shared memory; the warps take first-level vertices from a shared list and
// close their candidate sets (nearly all of at most 32 elements).  The list
// holds the vertices whose set is large enough: met one by one, empty sets took
// as long as the rows' build (random graph n = 5e5, m = 3e7: whole count 9.5 ->
// 8.3 ms).
template <bool COL>
__global__ void __launch_bounds__(kOwnWarps * 32, 8) k_close_own(Ctx cb)
{
    constexpr int NEED = 4;
    extern __shared__ __align__(16) char smem_close[];
    constexpr TeamLayout l = team_layout(4, 4, 1);
    constexpr OwnLayout o = own_layout();
    static_assert(kOwnWarps * l.total >= kSpanWords * 6, "the span table fits in the teams' place");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const Team t = team_at(smem_close + wid * l.total, l);
    uint32_t* sA = (uint32_t*)(smem_close + o.A);
    int32_t* sL = (int32_t*)(smem_close + o.L);
    uint32_t* sCol = (uint32_t*)(smem_close + o.col);
    uint32_t* lo = (uint32_t*)(smem_close + o.lo);
    uint32_t* hi = (uint32_t*)(smem_close + o.hi);
    __shared__ unsigned int s_next, s_sets;
    __shared__ uint8_t s_list[kOwnWarps * 32];
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
        const int Wd = (d + 31) >> 5;
        const int32_t ur = COL ? c.perm[r] : 0;
        for (int j = threadIdx.x; j < d; j += blockDim.x) {
            const int32_t x = c.adjp[b + j];
            sL[j] = x;
            if (COL) sCol[j] = cc::sample_label(c, ur, c.perm[x]);
            lo[j] = hi[j] = 0u;
        }
        for (int j = threadIdx.x; j < d * kOwnRS; j += blockDim.x) sA[j] = 0u;
        if (threadIdx.x == 0) {
            s_next = s_sets = 0u;
            s_tot = 0ull;
            s_wk = 0ull;
        }
        __syncthreads();
        if (COL) cc::class_flags_smem<true>(c, sCol, d, cb.k - 1, threadIdx.x, blockDim.x);
        cc::SpanTable S{(uint32_t*)smem_close, (uint16_t*)(smem_close + 4 * kSpanWords), 0, 0};
        cc::span_table_build(S, sL, d, kSpanWords);
        cc::build_rows<true, COL>(c, sL, sCol, d, sA, kOwnRS, wid, kOwnWarps, lane, ur, &S);
        __syncthreads();
        {  // one element per thread (d <= 128)
            const int e = threadIdx.x;
            int n = 0;
            if (e < d) {
                const uint4 x = *(const uint4*)(sA + e * kOwnRS);
                const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) n += __popc(q < wid ? 0u : (q == wid ? w[q] & mask_above(lane) : w[q]));
            }
            const uint32_t some = __ballot_sync(kFull, n >= NEED);
            unsigned int at = 0;
            if (lane == 0 && some) at = atomicAdd(&s_sets, (unsigned)__popc(some));
            at = __shfl_sync(kFull, at, 0);
            if (n >= NEED) s_list[at + __popc(some & mask_below(lane))] = (uint8_t)e;
        }
        __syncthreads();
        auto add = [&](int e, unsigned long long v) {
            const uint32_t v0 = (uint32_t)v, v1 = (uint32_t)(v >> 32);
            if (v0) {
                const uint32_t old = atomicAdd(&lo[e], v0);
                if (old + v0 < old) atomicAdd(&hi[e], 1u);
            }
            if (v1) atomicAdd(&hi[e], v1);
        };
        unsigned long long tot = 0, wk = 0;
        unsigned long long* wkp = c.work ? &wk : nullptr;
        for (;;) {
            unsigned int i = 0;
            if (lane == 0) i = atomicAdd(&s_next, 1u);
            i = __shfl_sync(kFull, i, 0);
            if (i >= s_sets) break;
            const int e1 = s_list[i];
            const uint32_t u = upper_word(sA, kOwnRS, e1, Wd, lane);
            const int n = (int)__reduce_add_sync(kFull, (unsigned)__popc(u));  // at least NEED
            if (n <= 32) list_set<1, 32>(t, u, Wd, lane, 0);
            else list_set<4, 32>(t, u, Wd, lane, 0);
            __syncwarp();
            auto credit = [&](int j, uint32_t K) { add((int)t.pos[j], K); };
            const unsigned long long sub = n <= 32 ? close_set<1, NEED, 32>(t, n, sA, kOwnRS, Wd, lane, 0, wkp, credit)
                                                   : close_set<4, NEED, 32>(t, n, sA, kOwnRS, Wd, lane, 0, wkp, credit);
            tot += sub;
            if (sub && lane == 0) add(e1, sub);
        }
        if (wkp) wk = cc::warp_sum64(wk);
        if (lane == 0 && tot) atomicAdd(&s_tot, tot);
        if (lane == 0 && wk) atomicAdd(&s_wk, wk);
        __syncthreads();
        if (threadIdx.x == 0) {
            add_total(c.total, s_tot);
            if (c.po && s_tot) c.po[r] = s_tot;
            if (c.pv && s_tot) atomicAdd(&c.pv[r], s_tot);
            if (c.work && s_wk) atomicAdd(c.work, s_wk);
        }
        if (c.pv)
            for (int j = threadIdx.x; j < d; j += blockDim.x) {
                const unsigned long long v = ((unsigned long long)hi[j] << 32) | lo[j];
                if (v) atomicAdd(&c.pv[sL[j]], v);
            }
        __syncthreads();
    }
}

// One launch per width that a set of a class with `chunks` words a row can have.
template <int NEED>
kc_status launch_bins(const Ctx& c, const Lists& L, int chunks, unsigned int* cur, cudaStream_t s)
{
    KC_TRY((launch_bin<1, NEED>(c, L, 0, cur, s)));
    KC_TRY((launch_bin<2, NEED>(c, L, 1, cur + 1, s)));
    if (chunks > 2) KC_TRY((launch_bin<3, NEED>(c, L, 2, cur + 2, s)));
    if (chunks > 3) KC_TRY((launch_bin<4, NEED>(c, L, 3, cur + 3, s)));
    if (chunks > 4) KC_TRY((launch_bin<5, NEED>(c, L, 4, cur + 4, s)));
    if (chunks > 5) KC_TRY((launch_bin<6, NEED>(c, L, 5, cur + 5, s)));
    if (chunks > 6) KC_TRY((launch_bin<8, NEED>(c, L, 6, cur + 6, s)));
    if (chunks > 8) KC_TRY((launch_bin<12, NEED>(c, L, 7, cur + 7, s)));
    if (chunks > 12) KC_TRY((launch_bin<16, NEED>(c, L, 8, cur + 8, s)));
    return KC_OK;
}

}  // namespace

// Whether the closing kernels count k in the class of W words with `items`
// owners (a list entry holds 22 bits of the owner's number).  k = 5 and 6: the
// sets of the first level need three or four vertices there; k >= 7 would need
// five.  k = 5 at 8 words stays with the search, whose sets are small there: whole
// counts on Chung-Lu n = 1e6, search against closing, 13.6 / 13.9 ms and with
// memberships 21.0 / 24.7; n = 3e5, 1.9 / 2.2 and 3.6 / 4.4 (R-MAT of scale 17: 2.8 /
// 2.6 and 4.6 / 5.8).
bool close_supported(int W, int k, int64_t items)
{
    return ((W == 16 && k == 5) || (W >= 8 && W <= 16 && k == 6)) && items < (1 << 22);
}

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
    return c.k == 6 ? launch_bins<4>(c, L, chunks, ctr + 32, s) : launch_bins<3>(c, L, chunks, ctr + 32, s);
}

// The 4-word class, k = 6.
kc_status close_own_launch(const Ctx& c, bool col, cudaStream_t s)
{
    const size_t smem = own_layout().total;
    auto go = [&](auto kern) -> kc_status {
        KC_CK(cc::allow_smem(kern, smem));
        const int grid =
            (int)std::min<int64_t>(c.nitems, (int64_t)num_sms() * cc::blocks_per_sm(kern, kOwnWarps * 32, smem));
        kern<<<grid, kOwnWarps * 32, smem, s>>>(c);
        KC_LAUNCHED();
        return KC_OK;
    };
    return col ? go(k_close_own<true>) : go(k_close_own<false>);
}

}  // namespace kc

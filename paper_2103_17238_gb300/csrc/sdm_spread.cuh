// Larger cells (above the shared-memory classes) when a plan holds few
// super-droplets in them: one step in two short launches spread over the
// whole chip.
//
// A lone box of 2^17 SDs leaves the device nearly idle: what bounds its step
// is the chain of dependent launches and memory latencies (six passes of the
// multi-pass path, 45 us; one CTA's serial work in the cluster path, 62 us for
// 16,000 SDs).  Here every cell is cut into nb buckets of equal key ranges,
// kSpreadMean SDs on average, each with a fixed room in global scratch:
//   1. spread_scatter_kernel  one Philox block (two SDs) per thread; a live
//      SD takes the next place of its bucket's room by one global atomic:
//      (32 key bits below the bucket's, rank), 8 bytes.  No counting pass.
//   2. spread_pairs_kernel    one warp per bucket: the bucket's entries in
//      order (counts of sub-buckets, then a register sort), its first position
//      from the sum of the counts before it (every CTA adds them up itself),
//      and its pairs: gathers, bound, certified filter, exact evaluation and
//      update as in the warp kernel.  A pair that crosses into the next bucket
//      takes that bucket's least entry.  The last CTA of a cell to have read
//      the counts clears them for the next step (the allocation-free step, whose
//      counts outlive a call, clears them ahead of its scatter instead).
// The order of entries within a room is left to the atomics; sorting by
// (key, rank) removes it, so results repeat bit for bit.
//
// Measured (us per step of one box, before -> after): 12,000 SDs 37 -> 8.4,
// 65,536 42 -> 11, 131,072 43 -> 15.  (Above 240,000 SDs sdm_record.cuh is faster.)  Three blocks of the second
// kernel per SM (80 registers) beat two (40 boxes of 12,000: 28 against 31) and
// four (64 registers: 28, but one box of 65,536 14.8 against 13.0).
//
// Mean 56 (40 and 28 took 48 and 56 us against 42 for 76 boxes of 12,000): 57 SDs fill a warp's 28 pairs in one round, and more than 128
// entries (the register sort's room) come once in 1e15 buckets; those, and
// entries that share their 32 + log2 nb key bits, are ranked by counting.  A
// room holds 192: beyond that (once in 1e40) the cell is left unstepped and
// the status says so.
#pragma once

#include "sdm_kernels.cuh"

namespace sdm {

constexpr int kSpreadMean = 56;
// A counter takes 16 bytes: packed, a lone cell's lie in a few L2 slices, which
// then serve all the atomics (box of 2^17: 15.1 us per step with 4 bytes, 15.4
// with 8, 14.4 with 16; four of them: 36.2, 31.4, 30.8).
constexpr int kSpreadStride = 4; // words from one counter to the next
constexpr int kSpreadRoom = 192;
constexpr int kSpreadFast = 128; // entries the register sort takes
constexpr int kSpreadNT = 256;   // threads per block of both kernels
constexpr int kSpreadW = kSpreadNT / 32;

// Words of nb counters.
__host__ __device__ constexpr int spread_words(int nb) { return nb * kSpreadStride; }

struct __align__(16) SpreadCell {
    const InstDev *run; // the run's record
    int32_t cell;       // the cell's index in the random streams
    int32_t off, n;     // its storage slots
    int32_t nb;         // buckets
    int32_t cnt;        // first counter's word; after the counters' words one of arrivals
    int32_t groups;     // CTAs of the second kernel
    int32_t room;       // first bucket's index among all rooms
    int32_t first;      // of a block's item: its first SD pair (scatter) or bucket (pairs)
};

struct SpreadScratch {
    uint32_t *cnt; // zero before a step, and in a plan again after it
    uint2 *rooms;  // kSpreadRoom entries per bucket
};

// A block's item in device memory (everything of its cell beside its place
// in it: one load to the run's record), or one cell as an argument.
struct PlanSpread {
    static constexpr bool kClears = true; // the counts, behind the step
    const SpreadCell *items;
    __device__ __forceinline__ SpreadCell cell(int &first) const
    {
        const SpreadCell c = items[blockIdx.x];
        first = c.first;
        return c;
    }
    __device__ __forceinline__ const InstDev *record(const SpreadCell &c) const { return c.run; }
    __device__ __forceinline__ void overflow(const SpreadCell &c) const
    {
        atomicOr(&const_cast<InstDev *>(c.run)->status, 2u);
    }
};

template <int PER_BLOCK>
struct OneSpread {
    static constexpr bool kClears = false;
    const InstDev *P;
    SpreadCell c;
    uint32_t *status;
    __device__ __forceinline__ SpreadCell cell(int &first) const
    {
        first = (int)blockIdx.x * PER_BLOCK;
        return c;
    }
    __device__ __forceinline__ const InstDev *record(const SpreadCell &) const { return P; }
    __device__ __forceinline__ void overflow(const SpreadCell &) const { set_wrong(status, kWrongRoom); }
};

// Programmatic dependent launch: the next kernel of the chain may become
// resident while this one runs, and waits here for the one before it to be
// complete.  No-ops where the launch does not ask for it.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename SRC>
__device__ __forceinline__ void spread_scatter(const SRC src, const SpreadScratch S, int64_t step_offset)
{
    chain_next();
    int first;
    const SpreadCell c = src.cell(first);
    const InstDev *P = src.record(c);
    const int q = first + (int)threadIdx.x;
    // the keys depend on nothing that the chain changes
    const uint4 w = draw4(P->seed, (uint32_t)q, (uint32_t)c.cell, P->step + step_offset, 0u);
    chain_wait();
    if (2 * q >= c.n)
        return;
    const longlong2 x2 = reinterpret_cast<const longlong2 *>(P->xi + c.off)[q];
    uint32_t b[2], sub[2], slot[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        // bucket and the 32 bits below it: the key times nb, from its top
        const uint64_t p = (uint64_t)(h ? w.z : w.x) * (uint32_t)c.nb + mulhi32(h ? w.w : w.y, (uint32_t)c.nb);
        b[h] = (uint32_t)(p >> 32);
        sub[h] = (uint32_t)p;
        slot[h] = 0xFFFFFFFFu;
        if ((h ? x2.y : x2.x) > 0)
            slot[h] = atomicAdd(S.cnt + c.cnt + b[h] * kSpreadStride, 1u);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (slot[h] < (uint32_t)kSpreadRoom)
            S.rooms[(int64_t)(c.room + (int)b[h]) * kSpreadRoom + slot[h]] = make_uint2(sub[h], (uint32_t)(2 * q + h));
}

struct SpreadSmem {
    uint32_t sub[kSpreadW][kSpreadRoom], rank[kSpreadW][kSpreadRoom]; // entries as they lie in the room
    uint32_t sorted[kSpreadW][kSpreadRoom + 1];                       // ranks in order, then the next bucket's first
    uint32_t hist[kSpreadW][kSpreadFast], word[kSpreadW][kSpreadFast];
    uint32_t before[kSpreadW], all[kSpreadW], big[kSpreadW];
    uint32_t count[kSpreadW], head[kSpreadW + 1], last;
};

__device__ __forceinline__ bool spread_less(uint32_t sa, uint32_t ra, uint32_t sb, uint32_t rb, uint64_t seed,
                                            uint32_t cell, int64_t s)
{
    if (sa != sb)
        return sa < sb;
    return ra != rb && key_less(big_key(seed, cell, s, ra), ra, big_key(seed, cell, s, rb), rb);
}

// Order of n entries by counting (full keys where the 32 bits are equal).
__device__ __noinline__ void spread_order_slow(const uint32_t *sub, const uint32_t *rank, uint32_t *sorted, uint32_t n,
                                               uint64_t seed, uint32_t cell, int64_t s)
{
    for (uint32_t e = threadIdx.x & 31; e < n; e += 32) {
        uint32_t at = 0;
        for (uint32_t m = 0; m < n; ++m)
            at += spread_less(sub[m], rank[m], sub[e], rank[e], seed, cell, s) ? 1u : 0u;
        sorted[at] = rank[e];
    }
}

// Rank of the least entry of the first bucket from b on that holds any (all
// lanes; 0 when there is none, in which case no pair needs it).
__device__ __forceinline__ uint32_t spread_first(const SpreadCell &c, const SpreadScratch &S, int b, uint64_t seed,
                                                 int64_t s)
{
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    uint32_t n = 0;
    for (; b < c.nb && (n = S.cnt[c.cnt + b * kSpreadStride]) == 0u; ++b)
        ;
    n = min(n, (uint32_t)kSpreadRoom);
    if (n == 0)
        return 0u;
    const uint2 *e = S.rooms + (int64_t)(c.room + b) * kSpreadRoom;
    uint2 best = make_uint2(0xFFFFFFFFu, 0xFFFFFFFFu);
    for (uint32_t i = lane; i < n; i += 32) {
        const uint2 x = e[i];
        if (best.y == 0xFFFFFFFFu || spread_less(x.x, x.y, best.x, best.y, seed, (uint32_t)c.cell, s))
            best = x;
    }
    const uint32_t m = __reduce_min_sync(FULL, best.x);
    unsigned who = __ballot_sync(FULL, best.x == m && best.y != 0xFFFFFFFFu);
    uint32_t r = __shfl_sync(FULL, best.y, __ffs(who) - 1);
    for (who &= who - 1u; who; who &= who - 1u) { // equal bits (once in 1e9)
        const uint32_t o = __shfl_sync(FULL, best.y, __ffs(who) - 1);
        if (spread_less(m, o, m, r, seed, (uint32_t)c.cell, s))
            r = o;
    }
    return r;
}

template <typename SRC>
__device__ __forceinline__ void spread_pairs(const SRC src, const SpreadScratch S, int64_t step_offset, SpreadSmem &M)
{
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr int E = kSpreadFast / 32;
    constexpr uint32_t SM = (uint32_t)kSpreadFast - 1u; // place in the room, below the key bits of a word
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    chain_next();
    int b0;
    const SpreadCell c = src.cell(b0);
    const InstDev *__restrict__ P = src.record(c);
    const uint64_t seed = P->seed;
    const int64_t s = P->step + step_offset;
    const uint32_t *cnt = S.cnt + c.cnt;
    const int b = b0 + warp;
    chain_wait();
    // this bucket's entries, while the counts are added up
    const uint32_t raw = b < c.nb ? cnt[b * kSpreadStride] : 0u;
    const uint32_t nk = min(raw, (uint32_t)kSpreadRoom);
    const uint2 *room = S.rooms + (int64_t)(c.room + b) * kSpreadRoom;
    uint2 ent[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const uint32_t e = lane + 32 * i;
        ent[i] = e < nk ? room[e] : make_uint2(0u, 0u);
    }
    uint32_t before = 0, all = 0, big = 0;
    for (int i = t; i < c.nb; i += kSpreadNT) {
        const uint32_t x = cnt[i * kSpreadStride];
        all += x;
        before += i < b0 ? x : 0u;
        big |= x > (uint32_t)kSpreadRoom ? 1u : 0u;
    }
    before = __reduce_add_sync(FULL, before);
    all = __reduce_add_sync(FULL, all);
    big = __reduce_or_sync(FULL, big);
    if (lane == 0) {
        M.before[warp] = before;
        M.all[warp] = all;
        M.big[warp] = big;
        M.count[warp] = nk;
    }
    // ---- order of the bucket
    uint32_t *sub = M.sub[warp], *rank = M.rank[warp], *sorted = M.sorted[warp];
    uint32_t *hist = M.hist[warp], *wrd = M.word[warp];
    reinterpret_cast<uint4 *>(hist)[lane] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const uint32_t e = lane + 32 * i;
        if (e < nk) {
            sub[e] = ent[i].x;
            rank[e] = ent[i].y;
        }
    }
    for (uint32_t e = lane + kSpreadFast; e < nk; e += 32) {
        const uint2 x = room[e];
        sub[e] = x.x;
        rank[e] = x.y;
    }
    __syncwarp();
    bool fast = nk <= (uint32_t)kSpreadFast;
    if (fast) { // uniform over the warp
        uint32_t word[E], slot[E];
#pragma unroll
        for (int i = 0; i < E; ++i) {
            word[i] = (ent[i].x & ~SM) | (uint32_t)(lane + 32 * i);
            slot[i] = 0;
            if ((uint32_t)(lane + 32 * i) < nk)
                slot[i] = atomicAdd(&hist[word[i] >> 25], 1u);
        }
        __syncwarp();
        const uint4 k = reinterpret_cast<const uint4 *>(hist)[lane];
        const uint32_t sum = k.x + k.y + k.z + k.w;
        uint32_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, incl, d);
            if (lane >= d)
                incl += y;
        }
        const uint32_t r0 = incl - sum;
        reinterpret_cast<uint4 *>(hist)[lane] = make_uint4(r0, r0 + k.x, r0 + k.x + k.y, r0 + k.x + k.y + k.z);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < E; ++i)
            if ((uint32_t)(lane + 32 * i) < nk)
                wrd[hist[word[i] >> 25] + slot[i]] = word[i];
        __syncwarp();
        // each lane's E consecutive words in registers, then swaps across lanes
        // (as the warp kernel's sort)
        const uint4 w4 = reinterpret_cast<const uint4 *>(wrd)[lane];
        uint32_t v[E] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int i = 0; i < E; ++i)
            if ((uint32_t)(E * lane + i) >= nk)
                v[i] = 0xFFFFFFFFu;
        sort_net<E>(v);
        for (int round = 0;; ++round) {
            const uint32_t pl = __shfl_up_sync(FULL, v[E - 1], 1), nf = __shfl_down_sync(FULL, v[0], 1);
            const bool lo_inv = lane > 0 && pl > v[0], hi_inv = lane < 31 && v[E - 1] > nf;
            if (!__any_sync(FULL, lo_inv || hi_inv))
                break;
            if (round == kMaxSwapRounds) {
                fast = false;
                break;
            }
            if (lo_inv)
                v[0] = pl;
            if (hi_inv)
                v[E - 1] = nf;
            sort_net<E>(v);
        }
        bool tie = false;
#pragma unroll
        for (int i = 0; i + 1 < E; ++i)
            tie |= ((v[i] ^ v[i + 1]) - 1u) < SM;
        const uint32_t nf = __shfl_down_sync(FULL, v[0], 1);
        if (lane < 31)
            tie |= ((v[E - 1] ^ nf) - 1u) < SM;
        fast &= !__any_sync(FULL, tie);
        if (fast)
#pragma unroll
            for (int i = 0; i < E; ++i)
                if ((uint32_t)(E * lane + i) < nk)
                    sorted[E * lane + i] = rank[v[i] & SM];
    }
    if (!fast)
        spread_order_slow(sub, rank, sorted, nk, seed, (uint32_t)c.cell, s);
    __syncwarp();
    if (warp == kSpreadW - 1) { // what follows the CTA's last bucket
        const uint32_t f = spread_first(c, S, b0 + kSpreadW, seed, s);
        if (lane == 0)
            M.head[kSpreadW] = f;
    }
    if (lane == 0)
        M.head[warp] = nk ? sorted[0] : 0u;
    __syncthreads();

    // ---- positions
    uint32_t start = 0, n_c = 0, bad = 0;
#pragma unroll
    for (int w = 0; w < kSpreadW; ++w) {
        start += M.before[w] + (w < warp ? M.count[w] : 0u);
        n_c += M.all[w];
        bad |= M.big[w];
    }
    if (t == 0) { // every thread's reads of the counts are done
        if constexpr (SRC::kClears) {
            __threadfence();
            M.last = atomicAdd(S.cnt + c.cnt + spread_words(c.nb), 1u) == (uint32_t)c.groups - 1u ? 1u : 0u;
        }
        if (bad && b0 == 0)
            src.overflow(c);
    }
    if (!bad && nk > 0) {
        uint32_t next = M.head[kSpreadW];
        for (int w = kSpreadW - 1; w > warp; --w)
            if (M.count[w])
                next = M.head[w];
        if (lane == 0)
            sorted[nk] = next;
        __syncwarp();
        const float ratio_f = u32_to_f32_rn((n_c & 1u) ? n_c : n_c - 1u);
        const PairConsts C = pair_consts(P);
        const float sc = C.dtdvf * ratio_f;
        int64_t *__restrict__ gxi = P->xi + c.off;
        double *__restrict__ gv = P->v + c.off;
        const uint32_t n_pairs = n_c / 2, l1 = min(n_pairs, (start + nk + 1u) / 2u);
        for (uint32_t l = (start + 1u) / 2u + lane; l < l1; l += 32) { // pairs whose first SD lies here
            uint32_t a = sorted[2 * l - start], bb = sorted[2 * l + 1 - start];
            int64_t xa = gxi[a], xb = gxi[bb];
            double va = gv[a], vb = gv[bb];
            const uint4 w = draw4(seed, l >> 1, (uint32_t)c.cell, s, 1u);
            const uint32_t wa = (l & 1u) ? w.z : w.x, wb = (l & 1u) ? w.w : w.y;
            if (xa < xb) { // j holds the larger multiplicity; ties keep the earlier
                const uint32_t tr = a;
                a = bb;
                bb = tr;
                const int64_t tx = xa;
                xa = xb;
                xb = tx;
                const double tv = va;
                va = vb;
                vb = tv;
            }
            const uint32_t ha = (uint32_t)__double2hiint(va), hb = (uint32_t)__double2hiint(vb);
            if (pair_prefilter_zero(C, sc, xa, ha, hb, wa))
                continue;
            const int32_t gf = pair_gamma_filter(C, ratio_f, xa, ha, hb, wa);
            if (gf == 0)
                continue;
            const int64_t g = gf > 0 ? cap_gamma(gf, xa, xb) : pair_gamma_exact(P, n_c, xa, xb, va, vb, wa, wb);
            if (g > 0) {
                const bool split = shima_update(g, xa, xb, va, vb);
                gxi[a] = xa;
                gxi[bb] = xb;
                gv[bb] = vb;
                if (split)
                    gv[a] = va;
            }
        }
    }
    if constexpr (SRC::kClears) {
        __syncthreads();
        if (M.last) // the counts and the arrivals are zero again for the next step
            for (int i = t; i <= spread_words(c.nb); i += kSpreadNT)
                S.cnt[c.cnt + i] = 0u;
    }
}

__global__ void __launch_bounds__(kSpreadNT) spread_scatter_kernel(PlanSpread src, SpreadScratch S, int64_t step_offset)
{
    spread_scatter(src, S, step_offset);
}

__global__ void __launch_bounds__(kSpreadNT, 3) spread_pairs_kernel(PlanSpread src, SpreadScratch S, int64_t step_offset)
{
    __shared__ __align__(16) SpreadSmem M;
    spread_pairs(src, S, step_offset, M);
}

// The counters of one cell to zero, ahead of its scatter.
__global__ void __launch_bounds__(kSpreadNT) one_spread_clear_kernel(SpreadCell c, SpreadScratch S)
{
    chain_next();
    const int b = (int)blockIdx.x * kSpreadNT + (int)threadIdx.x;
    if (b < c.nb)
        S.cnt[c.cnt + b * kSpreadStride] = 0u;
}

__global__ void __launch_bounds__(kSpreadNT) one_spread_scatter_kernel(const __grid_constant__ InstDev P, SpreadCell c,
                                                                       SpreadScratch S, uint32_t *status)
{
    spread_scatter(OneSpread<kSpreadNT>{&P, c, status}, S, 0);
}

__global__ void __launch_bounds__(kSpreadNT) one_spread_pairs_kernel(const __grid_constant__ InstDev P, SpreadCell c,
                                                                     SpreadScratch S, uint32_t *status)
{
    __shared__ __align__(16) SpreadSmem M;
    spread_pairs(OneSpread<kSpreadW>{&P, c, status}, S, 0, M);
}

// A cell's place in a plan's scratch (counters and rooms so far, advanced).
inline SpreadCell spread_cell(const InstDev *run, int32_t cell, int32_t off, int32_t n, int64_t &counters,
                              int64_t &rooms)
{
    SpreadCell c{};
    c.run = run;
    c.cell = cell;
    c.off = off;
    c.n = n;
    c.nb = std::max(1, (n + kSpreadMean - 1) / kSpreadMean);
    c.groups = (c.nb + kSpreadW - 1) / kSpreadW;
    c.cnt = (int32_t)counters;
    c.room = (int32_t)rooms;
    counters += spread_words(c.nb) + kSpreadStride;
    rooms += c.nb;
    return c;
}

} // namespace sdm

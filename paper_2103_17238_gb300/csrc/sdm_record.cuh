// Larger cells (above the shared-memory classes, up to 2^24 super-droplets)
// when a plan holds many super-droplets in them: one step in four launches,
// with a 16-byte record of every live SD carried through the sort.  (Measured
// per step, us, before -> after: 16 boxes of 2^20 480 -> 352, one 51 -> 31, one of 2^24
// 1024 -> 474, 200 of 16,000 124 -> 66, 1024 boxes of 2^8 .. 2^16 337 -> 222.)
//
// What bounds a step of such cells is not bandwidth but single-lane accesses:
// a load or store whose 32 lanes go to 32 places takes an SM's load/store unit
// 32 cycles (16 boxes of 2^20 SDs: 57 us per access of every SD).  The
// multi-pass path spends three of them on every SD (its rank scattered, its xi
// and its v gathered) and draws every key twice more.  Here:
//   1. rec_scatter_kernel  a chunk of SDs per block: one Philox block per two
//      SDs; places within (chunk, bucket) from shared atomics, the chunk's
//      piece of every bucket's room from one global atomic each; then
//      one 16-byte store per live SD: 32 key bits below the bucket's, rank, xi
//      truncated to binary32 and v's high word;
//   2. rec_scan_kernel     first positions of the buckets (above kRecSumSd; else
//      each bucket's block adds up the counts);
//   3. rec_pairs_kernel    one block per bucket: its records by one bulk copy,
//      ordered by their key bits; the pairs' bound (pair_prefilter_zero needs no
//      more than the record) on all of them, and only what it leaves
//      gathers its xi and v for the certified filter and the update;
//   4. rec_seam_kernel     the pairs that cross from one bucket into the next.
// Entries lie in a room in the order of the atomics; sorting by (key, rank)
// removes it, so results repeat bit for bit.
//
// Buckets hold up to kRecMean SDs on average, a room kRecRoom: 12 standard
// deviations more (once in 1e30); beyond it the cell is left unstepped and the
// status says so.
#pragma once

#include "sdm_spread.cuh"

namespace sdm {

constexpr int kRecMean = 1024; // (16 boxes of 2^20: 800 took 369 us a step against 353, 1280 349)
constexpr int kRecRoom = 1408;
// 1024 threads of 32 registers, two blocks per SM: the loads of xi and v, then the
// atomics, are what a block waits for (512 threads of 64 registers: 405 against
// 347 us; chunks of 8192, four pairs a thread: 489).
constexpr int kRecScatterNT = 1024;
constexpr int kRecChunk = 4096; // SDs per scatter block
// Five blocks of 256 per SM (48 registers): 354 us against 370 with four, 405 with three;
// 512 threads 457, six blocks (40 registers, spills) 399.
constexpr int kRecNT = 256; // threads of a bucket's block
// Groups of up to this many SDs have no scan launch: every bucket's block adds up its
// cell's counts (us, scan | sums: one box of 2^18 19.6 | 18.7, of 2^20 31.4 | 30.4, of 2^21
// 51.6 | 51.1; 16 of 2^15 23.0 | 21.7; but 32 of 2^17 88.8 | 89.6, 16 of 2^20 349 | 356, one
// of 2^24 462 | 512).
constexpr int64_t kRecSumSd = (int64_t)1 << 21;
constexpr int kRecSubLB = 9;    // sub-buckets inside a bucket
constexpr int kRecMaxBuckets = 16384; // (their counts take 64 KB of shared memory)
constexpr int kRecMaxSd = kRecMaxBuckets * kRecMean;

struct __align__(16) RecCell {
    const InstDev *run;
    int32_t cell;   // index in the random streams
    int32_t off, n; // storage slots
    int32_t nb;     // buckets
    int32_t first;  // first bucket among all cells' (counts, seams, rooms)
    int32_t start;  // its first position word among all cells' (nb + 1 each)
};

// Buckets of a cell of n SDs.
__host__ __device__ constexpr int rec_buckets(int n) { return (n + kRecMean - 1) / kRecMean; }

struct RecScratch {
    uint32_t *cnt;    // per bucket: entries; zero before a step's scatter
    uint32_t *start;  // per bucket: first position; a cell's count of live SDs behind its last
                      // (kRecVoid: a room overflowed)
    uint2 *seam;      // per bucket that holds any: ranks of its first and last SD (kRecVoid: its wait gave up)
    uint4 *rooms;     // kRecRoom records per bucket
};
constexpr uint32_t kRecVoid = 0xFFFFFFFFu;

// Polls of a bucket's wait for its records (a test's build lets some give up at once).
#ifndef SDM_REC_POLLS
#define SDM_REC_POLLS(bucket) kWaitPolls
#endif

__global__ void __launch_bounds__(kRecScatterNT, 2) rec_scatter_kernel(const BigChunk *__restrict__ work,
                                                                    const RecCell *__restrict__ cells, RecScratch S,
                                                                    int64_t step_offset)
{
    constexpr int QPT = kRecChunk / 2 / kRecScatterNT; // SD pairs per thread
    static_assert(QPT * kRecScatterNT * 2 == kRecChunk, "chunk = threads x pairs");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(smem_raw);
    chain_next();
    const BigChunk w = work[blockIdx.x];
    const RecCell c = cells[w.big];
    const InstDev *__restrict__ P = c.run;
    const int t = threadIdx.x, q0 = w.chunk * (kRecChunk / 2) + t;
    for (int i = t; i < c.nb; i += kRecScatterNT)
        s_cnt[i] = 0u;
    uint32_t sub[2 * QPT], at[2 * QPT]; // at: bucket above place in the chunk's piece
    const uint64_t seed = P->seed;
    const int64_t s = P->step + step_offset;
#pragma unroll
    for (int i = 0; i < QPT; ++i) { // the keys depend on nothing that the chain changes
        const uint4 k = draw4(seed, (uint32_t)(q0 + i * kRecScatterNT), (uint32_t)c.cell, s, 0u);
        const uint64_t p0 = (uint64_t)k.x * (uint32_t)c.nb + mulhi32(k.y, (uint32_t)c.nb);
        const uint64_t p1 = (uint64_t)k.z * (uint32_t)c.nb + mulhi32(k.w, (uint32_t)c.nb);
        at[2 * i] = (uint32_t)(p0 >> 32);
        sub[2 * i] = (uint32_t)p0;
        at[2 * i + 1] = (uint32_t)(p1 >> 32);
        sub[2 * i + 1] = (uint32_t)p1;
    }
    chain_wait();
    const longlong2 *gx = reinterpret_cast<const longlong2 *>(P->xi + c.off);
    const double2 *gv = reinterpret_cast<const double2 *>(P->v + c.off);
    longlong2 x[QPT];
    double2 v[QPT];
#pragma unroll
    for (int i = 0; i < QPT; ++i) { // every load first
        const int q = q0 + i * kRecScatterNT;
        const bool in = 2 * q < c.n;
        x[i] = in ? gx[q] : make_longlong2(0, 0);
        v[i] = in ? gv[q] : make_double2(1.0, 1.0);
    }
    float xf[2 * QPT]; // 0: dead
    uint32_t vh[2 * QPT];
#pragma unroll
    for (int i = 0; i < 2 * QPT; ++i) {
        const int64_t xi = (i & 1) ? x[i / 2].y : x[i / 2].x;
        xf[i] = xi > 0 ? xi2f(xi) : 0.0f;
        vh[i] = (uint32_t)__double2hiint((i & 1) ? v[i / 2].y : v[i / 2].x);
    }
    __syncthreads(); // the counts are zero
#pragma unroll
    for (int i = 0; i < 2 * QPT; ++i)
        at[i] = xf[i] != 0.0f ? (at[i] << 16) | atomicAdd(&s_cnt[at[i]], 1u) : 0xFFFFFFFFu;
    __syncthreads();
    for (int i = t; i < c.nb; i += kRecScatterNT) {
        const uint32_t k = s_cnt[i];
        if (k)
            s_cnt[i] = atomicAdd(S.cnt + c.first + i, k);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2 * QPT; ++i) {
        if (at[i] == 0xFFFFFFFFu)
            continue;
        const uint32_t b = at[i] >> 16, e = s_cnt[b] + (at[i] & 0xFFFFu);
        if (e < (uint32_t)kRecRoom)
            S.rooms[(int64_t)(c.first + (int)b) * kRecRoom + e] =
                make_uint4(sub[i], (uint32_t)(2 * (q0 + (i / 2) * kRecScatterNT) + (i & 1)),
                           __float_as_uint(xf[i]), vh[i]);
    }
}

// One block per cell: the buckets' first positions.
constexpr int kRecScanNT = 1024;
__global__ void __launch_bounds__(kRecScanNT) rec_scan_kernel(const RecCell *__restrict__ cells, RecScratch S)
{
    constexpr unsigned FULL = 0xFFFFFFFFu;
    __shared__ uint32_t s_w[32];
    chain_next();
    const RecCell c = cells[blockIdx.x];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t *cnt = S.cnt + c.first;
    uint32_t *start = S.start + c.start;
    chain_wait();
    uint32_t carry = 0, big = 0;
    for (int i0 = 0; i0 < c.nb; i0 += kRecScanNT) {
        const int i = i0 + t;
        const uint32_t x = i < c.nb ? cnt[i] : 0u;
        big |= x > (uint32_t)kRecRoom ? 1u : 0u;
        uint32_t incl = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, incl, d);
            if (lane >= d)
                incl += y;
        }
        if (lane == 31)
            s_w[warp] = incl;
        __syncthreads();
        const uint32_t w = s_w[lane];
        const uint32_t before = __reduce_add_sync(FULL, lane < warp ? w : 0u), all = __reduce_add_sync(FULL, w);
        if (i < c.nb)
            start[i] = carry + before + incl - x;
        carry += all;
        __syncthreads();
    }
    const int over = __syncthreads_or((int)big);
    if (t == 0) {
        start[c.nb] = over ? kRecVoid : carry;
        if (over)
            atomicOr(&const_cast<InstDev *>(c.run)->status, 2u);
    }
}

struct RecSmem {
    uint4 rec[kRecRoom];
    uint32_t word[kRecRoom]; // 21 key bits above the record's place, in sub-buckets; then (16 bits each) the order
    uint32_t hist[(1 << kRecSubLB) + 4];
    uint16_t list[kRecRoom / 2 + 2]; // pairs the bound leaves
    uint32_t warp[32], sum[2][kRecNT / 32];
    uint64_t bar;
    uint32_t n_list;
};

// A pair of SDs a, b in full: the certified filter, the exact evaluation where
// it cannot decide, the update.
__device__ __forceinline__ void rec_pair(const InstDev *P, const PairConsts &C, uint32_t n_c, float ratio_f,
                                         int64_t *__restrict__ gxi, double *__restrict__ gv, uint32_t a, uint32_t b,
                                         uint32_t wa, uint32_t wb)
{
    int64_t xa = gxi[a], xb = gxi[b];
    double va = gv[a], vb = gv[b];
    if (xa < xb) { // j holds the larger multiplicity; ties keep the earlier
        const uint32_t tr = a;
        a = b;
        b = tr;
        const int64_t tx = xa;
        xa = xb;
        xb = tx;
        const double tv = va;
        va = vb;
        vb = tv;
    }
    const int32_t gf = pair_gamma_filter(C, ratio_f, xa, va, vb, wa);
    if (gf == 0)
        return;
    const int64_t g = gf > 0 ? cap_gamma(gf, xa, xb) : pair_gamma_exact(P, n_c, xa, xb, va, vb, wa, wb);
    if (g > 0) {
        const bool split = shima_update(g, xa, xb, va, vb);
        gxi[a] = xa;
        gxi[b] = xb;
        gv[b] = vb;
        if (split)
            gv[a] = va;
    }
}

// SUM: a bucket's block adds up the counts itself and writes its first position
// for the seam kernel; else rec_scan_kernel has.
template <bool SUM>
__global__ void __launch_bounds__(kRecNT, 5) rec_pairs_kernel(const BigBucket *__restrict__ work,
                                                           const RecCell *__restrict__ cells, RecScratch S,
                                                           int64_t step_offset)
{
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr int NSB = 1 << kRecSubLB, NW = kRecNT / 32, HPT = NSB / kRecNT;
    constexpr int R = (kRecRoom + kRecNT - 1) / kRecNT;
    constexpr uint32_t EM = 2047u; // a record's place in a word
    static_assert(kRecRoom <= 2048 && kRecSubLB + 21 <= 32 && HPT >= 1 && HPT * kRecNT == NSB, "words");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    RecSmem &M = *reinterpret_cast<RecSmem *>(smem_raw);
    chain_next();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const BigBucket w = work[blockIdx.x];
    const RecCell c = cells[w.big];
    if (t == 0) {
        mbar_init(&M.bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        M.n_list = 0u;
    }
#pragma unroll
    for (int i = 0; i < HPT; ++i)
        M.hist[t + i * kRecNT] = 0u;
    const InstDev *__restrict__ P = c.run;
    const uint64_t seed = P->seed;
    const int64_t s = P->step + step_offset;
    const uint32_t cell = (uint32_t)c.cell;
    chain_wait();
    const uint4 *room = S.rooms + (int64_t)(c.first + w.bucket) * kRecRoom;
    uint32_t *st = S.start + c.start + w.bucket;
    uint32_t start, n_c, nk;
    if constexpr (SUM) {
        const uint32_t *cnt = S.cnt + c.first;
        uint32_t before = 0, all = 0, big = 0;
        for (int i = t; i < c.nb; i += kRecNT) {
            const uint32_t x = cnt[i];
            all += x;
            before += i < w.bucket ? x : 0u;
            big |= x > (uint32_t)kRecRoom ? 1u : 0u;
        }
        nk = cnt[w.bucket];
        before = __reduce_add_sync(FULL, before);
        all = __reduce_add_sync(FULL, all);
        if (lane == 0) {
            M.sum[0][warp] = before;
            M.sum[1][warp] = all;
        }
        const int over = __syncthreads_or((int)big);
        start = __reduce_add_sync(FULL, lane < NW ? M.sum[0][lane] : 0u);
        n_c = over ? kRecVoid : __reduce_add_sync(FULL, lane < NW ? M.sum[1][lane] : 0u);
        if (t == 0) {
            st[0] = start;
            if (w.bucket == 0) {
                st[c.nb] = n_c;
                if (over)
                    atomicOr(&const_cast<InstDev *>(P)->status, 2u);
            }
        }
    } else {
        start = st[0];
        n_c = st[c.nb - w.bucket];
        nk = (w.bucket + 1 < c.nb ? st[1] : n_c) - start;
    }
    if (n_c == kRecVoid || nk == 0) // uniform
        return;
    if (t == 0) {
        mbar_arrive_expect_tx(&M.bar, nk * 16u);
        bulk_g2s(M.rec, room, nk * 16u, &M.bar);
    }
    __syncthreads();
    const bool arrived = mbar_wait_bounded(&M.bar, 0u, SDM_REC_POLLS(w.bucket));
    if (!__syncthreads_and(arrived)) { // report, leave no ranks for the seams, wait (bounded) for the copy, leave
        if (t == 0) {
            atomicOr(&const_cast<InstDev *>(P)->status, 1u);
            S.seam[c.first + w.bucket] = make_uint2(kRecVoid, kRecVoid);
            mbar_wait_bounded(&M.bar, 0u);
        }
        return;
    }
    // ---- order of the bucket
    uint32_t word[R], slot[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint32_t e = (uint32_t)(t + r * kRecNT);
        if (e < nk) {
            const uint32_t sub = M.rec[e].x;
            word[r] = ((sub << kRecSubLB) & ~EM) | e;
            const uint32_t b = sub >> (32 - kRecSubLB);
            slot[r] = (b << 16) | atomicAdd(&M.hist[b], 1u);
        }
    }
    __syncthreads();
    {
        uint32_t k[HPT], sum = 0;
#pragma unroll
        for (int i = 0; i < HPT; ++i) {
            k[i] = M.hist[t * HPT + i];
            sum += k[i];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, incl, d);
            if (lane >= d)
                incl += y;
        }
        if (lane == 31)
            M.warp[warp] = incl;
        __syncthreads();
        uint32_t run = __reduce_add_sync(FULL, lane < warp && lane < NW ? M.warp[lane] : 0u) + incl - sum;
#pragma unroll
        for (int i = 0; i < HPT; ++i) {
            M.hist[t * HPT + i] = run;
            run += k[i];
        }
        if (t == 0)
            M.hist[NSB] = nk;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r)
        if ((uint32_t)(t + r * kRecNT) < nk)
            M.word[M.hist[slot[r] >> 16] + (slot[r] & 0xFFFFu)] = word[r];
    __syncthreads();
    // a record's place in the order: its sub-bucket's smaller words (about one)
    uint32_t pos[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if ((uint32_t)(t + r * kRecNT) >= nk)
            continue;
        const uint32_t lo = M.hist[slot[r] >> 16], hi = M.hist[(slot[r] >> 16) + 1u];
        uint32_t k = 0;
        bool tie = false;
        for (uint32_t m = lo; m < hi; ++m) {
            const uint32_t o = M.word[m];
            k += o < word[r] ? 1u : 0u;
            tie |= ((o ^ word[r]) - 1u) < EM; // another record with the same key bits
        }
        if (tie) { // (once in a thousand buckets) all 32 bits, then the keys
            const uint4 me = M.rec[word[r] & EM];
            k = 0;
            for (uint32_t m = lo; m < hi; ++m) {
                const uint4 o = M.rec[M.word[m] & EM];
                k += spread_less(o.x, o.y, me.x, me.y, seed, cell, s) ? 1u : 0u;
            }
        }
        pos[r] = lo + k;
    }
    __syncthreads();
    uint16_t *order = reinterpret_cast<uint16_t *>(M.word);
#pragma unroll
    for (int r = 0; r < R; ++r)
        if ((uint32_t)(t + r * kRecNT) < nk)
            order[pos[r]] = (uint16_t)(word[r] & EM);
    __syncthreads();
    if (t == 0)
        S.seam[c.first + w.bucket] = make_uint2(M.rec[order[0]].y, M.rec[order[nk - 1]].y);
    // ---- the pairs that lie in the bucket: the bound
    const PairConsts C = pair_consts(P);
    const float ratio_f = u32_to_f32_rn((n_c & 1u) ? n_c : n_c - 1u);
    const float sc = C.dtdvf * ratio_f;
    const uint32_t l0 = (start + 1u) / 2u, l1 = (start + nk) / 2u; // (2 l1 <= n_c)
    for (uint32_t q = l0 / 2u + (uint32_t)t; 2u * q < l1; q += kRecNT) {
        const uint4 u = draw4(seed, q, cell, s, 1u);
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h) {
            const uint32_t l = 2u * q + h;
            if (l < l0 || l >= l1)
                continue;
            const uint4 a = M.rec[order[2u * l - start]], b = M.rec[order[2u * l + 1u - start]];
            if (!pair_prefilter_zero(C, sc, fmaxf(__uint_as_float(a.z), __uint_as_float(b.z)), a.w, b.w, h ? u.z : u.x))
                M.list[atomicAdd(&M.n_list, 1u)] = (uint16_t)(l - l0);
        }
    }
    __syncthreads();
    // ---- what it leaves, a pair per thread
    int64_t *__restrict__ gxi = P->xi + c.off;
    double *__restrict__ gv = P->v + c.off;
    for (uint32_t i = (uint32_t)t; i < M.n_list; i += kRecNT) {
        const uint32_t l = l0 + M.list[i];
        const uint4 u = draw4(seed, l >> 1, cell, s, 1u);
        rec_pair(P, C, n_c, ratio_f, gxi, gv, M.rec[order[2u * l - start]].y, M.rec[order[2u * l + 1u - start]].y,
                 (l & 1u) ? u.z : u.x, (l & 1u) ? u.w : u.y);
    }
}

// A thread per bucket: the pair of its last SD and the first of the next bucket
// that holds any, when its last position is a pair's first.
constexpr int kRecSeamNT = 128;
__global__ void __launch_bounds__(kRecSeamNT) rec_seam_kernel(const BigBucket *__restrict__ work, int32_t n_work,
                                                              const RecCell *__restrict__ cells, RecScratch S,
                                                              int64_t step_offset)
{
    chain_next();
    const int i = (int)blockIdx.x * kRecSeamNT + (int)threadIdx.x;
    const BigBucket w = i < n_work ? work[i] : BigBucket{0, 0};
    const RecCell c = cells[w.big];
    chain_wait();
    if (i >= n_work)
        return;
    S.cnt[c.first + w.bucket] = 0u; // for the next step
    const uint32_t *st = S.start + c.start;
    const uint32_t n_c = st[c.nb], start = st[w.bucket];
    if (n_c == kRecVoid)
        return;
    const uint32_t end = w.bucket + 1 < c.nb ? st[w.bucket + 1] : n_c;
    if (end == start || !(end & 1u) || end >= n_c) // empty; a pair's second; the last of an odd count
        return;
    int b = w.bucket + 1;
    while ((b + 1 < c.nb ? st[b + 1] : n_c) == end) // (end < n_c: some bucket holds the next position)
        ++b;
    const uint32_t ra = S.seam[c.first + w.bucket].y, rb = S.seam[c.first + b].x;
    if (ra == kRecVoid || rb == kRecVoid) // a bucket whose wait gave up: its SDs stay as they are
        return;
    const InstDev *__restrict__ P = c.run;
    const uint32_t l = end / 2u;
    const uint4 u = draw4(P->seed, l >> 1, (uint32_t)c.cell, P->step + step_offset, 1u);
    rec_pair(P, pair_consts(P), n_c, u32_to_f32_rn((n_c & 1u) ? n_c : n_c - 1u), P->xi + c.off, P->v + c.off,
             ra, rb, (l & 1u) ? u.z : u.x, (l & 1u) ? u.w : u.y);
}

} // namespace sdm

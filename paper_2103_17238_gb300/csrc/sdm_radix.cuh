// Stable LSD radix sort of (key, value) pairs of 32 bits by 8-bit digits:
// super-droplets by group, in increasing id within a group (the input comes in
// id order).  Used by the sedimentation step and by sdm_set_attributes when
// the caller's cells are in no order.
#pragma once

#include "sdm_kernels.cuh"

namespace sdm {

constexpr int kRadixNT = 256;
// Keys per block and pass: 4096 (1,024 tiles of 4.19M keys make one wave; tiles
// of 2048 or 8192 took 0.224 and 0.241 ms against 0.210 per sort there), or 1024
// below 2^21 keys, where tiles of 4096 leave SMs with one or none (sdm_set_attributes of
// 975,000 in no order 150 against 141 us).
constexpr int kRadixRounds = 16, kRadixRoundsFew = 4;
constexpr int64_t kRadixFew = (int64_t)1 << 21;
constexpr int radix_rounds(int64_t n) { return n < kRadixFew ? kRadixRoundsFew : kRadixRounds; }
constexpr int kRadixBuckets = 256;                  // 8-bit digits

// hist[d * n_tiles + tile] = keys of the tile whose digit (key >> shift) & 255 is d.
template <int ROUNDS>
__global__ void __launch_bounds__(kRadixNT) radix_hist_kernel(const uint32_t *__restrict__ keys, int64_t n, int shift,
                                                              uint32_t *__restrict__ hist, int32_t n_tiles)
{
    __shared__ uint32_t h[kRadixBuckets];
    const int t = threadIdx.x;
    h[t] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (kRadixNT * ROUNDS);
    uint32_t k[ROUNDS]; // every load of the thread in flight at once
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int64_t i = base + (int64_t)r * kRadixNT + t;
        k[r] = i < n ? keys[i] : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r)
        if (base + (int64_t)r * kRadixNT + t < n)
            atomicAdd(&h[(k[r] >> shift) & 255u], 1u);
    __syncthreads();
    hist[(int64_t)t * n_tiles + blockIdx.x] = h[t];
}

// Block d: exclusive scan, in place, of the counts of digit d over the
// tiles (one contiguous row of hist), in chunks of 1024 with a running
// carry; total[d] = the row's sum.
__global__ void __launch_bounds__(1024) radix_row_scan_kernel(uint32_t *__restrict__ hist, int32_t n_tiles,
                                                              uint32_t *__restrict__ total)
{
    __shared__ uint32_t s[1024];
    __shared__ uint32_t s_warp[32];
    const int t = threadIdx.x;
    uint32_t *row = hist + (int64_t)blockIdx.x * n_tiles;
    uint32_t carry = 0;
    for (int32_t c0 = 0; c0 < n_tiles; c0 += 1024) {
        const int32_t i = c0 + t;
        s[t] = i < n_tiles ? row[i] : 0u;
        __syncthreads();
        const uint32_t sum = block_exclusive_scan<1024, 1024>(s, s_warp);
        if (i < n_tiles)
            row[i] = carry + s[t];
        carry += sum;
        __syncthreads();
    }
    if (t == 0)
        total[blockIdx.x] = carry;
}

// One block of 256: exclusive scan of the digit totals, in place.
__global__ void __launch_bounds__(kRadixBuckets) radix_digit_scan_kernel(uint32_t *__restrict__ total)
{
    __shared__ uint32_t s[kRadixBuckets];
    __shared__ uint32_t s_warp[32];
    s[threadIdx.x] = total[threadIdx.x];
    __syncthreads();
    block_exclusive_scan<kRadixBuckets, kRadixBuckets>(s, s_warp);
    total[threadIdx.x] = s[threadIdx.x];
}

// Stable scatter of one pass: tile keys in index order (round-major, thread
// minor); within a round, lanes of a warp with equal digits are ranked by
// __match_any_sync, warps by their per-digit counts in shared memory.
// vals_in null: the values are the indices.
template <int ROUNDS>
__global__ void __launch_bounds__(kRadixNT) radix_scatter_kernel(const uint32_t *__restrict__ keys_in,
                                                                 const uint32_t *__restrict__ vals_in, int64_t n,
                                                                 int shift, const uint32_t *__restrict__ offs,
                                                                 const uint32_t *__restrict__ digit_base,
                                                                 int32_t n_tiles, uint32_t *__restrict__ keys_out,
                                                                 uint32_t *__restrict__ vals_out)
{
    constexpr int NW = kRadixNT / 32;
    __shared__ uint32_t s_base[kRadixBuckets + 1];
    __shared__ uint32_t s_wcnt[NW][kRadixBuckets + 1];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    s_base[t] = digit_base[t] + offs[(int64_t)t * n_tiles + blockIdx.x];
    for (int i = t; i < NW * (kRadixBuckets + 1); i += kRadixNT)
        (&s_wcnt[0][0])[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (kRadixNT * ROUNDS);
    const unsigned lt = (1u << lane) - 1u;
    uint32_t kk[ROUNDS], vv[ROUNDS]; // every load of the thread in flight at once
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int64_t i = base + (int64_t)r * kRadixNT + t;
        kk[r] = i < n ? keys_in[i] : 0u;
        vv[r] = i < n ? (vals_in ? vals_in[i] : (uint32_t)i) : 0u;
    }
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int64_t i = base + (int64_t)r * kRadixNT + t;
        const bool valid = i < n;
        const uint32_t k = kk[r];
        const uint32_t v = vv[r];
        const uint32_t d = valid ? ((k >> shift) & 255u) : (uint32_t)kRadixBuckets;
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, d);
        const uint32_t rank = (uint32_t)__popc(peers & lt);
        if (rank == 0)
            s_wcnt[warp][d] = (uint32_t)__popc(peers);
        __syncthreads();
        if (valid) {
            uint32_t before = 0;
            for (int w = 0; w < warp; ++w)
                before += s_wcnt[w][d];
            const uint32_t pos = s_base[d] + before + rank;
            keys_out[pos] = k;
            vals_out[pos] = v;
        }
        __syncthreads();
        for (int dd = t; dd <= kRadixBuckets; dd += kRadixNT) {
            uint32_t sum = 0;
            for (int w = 0; w < NW; ++w) {
                sum += s_wcnt[w][dd];
                s_wcnt[w][dd] = 0;
            }
            if (dd < kRadixBuckets)
                s_base[dd] += sum;
        }
        __syncthreads();
    }
}

// Which of its two arrays radix_sort leaves the result in.
inline int radix_result(int bits) { return ((bits + 7) / 8) & 1; }

// Sorts n pairs by the low `bits` bits of their keys.  keys[0], vals[0] hold
// the input (vals[0] null: the values are 0 .. n - 1); keys[i], vals[i] are
// both written.  hist: kRadixBuckets x tiles counts, then kRadixBuckets
// totals.  Returns radix_result(bits).
inline int radix_sort(uint32_t *const keys[2], uint32_t *const vals[2], bool iota, int64_t n, int bits, uint32_t *hist,
                      cudaStream_t s)
{
    const int passes = (bits + 7) / 8;
    const int tile = kRadixNT * radix_rounds(n);
    const int32_t tiles = (int32_t)((n + tile - 1) / tile);
    const auto count = n < kRadixFew ? radix_hist_kernel<kRadixRoundsFew> : radix_hist_kernel<kRadixRounds>;
    const auto place = n < kRadixFew ? radix_scatter_kernel<kRadixRoundsFew> : radix_scatter_kernel<kRadixRounds>;
    uint32_t *digit_total = hist + (size_t)kRadixBuckets * tiles;
    int cur = 0;
    for (int p = 0; p < passes; ++p) {
        count<<<tiles, kRadixNT, 0, s>>>(keys[cur], n, 8 * p, hist, tiles);
        radix_row_scan_kernel<<<kRadixBuckets, 1024, 0, s>>>(hist, tiles, digit_total);
        radix_digit_scan_kernel<<<1, kRadixBuckets, 0, s>>>(digit_total);
        place<<<tiles, kRadixNT, 0, s>>>(keys[cur], p == 0 && iota ? nullptr : vals[cur], n, 8 * p, hist, digit_total,
                                         tiles, keys[cur ^ 1], vals[cur ^ 1]);
        cur ^= 1;
    }
    return cur;
}

// Words of radix_sort's hist for up to n pairs.
inline size_t radix_hist_words(int64_t n)
{
    auto words = [](int64_t m) {
        const int64_t tile = kRadixNT * radix_rounds(m);
        return (size_t)kRadixBuckets * (size_t)((m + tile - 1) / tile + 1);
    };
    return std::max(words(n), words(std::min(n, kRadixFew - 1)));
}

} // namespace sdm

// Sedimentation step (sdm_set_positions, sdm_sedimentation_step,
// sdm_get_positions in include/sdm.h).
//
// The paper lists particle displacement among the dynamics of its framework
// and shows sedimenting drizzle in its 2-D example; it prints no formulae.
// Reading: every live SD falls by its Rogers-Yau speed times dt, the speed
// taken from the binary32 radius twin of its volume (the KFP32 arithmetic)
// and the distance widened exactly to binary64; positions are heights above
// the bottom of the SD's cell, so a step needs no division.
//
// One step on the device, for layouts whose largest cell holds up to 1024
// slots.  Most SDs stay in their cell (over 95% per second on a cloud's
// grid), both layouts keep a cell's SDs in increasing id, and a cell receives
// from few others: so nothing is sorted as a whole.
//   sed_fall_kernel      one warp per cell: the fall; per slot its new height
//                        (negative: leaves the cell), the movers of the cell
//                        (new group, id, slot, place among the group's
//                        arrivals), the water that leaves through the bottom;
//   sed_offsets_kernel   the new cells' offsets (even) and their arrivals', the
//                        precipitated total, rounded from an exact sum;
//   sed_deal_kernel      the movers to their group's arrivals;
//   sed_merge_kernel     one warp per new cell: its arrivals sorted by id, its
//                        stayers streamed through, each moved up by the
//                        arrivals of lower id; the new layout with its padding
//                        (a cell with many arrivals: by the whole block; with
//                        over kSedRunKeys of them in one cell it leaves all as
//                        it was, and the step is taken again by the sort).
// 112 B per SD (xi, v, heights; heights out; the layout in and out).  The
// refresh of the context's own launch plan and the read-back run on a side
// stream beside the last two; the host waits for the read-back only.
// Measured on the 4.19M-SD grid (us): fall 36, offsets 11, deal 7, merge 40, where
// the sort of all SDs took 210 in all.  When every SD moves (4096 cells of 200, 500, 800
// SDs, one level per step) a step takes 53, 128, 196 us against 94, 147, 202 sorted.
//
// With larger cells (a warp would take too long), a stable sort of all SDs:
//   sed_group_kernel     where the last step went by cells: every slot's group;
//   sed_move_kernel      per slot (four per thread): the fall, the new group
//                        of every SD (the cells, then n_cells for outside the
//                        domain) as a key in SD-id order, counts per new
//                        group, the water that leaves through the bottom;
//   sed_scan_kernel      new group offsets (unpadded and padded to even
//                        slots) and the precipitated total, as above;
//   radix_sort           (sdm_radix.cuh) of the keys: per-tile digit counts, a
//                        scan of each digit's row, a scan of the digit totals,
//                        a ranked scatter;
//   sed_gather_kernel    the new layout, gathered from the old one;
//   sed_pad_kernel       its padding slots.
// The two layouts swap; the host reads the new offsets for the launch plan.
//
// Compiled as part of the library's single translation unit (included at the
// end of sdm_runtime.cu).

namespace {

constexpr int kSedNT = 256;

// ------------------------------------------------------------------ kernels
// zeta of every slot from z (SD-id order): z - (level) dz with level =
// (cbase + c) / nx, which must lie in [0, dz) (zeta_in: z already holds
// zeta); flags bit 0 and the complement of the
// first bad id on failure.  SDs outside the
// domain and padding slots get zeta 0.  A warp takes 128 slots of a group at a
// time, the ids and then the heights of all in flight together (43 us for
// 4.19M SDs one by one).
constexpr int kSedRun = 4; // times 32 slots per warp and round

__global__ void __launch_bounds__(kSedNT) sed_set_kernel(const int32_t *__restrict__ cell_off, int32_t n_cells,
                                                         int64_t n_slots, const int32_t *__restrict__ id_of_slot,
                                                         const double *__restrict__ z, int32_t nx, double dz,
                                                         int32_t cbase, int zeta_in, double *__restrict__ zeta,
                                                         uint32_t *__restrict__ flags,
                                                         unsigned long long *__restrict__ bad)
{
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int g = gw; g <= n_cells; g += nw) {
        const int64_t lo = cell_off[g], hi = g < n_cells ? cell_off[g + 1] : n_slots;
        const double base = zeta_in ? 0.0 : __dmul_rn((double)((g + cbase) / nx), dz);
        for (int64_t s0 = lo; s0 < hi; s0 += 32 * kSedRun) {
            int32_t id[kSedRun];
            double zz[kSedRun];
#pragma unroll
            for (int u = 0; u < kSedRun; ++u)
                id[u] = s0 + 32 * u + lane < hi ? id_of_slot[s0 + 32 * u + lane] : -1;
#pragma unroll
            for (int u = 0; u < kSedRun; ++u)
                zz[u] = id[u] >= 0 && g < n_cells ? z[id[u]] : 0.0;
#pragma unroll
            for (int u = 0; u < kSedRun; ++u) {
                const int64_t s = s0 + 32 * u + lane;
                if (s >= hi)
                    break;
                double zt = 0.0;
                if (id[u] >= 0 && g < n_cells) {
                    zt = zeta_in ? zz[u] : __dsub_rn(zz[u], base);
                    // a -0 height becomes +0 (the fall tests signs bitwise)
                    if (__double_as_longlong(zt) == (long long)0x8000000000000000ll)
                        zt = 0.0;
                    // in [0, dz): by the bit patterns (NaN and negative ones are above)
                    if ((unsigned long long)__double_as_longlong(zt) >= (unsigned long long)__double_as_longlong(dz)) {
                        atomicOr(flags, 1u);
                        atomicMax(bad, ~(unsigned long long)id[u]);
                        zt = 0.0;
                    }
                }
                zeta[s] = zt;
            }
        }
    }
}

// Last of the groups lo .. hi whose first slot is at or before s (lo's is).
__device__ __forceinline__ int32_t sed_group_of(const int32_t *__restrict__ cell_off, int32_t lo, int32_t hi, int64_t s)
{
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo + 1) >> 1);
        if (cell_off[mid] <= s)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// group[slot] = the slot's group, for the sorted path: a warp per kSedGroupRun times
// 32 slots, whatever the groups' sizes, as a group may hold them all (a warp per
// group took 0.43 ms for one cell of 2^22).
constexpr int kSedGroupRun = 8;
__global__ void __launch_bounds__(kSedNT) sed_group_kernel(const int32_t *__restrict__ cell_off, int32_t n_cells,
                                                           int64_t n_slots, int32_t *__restrict__ group)
{
    const int lane = threadIdx.x & 31;
    const int64_t s0 = (((int64_t)blockIdx.x * kSedNT + threadIdx.x) >> 5) * (32 * kSedGroupRun);
    if (s0 >= n_slots)
        return;
    const int64_t s1 = min(n_slots, s0 + 32 * kSedGroupRun);
    const int32_t lo = sed_group_of(cell_off, 0, n_cells, s0), hi = sed_group_of(cell_off, lo, n_cells, s1 - 1);
    for (int64_t s = s0 + lane; s < s1; s += 32)
        group[s] = sed_group_of(cell_off, lo, hi, s);
}

// z[id] = ((cbase + c) / nx) dz + zeta (0 outside) and cell[id] = c (-1
// outside).  zeta_out[id] = zeta of the slot, and gcell[id] = cbase + c
// inside, else emig[id]: the cell of another piece of the grid that the SD
// entered through this piece's bottom in the last sedimentation step, or -1
// (zeta_out then its height in that cell, else 0).
__global__ void __launch_bounds__(kSedNT) sed_get_kernel(const int32_t *__restrict__ cell_off, int32_t n_cells,
                                                         int64_t n_slots, const int32_t *__restrict__ id_of_slot,
                                                         const double *__restrict__ zeta, int32_t nx, double dz,
                                                         int32_t cbase, const int32_t *__restrict__ emig,
                                                         double *__restrict__ z, int32_t *__restrict__ cell,
                                                         double *__restrict__ zeta_out, int32_t *__restrict__ gcell)
{
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    const bool heights = z || zeta_out;
    for (int g = gw; g <= n_cells; g += nw) {
        const int64_t lo = cell_off[g], hi = g < n_cells ? cell_off[g + 1] : n_slots;
        const double base = g < n_cells && z ? __dmul_rn((double)((g + cbase) / nx), dz) : 0.0;
        for (int64_t s0 = lo; s0 < hi; s0 += 32 * kSedRun) {
            int32_t id[kSedRun];
            double zt[kSedRun];
#pragma unroll
            for (int u = 0; u < kSedRun; ++u) { // every load first
                const int64_t s = s0 + 32 * u + lane;
                id[u] = s < hi ? id_of_slot[s] : -1;
                zt[u] = s < hi && heights ? zeta[s] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < kSedRun; ++u) {
                if (id[u] < 0)
                    continue;
                if (z)
                    z[id[u]] = g < n_cells ? __dadd_rn(base, zt[u]) : 0.0;
                if (cell)
                    cell[id[u]] = g < n_cells ? g : -1;
                if (zeta_out)
                    zeta_out[id[u]] = zt[u];
                if (gcell)
                    gcell[id[u]] = g < n_cells ? g + cbase : (emig ? emig[id[u]] : -1);
            }
        }
    }
}

// The fall of every SD, four slots per thread (grid-stride, all loads
// issued before use).  key[id] = its new group (n_cells: outside), val[id]
// = its slot, zeta_new[slot] = its new height; counts[new group] (one
// atomic per run of equal groups among a warp's 32 consecutive slots);
// precip: the exact sum of xi v of the SDs that fell through the bottom of
// the grid.
// Levels are counted from the grid's bottom (cell cbase + c): an SD that
// leaves this piece's lowest level into a level of another piece becomes
// outside here, with emig[id] = its new cell there and zeta_new its height
// in it (emig[id] = -1 for every other SD).
constexpr int kSedU = 4;
constexpr int kSedMaxBlocks = 4096;

// The binary64 value of a binary32, exactly, on the integer pipe for normal
// numbers (zero, subnormals and non-finite values by the conversion).
__device__ __forceinline__ double f2d_exact(float f)
{
    const uint32_t b = __float_as_uint(f);
    const uint32_t e = (b >> 23) & 0xFFu;
    if (e == 0u || e == 0xFFu)
        return (double)f;
    return __longlong_as_double((long long)(((uint64_t)(b & 0x80000000u) << 32) | ((uint64_t)(e + 896u) << 52) |
                                            ((uint64_t)(b & 0x7FFFFFu) << 29)));
}

// x < 0 for the heights of this step (never -0: they start >= +0, and
// x - x and x + y round to +0) by the sign bit, on the integer pipe.
__device__ __forceinline__ bool dneg(double x) { return __double2hiint(x) < 0; }

// x >= y for non-negative binary64 values: their bit patterns order alike.
__device__ __forceinline__ bool dge_pos(double x, double y)
{
    return __double_as_longlong(x) >= __double_as_longlong(y);
}

// The fall of one live SD of cell g: its new cell c (negative, or another
// piece's when c + cbase < 0 ends the fall: out of the grid) and height.
struct Fall {
    int32_t c;
    double z;
};

// The height after the fall (negative: below the cell's bottom).
__device__ __forceinline__ double sed_drop(const PairConsts &C, double v, double zt, float dt32)
{
    bool in_range;
    const float vf = d2f_rn(v, in_range);
    return __dsub_rn(zt, f2d_exact(__fmul_rn(vt32c(C, radius32(vf)), dt32)));
}

__device__ __forceinline__ Fall sed_levels(double zz, int32_t g, int32_t nx, double dz, int32_t cbase)
{
    // crossing k levels takes cell c to c - k nx; below the grid's level 0
    // exactly when cbase + c is negative (0 <= column < nx)
    int32_t c = g;
    while (dneg(zz)) { // at most as many levels as the SD falls through
        c -= nx;
        if (c + cbase < 0)
            return Fall{c, 0.0};
        zz = __dadd_rn(zz, dz);
    }
    if (dge_pos(zz, dz)) { // zeta + dz rounded up to dz: on the boundary, level above
        c += nx;
        zz = 0.0;
    }
    return Fall{c, zz};
}

__device__ __forceinline__ Fall sed_fall(const PairConsts &C, double v, double zt, float dt32, int32_t g, int32_t nx,
                                         double dz, int32_t cbase)
{
    return sed_levels(sed_drop(C, v, zt, dt32), g, nx, dz, cbase);
}

// The precipitated water: an exact sum, so that it depends neither on the order
// of its terms nor on the path that takes the step.  A term xi v is an integer
// in units of 2^-1074, added as digits of 32 bits to signed 64-bit bins (bin i
// weighs 2^(32 i - 1074); 2^31 terms fit), and the sum of all is rounded once.
// (In binary64, as it was, a term took the narrow pipe's additions: a step in
// which all of 16,384 cells of 256 fall out 254 us, 237 now.)
constexpr int kExactBins = 72;
typedef unsigned long long ExactBin; // two's complement

// Adds xi v of the lanes with `on` (all lanes of the warp call it).  Lanes whose
// digits lie in the same bins, with the same sign, share their additions.
__device__ __noinline__ void exact_add(ExactBin *bins, bool on, int64_t xi, double v)
{
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    const uint64_t bits = (uint64_t)__double_as_longlong(v);
    const uint32_t e = (uint32_t)(bits >> 52) & 0x7FFu;
    const uint64_t m = (bits & 0xFFFFFFFFFFFFFull) | (e ? 1ull << 52 : 0ull);
    const uint32_t at = e ? e - 1u : 0u, sh = at & 31u; // the last place of v weighs 2^(at - 1074)
    const uint64_t lo = (uint64_t)xi * m, hi = __umul64hi((uint64_t)xi, m);
    const uint64_t w0 = lo << sh, w1 = (hi << sh) | (sh ? lo >> (64u - sh) : 0ull), w2 = sh ? hi >> (64u - sh) : 0ull;
    const uint32_t digit[5] = {(uint32_t)w0, (uint32_t)(w0 >> 32), (uint32_t)w1, (uint32_t)(w1 >> 32), (uint32_t)w2};
    const uint32_t group = (at >> 5) | (uint32_t)(bits >> 63) << 8;
    for (unsigned todo = __ballot_sync(FULL, on); todo;) {
        const uint32_t g = __shfl_sync(FULL, group, __ffs(todo) - 1);
        const bool mine = on && group == g;
        ExactBin sum = 0;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const uint32_t d = mine ? digit[k] : 0u;
            const uint32_t low = __reduce_add_sync(FULL, d & 0xFFFFu), high = __reduce_add_sync(FULL, d >> 16);
            if (lane == k)
                sum = ((ExactBin)high << 16) + low;
        }
        if (lane < 5 && sum)
            atomicAdd(&bins[(g & 0xFFu) + lane], g >> 8 ? 0ull - sum : sum);
        todo &= ~__ballot_sync(FULL, mine);
    }
}

// The block's bins, zero before use (a barrier between), and into the sum of all blocks.
__device__ __forceinline__ void exact_clear(ExactBin *bins)
{
    for (int i = threadIdx.x; i < kExactBins; i += blockDim.x)
        bins[i] = 0ull;
}

__device__ __forceinline__ void exact_flush(const ExactBin *bins, ExactBin *total)
{
    __syncthreads();
    for (int i = threadIdx.x; i < kExactBins; i += blockDim.x)
        if (bins[i])
            atomicAdd(&total[i], bins[i]);
}

// *out = the sum rounded to nearest even; total is zero again (one warp).
__device__ __forceinline__ void exact_round(ExactBin *total, double *out)
{
    __shared__ uint32_t s_digit[kExactBins];
    __shared__ long long s_bin[kExactBins];
    const int lane = threadIdx.x & 31;
    int first = kExactBins, last = -1;
    for (int i = lane; i < kExactBins; i += 32) {
        const ExactBin b = total[i];
        s_bin[i] = (long long)b;
        s_digit[i] = 0u;
        if (b) {
            total[i] = 0ull;
            first = min(first, i);
            last = i;
        }
    }
    first = __reduce_min_sync(0xFFFFFFFFu, first);
    last = __reduce_max_sync(0xFFFFFFFFu, last);
    __syncwarp();
    if (lane != 0)
        return;
    bool minus = false;
    long long carry = 0;
    int end = kExactBins;
    for (int pass = 0; pass < 2; ++pass) { // a negative sum's digits in the second, of its negative
        carry = 0;
        for (int i = first; i < kExactBins && (i <= last || carry != 0); ++i) {
            carry += minus ? -s_bin[i] : s_bin[i];
            s_digit[i] = (uint32_t)carry;
            carry >>= 32;
            end = i + 1;
            if (i > last && carry == -1 && s_digit[i] == 0xFFFFFFFFu)
                break; // the sign, from here up
        }
        if (carry >= 0)
            break;
        minus = true;
    }
    int t = end - 1;
    while (t >= first && s_digit[t] == 0u)
        --t;
    if (t < first) {
        *out = 0.0;
        return;
    }
    const uint32_t d2 = s_digit[t], d1 = t > 0 ? s_digit[t - 1] : 0u, d0 = t > 1 ? s_digit[t - 2] : 0u;
    const int lz = __clz((int)d2);
    uint64_t n = (uint64_t)d2 << 32 | d1;
    n = lz ? (n << lz) | (d0 >> (32 - lz)) : n;
    bool below = (lz ? d0 << lz : d0) != 0u;
    for (int i = first; i < t - 2; ++i)
        below |= s_digit[i] != 0u;
    const int w = 32 * (t - 1) - lz - 1074; // the sum is n 2^w and a little
    double r;
    if (w + 1085 >= 1 && w + 1085 <= 2045)
        r = u64_to_double(n, below, w);
    else // the ends of the range, which no volume of water comes near
        r = ldexp(__ull2double_rn(n), w);
    *out = minus ? -r : r;
}

__global__ void __launch_bounds__(kSedNT) sed_move_kernel(const InstDev *__restrict__ P, int32_t n_cells, int64_t n_slots,
                                                          int32_t nx, double dz, float dt32,
                                                          const double *__restrict__ zeta,
                                                          const int32_t *__restrict__ group,
                                                          const int32_t *__restrict__ id_of_slot,
                                                          uint32_t *__restrict__ key, uint32_t *__restrict__ val,
                                                          double *__restrict__ zeta_new, uint32_t *__restrict__ counts,
                                                          ExactBin *__restrict__ precip, int32_t cbase,
                                                          int32_t *__restrict__ emig)
{
    constexpr unsigned FULL = 0xFFFFFFFFu;
    __shared__ ExactBin s_precip[kExactBins];
    exact_clear(s_precip);
    __syncthreads();
    const PairConsts C = pair_consts(P);
    const int lane = threadIdx.x & 31;
    const int64_t *__restrict__ gxi = P->xi;
    const double *__restrict__ gv = P->v;
    const int64_t stride = (int64_t)gridDim.x * kSedNT;
    // warp-uniform trip count: every lane runs every round (shuffles, ballots)
    for (int64_t w0 = ((int64_t)blockIdx.x * kSedNT + (threadIdx.x & ~31)); w0 < n_slots; w0 += kSedU * stride) {
        int32_t id[kSedU], g[kSedU];
        int64_t x[kSedU];
        double vv[kSedU], zt[kSedU];
#pragma unroll
        for (int u = 0; u < kSedU; ++u) {
            const int64_t sl = w0 + u * stride + lane;
            const bool in = sl < n_slots;
            id[u] = in ? id_of_slot[sl] : -1;
            g[u] = in ? group[sl] : 0;
            x[u] = in ? gxi[sl] : 0;
            vv[u] = in ? gv[sl] : 1.0;
            zt[u] = in ? zeta[sl] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kSedU; ++u) {
            const int64_t sl = w0 + u * stride + lane;
            int32_t ng = -1; // -1: no SD in this slot
            bool fell = false;
            if (id[u] >= 0) {
                double zn = 0.0;
                int32_t em = -1;
                ng = n_cells;
                if (g[u] < n_cells && x[u] > 0) {
                    const Fall f = sed_fall(C, vv[u], zt[u], dt32, g[u], nx, dz, cbase);
                    if (f.c + cbase < 0) {
                        fell = true;
                    } else {
                        zn = f.z;
                        if (f.c >= 0)
                            ng = f.c;
                        else // into another piece of the grid
                            em = f.c + cbase;
                    }
                }
                key[id[u]] = (uint32_t)ng;
                val[id[u]] = (uint32_t)sl;
                zeta_new[sl] = zn;
                emig[id[u]] = em;
            }
            if (__any_sync(FULL, fell))
                exact_add(s_precip, fell, x[u], vv[u]);
            const int32_t nxt = __shfl_down_sync(FULL, ng, 1);
            const bool end = lane == 31 || nxt != ng;
            const unsigned ends = __ballot_sync(FULL, end);
            if (end && ng >= 0) {
                const unsigned below = ends & ((1u << lane) - 1u);
                const int start = below ? 32 - __clz(below) : 0;
                atomicAdd(&counts[ng], (uint32_t)(lane - start + 1));
            }
        }
    }
    exact_flush(s_precip, precip);
}

// One block: ustart = exclusive scan of counts[0 .. n_groups) (total at
// ustart[n_groups]); poff the same with every count rounded up to even;
// *precip_total = the rounded sum of the bins.  Both scans
// run at once on packed 64-bit sums (unpadded below, padded above: neither
// exceeds 2^31), 8 consecutive groups per thread, tiles of 8192 groups.
__global__ void __launch_bounds__(1024) sed_scan_kernel(const uint32_t *__restrict__ counts, int32_t n_groups,
                                                        int32_t *__restrict__ ustart, int32_t *__restrict__ poff,
                                                        ExactBin *__restrict__ precip,
                                                        double *__restrict__ precip_total)
{
    constexpr int E = 8, TILE = 1024 * E;
    __shared__ uint32_t s_c[TILE];
    __shared__ unsigned long long s_w[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    unsigned long long carry = 0;
    for (int32_t g0 = 0; g0 < n_groups; g0 += TILE) {
        {
            uint32_t c[E]; // the tile's loads all in flight at once
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int i = t + e * 1024;
                c[e] = g0 + i < n_groups ? counts[g0 + i] : 0u;
            }
#pragma unroll
            for (int e = 0; e < E; ++e)
                s_c[t + e * 1024] = c[e];
        }
        __syncthreads();
        unsigned long long v[E], sum = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t c = s_c[t * E + e];
            v[e] = (unsigned long long)c | ((unsigned long long)((c + 1u) & ~1u) << 32);
            sum += v[e];
        }
        unsigned long long x = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x, d);
            if (lane >= d)
                x += y;
        }
        if (lane == 31)
            s_w[warp] = x;
        __syncthreads();
        if (warp == 0) {
            unsigned long long w = s_w[lane];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, w, d);
                if (lane >= d)
                    w += y;
            }
            s_w[lane] = w; // inclusive totals of warps 0 .. lane
        }
        __syncthreads();
        // the two results through shared memory, so that the writes to
        // global memory are coalesced (consecutive threads, consecutive groups)
        const unsigned long long base0 = carry + (warp > 0 ? s_w[warp - 1] : 0ull) + x - sum;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            unsigned long long base = base0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                s_c[t * E + e] = (uint32_t)(half ? base >> 32 : base);
                base += v[e];
            }
            __syncthreads();
            int32_t *out = half ? poff : ustart;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int32_t g = g0 + t + e * 1024;
                if (g < n_groups)
                    out[g] = (int32_t)s_c[t + e * 1024];
            }
            __syncthreads();
        }
        carry += s_w[31];
    }
    if (t == 0) {
        ustart[n_groups] = (int32_t)(uint32_t)carry;
        poff[n_groups] = (int32_t)(uint32_t)(carry >> 32);
    }
    if (warp == 0)
        exact_round(precip, precip_total);
}

// The new layout: the j-th SD in (group, id) order goes to slot
// poff[g] + (j - ustart[g]).
__global__ void sed_gather_kernel(int64_t n_sd, const uint32_t *__restrict__ keys, const uint32_t *__restrict__ vals,
                                  const int32_t *__restrict__ ustart, const int32_t *__restrict__ poff,
                                  const int64_t *__restrict__ xi, const double *__restrict__ v,
                                  const double *__restrict__ zeta_new, const int32_t *__restrict__ id_of_slot,
                                  int64_t *__restrict__ xi2, double *__restrict__ v2, double *__restrict__ zeta2,
                                  int32_t *__restrict__ id2, int32_t *__restrict__ group2)
{
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n_sd; j += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t g = keys[j], s = vals[j];
        const int64_t p = poff[g] + (j - ustart[g]);
        xi2[p] = xi[s];
        v2[p] = v[s];
        zeta2[p] = zeta_new[s];
        id2[p] = id_of_slot[s];
        group2[p] = (int32_t)g;
    }
}

// The padding slot after every odd group of the new layout.
__global__ void sed_pad_kernel(int32_t n_groups, const int32_t *__restrict__ ustart, const int32_t *__restrict__ poff,
                               int64_t *__restrict__ xi2, double *__restrict__ v2, double *__restrict__ zeta2,
                               int32_t *__restrict__ id2, int32_t *__restrict__ group2)
{
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n_groups; g += gridDim.x * blockDim.x) {
        for (int32_t p = poff[g] + (ustart[g + 1] - ustart[g]); p < poff[g + 1]; ++p) {
            xi2[p] = 0;
            v2[p] = 1.0;
            zeta2[p] = 0.0;
            id2[p] = -1;
            group2[p] = g;
        }
    }
}

// ------------------------------------------------- cells of up to kSedByCell
constexpr int kSedByCell = 1024;  // slots of the largest cell that a warp takes
constexpr int kSedFewCells = 608, kSedFewLargest = 800; // sdm_sedimentation_step's rule for few cells
constexpr int kSedArrive = 256;   // arrivals of a cell that a warp takes; more by its block
constexpr int kSedMergeNT = 128;
constexpr int kSedRunKeys = kSedArrive * (kSedMergeNT / 32); // arrivals of a cell that a block takes
constexpr int kSedFew = 12;       // arrivals up to which each is compared with every stayer, by ballots

// What the movers of the cells and the arrivals of the groups are kept in.
// Cell c's movers take places [cell_off[c], + left[c]) of the mover arrays;
// group g's arrivals [first[g], + arr[g]) of the arrival arrays.
struct SedMoves {
    uint32_t *group, *id, *slot, *place; // per mover: new group, id, slot, place among the group's arrivals
    uint32_t *a_id, *a_slot;             // per arrival
    uint32_t *stay, *arr, *left;         // per group: SDs that stay; per cell: SDs that arrive, movers
    uint32_t *out, *out_next;            // SDs that arrive outside the domain; the next step's count
    int32_t *first;                      // n_groups
    uint32_t *moved, *piled; // how many SDs move; whether a cell receives more than kSedRunKeys
};

// A warp first takes every SD's height down; the few that leave their cell (or
// are dead, or padding) wait in shared memory and are followed 32 at a time, so
// that their levels, each a binary64 addition, and their places are not paid by
// every 32 slots that hold one.
constexpr int kSedWait = 64; // entries: below 32 left from before, and up to 32 new ones

__global__ void __launch_bounds__(kSedNT) sed_fall_kernel(const InstDev *__restrict__ P,
                                                          const int32_t *__restrict__ cell_off, int32_t n_cells,
                                                          int64_t n_slots, int32_t nx, double dz, float dt32,
                                                          const double *__restrict__ zeta,
                                                          const int32_t *__restrict__ id_of_slot,
                                                          double *__restrict__ zeta_new, SedMoves M,
                                                          ExactBin *__restrict__ precip, int32_t cbase,
                                                          int32_t *__restrict__ emig)
{
    constexpr unsigned FULL = 0xFFFFFFFFu;
    __shared__ ExactBin s_precip[kExactBins];
    exact_clear(s_precip);
    __syncthreads();
    __shared__ double s_z[kSedNT / 32][kSedWait];
    __shared__ int32_t s_slot[kSedNT / 32][kSedWait]; // with the sign bit for an SD that does not fall (dead, padding)
    const PairConsts C = pair_consts(P);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t *__restrict__ gxi = P->xi;
    const double *__restrict__ gv = P->v;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int g = gw; g < n_cells; g += nw) { // uniform over the warp
        const int32_t lo = cell_off[g], hi = cell_off[g + 1];
        uint32_t stay = 0, left = 0, wait = 0; // uniform
        auto follow = [&](uint32_t n) {        // the first n <= 32 waiting entries
            int32_t ng = n_cells, em = -1, id = -1, sl = 0;
            double zn = 0.0;
            bool fell = false;
            if (lane < (int)n) {
                const int32_t e = s_slot[warp][lane];
                sl = e & 0x7FFFFFFF;
                id = id_of_slot[sl];
                if (e >= 0) {
                    const Fall f = sed_levels(s_z[warp][lane], g, nx, dz, cbase);
                    if (f.c + cbase < 0) {
                        fell = true;
                    } else {
                        zn = f.z;
                        if (f.c >= 0)
                            ng = f.c;
                        else // into another piece of the grid
                            em = f.c + cbase;
                    }
                }
            }
            if (__any_sync(FULL, fell))
                exact_add(s_precip, fell, fell ? gxi[sl] : 0, fell ? gv[sl] : 0.0);
            // (level 0 dz above: zeta + dz rounded up to dz, so it stays after all)
            const bool keep = lane < (int)n && ng == g;
            stay += (uint32_t)__popc(__ballot_sync(FULL, keep));
            if (lane < (int)n) // stayers +zn, the others (padding too) with the sign bit set
                zeta_new[sl] = keep ? zn : __hiloint2double(__double2hiint(zn) | (int)0x80000000, __double2loint(zn));
            const bool go = id >= 0 && !keep;
            const unsigned mv = __ballot_sync(FULL, go);
            const unsigned out = __ballot_sync(FULL, go && ng == n_cells);
            uint32_t place = 0;
            if (out && lane == __ffs(out) - 1) // one counter for all that leave the domain
                place = atomicAdd(M.out, (uint32_t)__popc(out));
            place = __shfl_sync(FULL, place, out ? __ffs(out) - 1 : 0) + (uint32_t)__popc(out & lt);
            // one addition per group among the lanes (in heavy rain all 32 enter the same cell)
            const bool in = go && ng != n_cells;
            const unsigned same = __match_any_sync(FULL, in ? ng : -1 - lane);
            const int head = __ffs(same) - 1;
            uint32_t first = 0;
            if (in && lane == head)
                first = atomicAdd(&M.arr[ng], (uint32_t)__popc(same));
            first = __shfl_sync(FULL, first, head);
            if (go) {
                if (in)
                    place = first + (uint32_t)__popc(same & lt);
                const uint32_t at = (uint32_t)lo + left + (uint32_t)__popc(mv & lt);
                M.group[at] = (uint32_t)ng;
                M.id[at] = (uint32_t)id;
                M.slot[at] = (uint32_t)sl;
                M.place[at] = place;
                if (em >= 0)
                    emig[id] = em;
            }
            left += (uint32_t)__popc(mv);
        };
        for (int32_t s0 = lo; s0 < hi; s0 += 32 * kSedRun) {
            int64_t x[kSedRun];
            double vv[kSedRun], zt[kSedRun];
#pragma unroll
            for (int u = 0; u < kSedRun; ++u) { // every load first
                const int32_t sl = s0 + 32 * u + lane;
                const bool in = sl < hi;
                x[u] = in ? gxi[sl] : 0;
                vv[u] = in ? gv[sl] : 1.0;
                zt[u] = in ? zeta[sl] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < kSedRun; ++u) {
                if (s0 + 32 * u >= hi) // uniform over the warp
                    break;
                const int32_t sl = s0 + 32 * u + lane;
                const double zz = sed_drop(C, vv[u], zt[u], dt32);
                const bool keep = x[u] > 0 && !dneg(zz);
                const unsigned km = __ballot_sync(FULL, keep), wm = __ballot_sync(FULL, sl < hi) & ~km;
                stay += (uint32_t)__popc(km);
                if (keep) {
                    zeta_new[sl] = zz;
                } else if (sl < hi) {
                    const uint32_t at = wait + (uint32_t)__popc(wm & lt);
                    s_z[warp][at] = zz;
                    s_slot[warp][at] = sl | (x[u] > 0 ? 0 : (int32_t)0x80000000);
                }
                wait += (uint32_t)__popc(wm);
                if (wait >= 32u) {
                    __syncwarp();
                    follow(32u);
                    __syncwarp();
                    wait -= 32u;
                    if (lane < (int)wait) { // the rest to the front
                        s_z[warp][lane] = s_z[warp][32 + lane];
                        s_slot[warp][lane] = s_slot[warp][32 + lane];
                    }
                    __syncwarp();
                }
            }
        }
        __syncwarp();
        if (wait)
            follow(wait);
        __syncwarp();
        if (lane == 0) {
            M.stay[g] = stay;
            M.left[g] = left;
        }
    }
    if (gw == 0 && lane == 0) { // those outside stay there (their last slot may be padding)
        *M.piled = 0u;
        const int32_t lo = cell_off[n_cells];
        M.stay[n_cells] = (uint32_t)(n_slots - lo) - (n_slots > lo && id_of_slot[n_slots - 1] < 0 ? 1u : 0u);
    }
    exact_flush(s_precip, precip);
}

// Sums over the groups of a block of 1024, for sed_offsets_kernel over many.
__device__ __forceinline__ unsigned long long sed_sizes(const SedMoves &M, int g, int n_groups)
{
    const uint32_t a = g == n_groups - 1 ? *M.out : M.arr[g];
    return (unsigned long long)((M.stay[g] + a + 1u) & ~1u) | ((unsigned long long)a << 32);
}

__device__ __forceinline__ unsigned long long sed_block_sum(unsigned long long x, unsigned long long *s_w)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1)
        x += __shfl_down_sync(0xFFFFFFFFu, x, d);
    if ((threadIdx.x & 31) == 0)
        s_w[threadIdx.x >> 5] = x;
    __syncthreads();
    unsigned long long t = s_w[threadIdx.x & 31];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1)
        t += __shfl_xor_sync(0xFFFFFFFFu, t, d);
    __syncthreads();
    return t;
}

__global__ void __launch_bounds__(1024) sed_totals_kernel(SedMoves M, int32_t n_groups,
                                                          unsigned long long *__restrict__ totals)
{
    __shared__ unsigned long long s_w[32];
    const int g = blockIdx.x * 1024 + threadIdx.x;
    const unsigned long long t = sed_block_sum(g < n_groups ? sed_sizes(M, g, n_groups) : 0ull, s_w);
    if (threadIdx.x == 0)
        totals[blockIdx.x] = t;
}

// poff[g] = first slot of group g (every group an even number), M.first[g] =
// its first arrival; block 0 also rounds the precipitated water.  The groups
// before a block are summed by the block itself (up to 64 blocks: totals
// null), or their blocks' totals.
__global__ void __launch_bounds__(1024) sed_offsets_kernel(SedMoves M, int32_t n_groups,
                                                           const unsigned long long *__restrict__ totals,
                                                           int32_t *__restrict__ poff,
                                                           ExactBin *__restrict__ precip,
                                                           double *__restrict__ precip_total)
{
    __shared__ unsigned long long s_w[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int g = blockIdx.x * 1024 + t;
    unsigned long long before = 0;
    if (totals)
        for (int i = t; i < (int)blockIdx.x; i += 1024)
            before += totals[i];
    else
        for (int i = t; i < (int)blockIdx.x * 1024; i += 4 * 1024) { // four loads in flight
            unsigned long long q[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                q[u] = i + u * 1024 < (int)blockIdx.x * 1024 ? sed_sizes(M, i + u * 1024, n_groups) : 0ull;
            before += (q[0] + q[1]) + (q[2] + q[3]);
        }
    const unsigned long long mine = g < n_groups ? sed_sizes(M, g, n_groups) : 0ull;
    before = sed_block_sum(before, s_w);
    unsigned long long x = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x, d);
        if (lane >= d)
            x += y;
    }
    if (lane == 31)
        s_w[warp] = x;
    __syncthreads();
    unsigned long long w = lane < warp ? s_w[lane] : 0ull;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1)
        w += __shfl_xor_sync(0xFFFFFFFFu, w, d);
    const unsigned long long at = before + w + x - mine;
    if (g < n_groups) {
        poff[g] = (int32_t)(uint32_t)at;
        M.first[g] = (int32_t)(uint32_t)(at >> 32);
        if (g == n_groups - 1)
            poff[n_groups] = (int32_t)(uint32_t)(at + mine);
    }
    if (g < n_groups - 1 && M.arr[g] > (uint32_t)kSedRunKeys)
        *M.piled = 1u;
    if (g == n_groups - 1)
        *M.moved = (uint32_t)((at + mine) >> 32);
    if (blockIdx.x == 0 && warp == 0)
        exact_round(precip, precip_total);
}

__global__ void __launch_bounds__(kSedNT) sed_deal_kernel(const int32_t *__restrict__ cell_off, int32_t n_cells,
                                                          SedMoves M)
{
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int g = gw; g < n_cells; g += nw) {
        const uint32_t lo = (uint32_t)cell_off[g], n = M.left[g];
        for (uint32_t i = lane; i < n; i += 32) {
            const uint32_t at = (uint32_t)M.first[M.group[lo + i]] + M.place[lo + i];
            M.a_id[at] = M.id[lo + i];
            M.a_slot[at] = M.slot[lo + i];
        }
    }
}

// A layout's arrays.
struct SedLayout {
    int64_t *xi;
    double *v, *zeta;
    int32_t *id;
    __device__ __forceinline__ void put(int64_t p, int64_t x, double w, double z, int32_t i) const
    {
        xi[p] = x;
        v[p] = w;
        zeta[p] = z;
        id[p] = i;
    }
};

// First place in the n ascending numbers at or above x.
template <typename F>
__device__ __forceinline__ uint32_t sed_lower(uint32_t n, uint32_t x, F &&at)
{
    uint32_t lo = 0;
    while (lo < n) {
        const uint32_t mid = (lo + n) >> 1;
        if (at(mid) < x)
            lo = mid + 1;
        else
            n = mid;
    }
    return lo;
}

// A cell with more than kSedArrive arrivals, by the whole block: the arrivals
// sorted, the stayers' ids and counts in shared memory, every SD's place by
// binary searches.  (By one warp that counted: 2.5 ms for 4096 cells of 1000 SDs
// of which 600 fall into the next cell, 0.10 here.)
struct SedHeavy {
    uint32_t id[kSedByCell];
    uint16_t stay[kSedByCell + 2]; // stayers before a slot
    uint32_t warp[kSedMergeNT / 32];
};

__device__ __noinline__ void sed_merge_heavy(int g, const int32_t *__restrict__ cell_off, SedMoves M,
                                             const int64_t *__restrict__ xi, const double *__restrict__ v,
                                             const double *__restrict__ zeta_new,
                                             const int32_t *__restrict__ id_of_slot, const int32_t *__restrict__ poff,
                                             SedLayout L, unsigned long long *key, SedHeavy &H)
{
    constexpr int E = kSedByCell / kSedMergeNT; // slots per thread
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int32_t lo = cell_off[g], p0 = poff[g], p1 = poff[g + 1];
    const uint32_t n = (uint32_t)(cell_off[g + 1] - lo), A = M.arr[g], a0 = (uint32_t)M.first[g];
    uint32_t keep = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t i = (uint32_t)(t * E + e);
        H.id[i] = i < n ? (uint32_t)id_of_slot[lo + i] : 0xFFFFFFFFu; // (padding: -1, above all)
        keep |= (i < n && !dneg(zeta_new[lo + i]) ? 1u : 0u) << e;
    }
    uint32_t incl = (uint32_t)__popc(keep);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d)
            incl += y;
    }
    if (lane == 31)
        H.warp[warp] = incl;
    __syncthreads();
    uint32_t before = incl - (uint32_t)__popc(keep), n_stay = 0;
    for (int w = 0; w < kSedMergeNT / 32; ++w) {
        before += w < warp ? H.warp[w] : 0u;
        n_stay += H.warp[w];
    }
#pragma unroll
    for (int e = 0; e < E; ++e)
        H.stay[t * E + e] = (uint16_t)(before + (uint32_t)__popc(keep & ((1u << e) - 1u)));
    if (t == 0)
        H.stay[kSedByCell] = (uint16_t)n_stay;
    uint32_t P2 = 1;
    while (P2 < A)
        P2 <<= 1;
    for (uint32_t i = t; i < P2; i += kSedMergeNT)
        key[i] = i < A ? ((unsigned long long)M.a_id[a0 + i] << 32) | M.a_slot[a0 + i] : ~0ull;
    __syncthreads();
    bool back = false; // those of one cell come in order
    for (uint32_t i = t; i + 1 < A; i += kSedMergeNT)
        back |= key[i] > key[i + 1];
    for (uint32_t k = __syncthreads_or(back) ? 2u : 2u * P2; k <= P2; k <<= 1) // bitonic
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t i = t; i < P2 / 2; i += kSedMergeNT) {
                const uint32_t a = 2 * i - (i & (j - 1)), b = a + j;
                const unsigned long long ka = key[a], kb = key[b];
                if ((ka > kb) == ((a & k) == 0)) {
                    key[a] = kb;
                    key[b] = ka;
                }
            }
            __syncthreads();
        }
    auto arrivals_below = [&](uint32_t id) {
        return sed_lower(A, id, [&](uint32_t i) { return (uint32_t)(key[i] >> 32); });
    };
    for (uint32_t i = t; i < n; i += kSedMergeNT) {
        const double z = zeta_new[lo + i];
        if (!dneg(z))
            L.put((int64_t)p0 + H.stay[i] + arrivals_below(H.id[i]), xi[lo + i], v[lo + i], z, (int32_t)H.id[i]);
    }
    for (uint32_t j = t; j < A; j += kSedMergeNT) {
        const uint32_t id = (uint32_t)(key[j] >> 32), slot = (uint32_t)key[j];
        const uint32_t at = j + H.stay[sed_lower(n, id, [&](uint32_t i) { return H.id[i]; })];
        L.put((int64_t)p0 + at, xi[slot], v[slot], fabs(zeta_new[slot]), (int32_t)id);
    }
    __syncthreads(); // the shared arrays and the count are read
    if (t == 0) {
        if (p0 + (int32_t)(n_stay + A) < p1) // the padding slot of an odd cell
            L.put(p1 - 1, 0, 1.0, 0.0, -1);
        M.arr[g] = 0u; // for the next step
    }
}

// Nine blocks per SM (56 registers): with eight (64) a step of the 4.19M-SD grid takes
// 4.7 us more.
__global__ void __launch_bounds__(kSedMergeNT, 9) sed_merge_kernel(const int32_t *__restrict__ cell_off, int32_t n_cells,
                                                                SedMoves M, const int64_t *__restrict__ xi,
                                                                const double *__restrict__ v,
                                                                const double *__restrict__ zeta_new,
                                                                const int32_t *__restrict__ id_of_slot,
                                                                const int32_t *__restrict__ poff, SedLayout L,
                                                                InstDev *__restrict__ rec, int64_t step)
{
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr int W = kSedMergeNT / 32;
    __shared__ unsigned long long s_key[W][kSedArrive]; // arrivals: id above slot, in order
    __shared__ union {
        uint32_t below[W][kSedArrive]; // stayers that follow t arrivals and no more
        SedHeavy heavy;
    } s_u;
    static_assert(kSedByCell % kSedMergeNT == 0 && kSedRunKeys == W * kSedArrive, "the block's arrays");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    unsigned long long *key = s_key[warp];
    uint32_t *below = s_u.below[warp];
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    // a cell's numbers, one per lane, loaded a cell ahead
    auto numbers = [&](int g) -> uint32_t {
        if (lane == 7) // (the same for every cell)
            return *M.piled;
        if (g >= n_cells || lane > 6)
            return 0u;
        if (lane < 4)
            return (uint32_t)(lane < 2 ? cell_off : poff)[g + (lane & 1)];
        return lane == 4 ? M.arr[g] : (lane == 5 ? (uint32_t)M.first[g] : M.stay[g]);
    };
    uint32_t ahead = numbers(gw);
    if (__syncthreads_or(lane == 7 && ahead != 0u)) { // taken again by the sort: the counts are made ready, no more
        for (int g = gw; g < n_cells; g += nw)
            if (lane == 0)
                M.arr[g] = 0u;
        if (blockIdx.x == 0 && threadIdx.x == 0)
            *M.out_next = 0u;
        return;
    }
    int heavy = 0;
    for (int g = gw; g < n_cells; g += nw) { // uniform over the warp
        const int32_t lo = __shfl_sync(FULL, ahead, 0), hi = __shfl_sync(FULL, ahead, 1);
        const int32_t p0 = __shfl_sync(FULL, ahead, 2), p1 = __shfl_sync(FULL, ahead, 3);
        const uint32_t A = __shfl_sync(FULL, ahead, 4), a0 = __shfl_sync(FULL, ahead, 5);
        const uint32_t n_stay = __shfl_sync(FULL, ahead, 6);
        ahead = numbers(g + nw);
        if (A > (uint32_t)kSedArrive) { // later, by the block
            heavy = 1;
            continue;
        }
        int64_t x[kSedRun];
        double w[kSedRun], z[kSedRun];
        int32_t id[kSedRun];
        auto fetch = [&](int32_t s0) { // 128 slots, every load together
#pragma unroll
            for (int u = 0; u < kSedRun; ++u) {
                const int32_t sl = s0 + 32 * u + lane;
                const bool in = sl < hi;
                z[u] = in ? zeta_new[sl] : -1.0;
                x[u] = in ? xi[sl] : 0;
                w[u] = in ? v[sl] : 1.0;
                id[u] = in ? id_of_slot[sl] : -1;
            }
        };
        fetch(lo); // on its way while the arrivals are sorted
        if (A > 0) {
            uint32_t P2 = 1;
            while (P2 < A)
                P2 <<= 1;
            for (uint32_t i = lane; i < P2; i += 32) {
                key[i] = i < A ? ((unsigned long long)M.a_id[a0 + i] << 32) | M.a_slot[a0 + i] : ~0ull;
                below[i] = 0u;
            }
            __syncwarp();
            bool back = false; // those of one cell come in order
            for (uint32_t i = lane; i + 1 < A; i += 32)
                back |= key[i] > key[i + 1];
            for (uint32_t k = __any_sync(FULL, back) ? 2u : 2u * P2; k <= P2; k <<= 1) // bitonic
                for (uint32_t j = k >> 1; j > 0; j >>= 1) {
                    for (uint32_t i = lane; i < P2 / 2; i += 32) {
                        const uint32_t a = 2 * i - (i & (j - 1)), b = a + j;
                        const unsigned long long ka = key[a], kb = key[b];
                        if ((ka > kb) == ((a & k) == 0)) {
                            key[a] = kb;
                            key[b] = ka;
                        }
                    }
                    __syncwarp();
                }
        }
        uint32_t done = 0; // stayers so far
        uint32_t mine = 0;
        for (int32_t s0 = lo; s0 < hi; s0 += 32 * kSedRun) {
#pragma unroll
            for (int u = 0; u < kSedRun; ++u) {
                if (s0 + 32 * u >= hi) // uniform over the warp
                    break;
                const bool keep = !dneg(z[u]);
                const unsigned km = __ballot_sync(FULL, keep);
                uint32_t t = 0; // arrivals of lower id
                if (A <= (uint32_t)kSedFew) {
                    for (uint32_t k = 0; k < A; ++k) {
                        const bool above = keep && (uint32_t)(key[k] >> 32) < (uint32_t)id[u];
                        t += above ? 1u : 0u;
                        const uint32_t c = (uint32_t)__popc(km & ~__ballot_sync(FULL, above));
                        mine += lane == (int)k ? c : 0u; // lane k: stayers of lower id than arrival k
                    }
                } else {
                    uint32_t end = A;
                    while (t < end) { // first arrival above this id
                        const uint32_t mid = (t + end) >> 1;
                        if ((uint32_t)(key[mid] >> 32) < (uint32_t)id[u])
                            t = mid + 1;
                        else
                            end = mid;
                    }
                    // stayers before each arrival: t does not fall along the kept lanes, one
                    // addition per run of equal t (those after the last need none)
                    const unsigned same = __match_any_sync(FULL, keep ? t : 0xFFFFFFFFu);
                    if (keep && t < A && (same & lt) == 0u)
                        below[t] += (uint32_t)__popc(same);
                    __syncwarp();
                }
                if (keep)
                    L.put((int64_t)p0 + done + (uint32_t)__popc(km & lt) + t, x[u], w[u], z[u], id[u]);
                done += (uint32_t)__popc(km);
            }
            if (s0 + 32 * kSedRun < hi)
                fetch(s0 + 32 * kSedRun);
        }
        uint32_t carry = 0; // stayers before the arrivals of this round
        for (uint32_t j0 = 0; j0 < A; j0 += 32) {
            const uint32_t j = j0 + lane;
            uint32_t slot = 0, id_a = 0, at = 0;
            if (A <= (uint32_t)kSedFew) {
                if (j < A) {
                    id_a = (uint32_t)(key[j] >> 32);
                    slot = (uint32_t)key[j];
                    at = j + mine;
                }
            } else {
                uint32_t c = j < A ? below[j] : 0u;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(FULL, c, d);
                    if (lane >= d)
                        c += y;
                }
                if (j < A) {
                    id_a = (uint32_t)(key[j] >> 32);
                    slot = (uint32_t)key[j];
                    at = j + carry + c;
                }
                carry += __shfl_sync(FULL, c, 31);
            }
            if (j < A)
                L.put((int64_t)p0 + at, xi[slot], v[slot], fabs(zeta_new[slot]), (int32_t)id_a);
        }
        if (lane == 0) {
            if (p0 + (int32_t)(n_stay + A) < p1) // the padding slot of an odd cell
                L.put(p1 - 1, 0, 1.0, 0.0, -1);
            M.arr[g] = 0u; // for the next step
        }
        __syncwarp();
    }
    if (__syncthreads_or(heavy)) // what is left of the block's cells
        for (int g0 = blockIdx.x * W; g0 < n_cells; g0 += nw)
            for (int g = g0; g < min(g0 + W, n_cells); ++g)
                if (M.arr[g] > (uint32_t)kSedArrive) // uniform: cleared behind a barrier
                    sed_merge_heavy(g, cell_off, M, xi, v, zeta_new, id_of_slot, poff, L, &s_key[0][0],
                                    s_u.heavy);
    if (blockIdx.x == 0 && threadIdx.x == 0) { // the run's record: nothing here reads it
        *M.out_next = 0u;
        rec->xi = L.xi;
        rec->v = L.v;
        rec->cell_off = poff;
        rec->step = step;
    }
    // outside the domain: those that were, in their order, then the arrivals
    const int32_t lo = cell_off[n_cells], p0 = poff[n_cells], p1 = poff[n_cells + 1];
    const uint32_t n_out = M.stay[n_cells], A = *M.out, a0 = (uint32_t)M.first[n_cells];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p1 - p0; i += (int64_t)gridDim.x * blockDim.x) {
        if (i < n_out) {
            L.put(p0 + i, xi[lo + i], v[lo + i], 0.0, id_of_slot[lo + i]);
        } else if (i < (int64_t)n_out + A) {
            const uint32_t s = M.a_slot[a0 + (i - n_out)];
            L.put(p0 + i, xi[s], v[s], fabs(zeta_new[s]), (int32_t)M.a_id[a0 + (i - n_out)]);
        } else {
            L.put(p0 + i, 0, 1.0, 0.0, -1);
        }
    }
}

// -------------------------------------------------------------------- host
// The second layout (swapped with the context's after every step, so both
// sets are freed through their current pointers) and the scratch.
struct SedBuffers {
    int64_t *xi2 = nullptr;
    double *v2 = nullptr;
    double *zeta2 = nullptr;
    int32_t *id2 = nullptr;
    int32_t *group = nullptr;     // sorted path: group of every slot of the current layout;
    int32_t *group2 = nullptr;    //   else the arrivals' ids and slots
    bool group_valid = false;     // group holds the current layout's
    int32_t *cell_off2 = nullptr; // n_cells + 2
    double *zeta_new = nullptr;   // per slot of the old layout
    uint32_t *keys[2] = {}; // sorted path: keys and slots; else the movers' new groups, ids,
    uint32_t *vals[2] = {}; //   slots and places
    uint32_t *moves = nullptr; // per group: stayers, arrivals, movers, first arrival; then block totals
    int parity = 0;            // which of the two counts of SDs leaving the domain (behind the cells'
                               //   arrivals) the next step uses; all arrivals are zero between steps
    uint32_t *counts = nullptr; // n_cells + 1
    int32_t *ustart = nullptr;  // n_cells + 2
    ExactBin *precip = nullptr; // the precipitated water's bins (zero between steps), then its sum, the
                                //   movers' count and the mark of a pile
    int sorted_left = 0;        // steps that take the sorted path before the cells are tried again
    uint32_t *hist = nullptr;   // 256 x tiles, then 256 digit totals
    uint32_t *flags = nullptr;  // flags, then the first bad id (8-byte aligned)
    int32_t *emig = nullptr;    // per SD id: its cell in another piece of the grid after the last step, or -1
    void *h_read = nullptr;     // pinned: the new offsets, the precipitated total and the plan's class counts
    cudaStream_t side = nullptr; // the offset scan (and the plan's refresh) beside the radix sort
    cudaEvent_t fork = nullptr, join = nullptr;
};

// Bytes of the pinned read-back buffer for n_cells cells: n_cells + 2
// offsets, the precipitated total (8-byte aligned) with the movers' count and the
// mark of a pile, and the class-count words.
size_t sed_read_bytes(int32_t n_cells) { return (((size_t)n_cells + 2) * 4 + 7) / 8 * 8 + 16 + sizeof(uint32_t) * (kNumClass + 1); }

void sed_release(sdm_ctx *ctx)
{
    if (ctx->sed) {
        SedBuffers &b = *ctx->sed;
        void *bufs[] = {b.xi2,      b.v2,       b.zeta2,    b.id2,    b.group,  b.group2,
                        b.cell_off2, b.zeta_new, b.keys[0], b.keys[1], b.vals[0], b.vals[1],
                        b.counts,   b.ustart,   b.precip,   b.hist,   b.flags,  b.emig,
                        b.moves};
        for (void *p : bufs)
            ctx->mem.put(p, 0);
        if (b.h_read || b.side) {
            cudaStreamSynchronize(ctx->stream); // no read-back in flight, the side stream joined
            if (b.side)
                cudaStreamSynchronize(b.side);
        }
        if (b.h_read)
            cudaFreeHost(b.h_read);
        if (b.side)
            cudaStreamDestroy(b.side);
        if (b.fork)
            cudaEventDestroy(b.fork);
        if (b.join)
            cudaEventDestroy(b.join);
        delete ctx->sed;
        ctx->sed = nullptr;
    }
    ctx->mem.put(ctx->d_zeta, 0);
    ctx->d_zeta = nullptr;
}

template <typename T>
T *sed_get(sdm_ctx *ctx, size_t count)
{
    return static_cast<T *>(ctx->mem.get(sizeof(T) * (count > 0 ? count : 1)));
}

// Words of one of the per-group arrays of SedBuffers::moves (a multiple of 2:
// the totals behind them are 8-byte words).
size_t sed_stride(int32_t n_cells) { return ((size_t)n_cells + 5) & ~(size_t)1; }

sdm_status sed_alloc(sdm_ctx *ctx)
{
    if (ctx->sed)
        return SDM_OK;
    ctx->sed = new (std::nothrow) SedBuffers();
    if (!ctx->sed)
        return fail(&ctx->error, SDM_ENOMEM, "host allocation failed");
    SedBuffers &b = *ctx->sed;
    const int64_t slots = ctx->n_slots_cap, cap = ctx->capacity_sd;
    const int32_t nc = ctx->cfg.n_cells;
    ctx->d_zeta = (double *)ctx->mem.get(sizeof(double) * slots);
    b.xi2 = sed_get<int64_t>(ctx, slots);
    b.v2 = sed_get<double>(ctx, slots);
    b.zeta2 = sed_get<double>(ctx, slots);
    b.id2 = sed_get<int32_t>(ctx, slots);
    b.group = sed_get<int32_t>(ctx, slots);
    b.group2 = sed_get<int32_t>(ctx, slots);
    b.cell_off2 = sed_get<int32_t>(ctx, (size_t)nc + 2);
    b.zeta_new = sed_get<double>(ctx, slots);
    for (int i = 0; i < 2; ++i) {
        b.keys[i] = sed_get<uint32_t>(ctx, slots);
        b.vals[i] = sed_get<uint32_t>(ctx, slots);
    }
    b.counts = sed_get<uint32_t>(ctx, (size_t)nc + 1);
    b.ustart = sed_get<int32_t>(ctx, (size_t)nc + 2);
    b.precip = sed_get<ExactBin>(ctx, (size_t)kExactBins + 2);
    b.hist = sed_get<uint32_t>(ctx, radix_hist_words(cap));
    b.flags = sed_get<uint32_t>(ctx, 4);
    b.moves = sed_get<uint32_t>(ctx, 4 * sed_stride(nc) + 2 * ((size_t)nc / 1024 + 1));
    b.emig = sed_get<int32_t>(ctx, cap);
    if (cudaMallocHost(&b.h_read, sed_read_bytes(nc)) != cudaSuccess) {
        cudaGetLastError();
        b.h_read = nullptr;
    }
    if (cudaStreamCreateWithFlags(&b.side, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&b.fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&b.join, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        sed_release(ctx);
        return fail(&ctx->error, SDM_ENOMEM, "sedimentation stream and events: creation failed");
    }
    const bool ok = ctx->d_zeta && b.xi2 && b.v2 && b.zeta2 && b.id2 && b.group && b.group2 && b.cell_off2 &&
                    b.zeta_new && b.keys[0] && b.keys[1] && b.vals[0] && b.vals[1] && b.counts && b.ustart &&
                    b.precip && b.hist && b.flags && b.emig && b.moves && b.h_read;
    if (!ok) {
        sed_release(ctx);
        return fail(&ctx->error, SDM_ENOMEM, "sedimentation buffers: device allocation failed");
    }
    if (cudaMemsetAsync(b.moves, 0, sizeof(uint32_t) * 2 * sed_stride(nc), ctx->stream) != cudaSuccess ||
        cudaMemsetAsync(b.precip, 0, sizeof(ExactBin) * kExactBins, ctx->stream) != cudaSuccess) {
        cudaGetLastError();
        sed_release(ctx);
        return fail(&ctx->error, SDM_ECUDA, "sedimentation buffers: clearing failed");
    }
    ctx->device_bytes += slots * (8 + 8 + 8 + 8 + 4 + 4 + 4 + 8 + 16) + cap * 4 + ((int64_t)nc + 2) * 32 +
                         (int64_t)radix_hist_words(cap) * 4;
    return SDM_OK;
}

int sed_grid(int32_t n_groups)
{
    return std::max(1, std::min((n_groups + kSedNT / 32 - 1) / (kSedNT / 32), 152 * 16));
}

} // namespace

namespace {

// sdm_set_positions (zeta_in = 0: z above the grid's bottom) and
// sdm_set_heights (zeta_in = 1: z holds the heights above the cells' bottoms)
sdm_status set_positions_impl(sdm_ctx *ctx, const double *z, int32_t nx, double dz, int on_device, int zeta_in)
{
    sdm_status st = ctx_usable(ctx);
    if (st != SDM_OK)
        return st;
    if (!ctx->has_attributes)
        return fail(&ctx->error, SDM_ESTATE, "sdm_set_attributes has not been called");
    const int32_t nc = ctx->cfg.n_cells;
    if (!z || nx < 1 || nc % nx != 0 || !(std::isfinite(dz) && dz > 0.0))
        return fail(&ctx->error, SDM_EINVAL, "need z, nx >= 1 dividing n_cells = %d, and a finite dz > 0", nc);
    if (ctx->cfg.cell_base % nx != 0)
        return fail(&ctx->error, SDM_EINVAL, "nx = %d must divide cell_base = %d (pieces of a grid are whole levels)",
                    nx, ctx->cfg.cell_base);
    st = sed_alloc(ctx);
    if (st != SDM_OK)
        return st;
    cudaStream_t s = ctx->stream;
    const double *dz_arr = z;
    void *stage = nullptr;
    const size_t bz = sizeof(double) * ctx->n_sd;
    if (!on_device) {
        stage = ctx->mem.get(bz);
        if (!stage)
            return fail(&ctx->error, SDM_ENOMEM, "staging allocation failed");
        CTX_CUDA(ctx, cudaMemcpyAsync(stage, z, bz, cudaMemcpyHostToDevice, s));
        dz_arr = (const double *)stage;
    }
    uint32_t *d_flags = ctx->sed->flags;
    unsigned long long *d_bad = (unsigned long long *)(d_flags + 2);
    CTX_CUDA(ctx, cudaMemsetAsync(d_flags, 0, 16, s));
    sed_set_kernel<<<sed_grid(nc + 1), kSedNT, 0, s>>>(ctx->d_cell_off, nc, ctx->n_slots, ctx->d_id_of_slot, dz_arr,
                                                        nx, dz, ctx->cfg.cell_base, zeta_in, ctx->d_zeta, d_flags,
                                                        d_bad);
    ctx->sed->group_valid = false;
    ctx->sed->sorted_left = 0;
    if (ctx->cfg.cell_base > 0) // only a piece of a grid has emigrants
        CTX_CUDA(ctx, cudaMemsetAsync(ctx->sed->emig, 0xFF, sizeof(int32_t) * ctx->n_sd, s));
    CTX_CUDA(ctx, cudaGetLastError());
    CTX_CUDA(ctx, cudaMemcpyAsync(ctx->sed->h_read, d_flags, 16, cudaMemcpyDeviceToHost, s));
    CTX_CUDA(ctx, cudaStreamSynchronize(s));
    const uint32_t flags = *(const uint32_t *)ctx->sed->h_read;
    const unsigned long long bad = ~((const unsigned long long *)ctx->sed->h_read)[1];
    ctx->mem.put(stage, bz);
    if (flags & 1u) {
        ctx->has_positions = false;
        return fail(&ctx->error, SDM_EINVAL,
                    zeta_in ? "SD %llu: zeta must lie in [0, dz)" : "SD %llu: z must lie in its cell's level [iz dz, (iz + 1) dz)",
                    bad);
    }
    ctx->nx = nx;
    ctx->dz = dz;
    ctx->has_positions = true;
    return SDM_OK;
}

} // namespace

extern "C" sdm_status sdm_set_positions(sdm_ctx *ctx, const double *z, int32_t nx, double dz, int on_device)
{
    NvtxRange nvtx_range("sdm_set_positions");
    return set_positions_impl(ctx, z, nx, dz, on_device, 0);
}

extern "C" sdm_status sdm_set_heights(sdm_ctx *ctx, const double *zeta, int32_t nx, double dz, int on_device)
{
    NvtxRange nvtx_range("sdm_set_heights");
    return set_positions_impl(ctx, zeta, nx, dz, on_device, 1);
}

extern "C" sdm_status sdm_sedimentation_step(sdm_ctx *ctx, double *precipitated)
{
    NvtxRange nvtx_range("sdm_sedimentation_step");
    sdm_status st = ctx_usable(ctx);
    if (st != SDM_OK)
        return st;
    if (!ctx->has_attributes || !ctx->has_positions)
        return fail(&ctx->error, SDM_ESTATE, "sdm_set_positions has not been called for the current attributes");
    SedBuffers &b = *ctx->sed;
    cudaStream_t s = ctx->stream;
    const int32_t nc = ctx->cfg.n_cells, n_groups = nc + 1;
    const int64_t n = ctx->n_sd;
    sdm_batch *sb = ctx->self_batch;
    const bool refresh = sb && sb->plan.refreshable && same_tuning(sb->plan.tuning, current_tuning());
    double *precip_sum = reinterpret_cast<double *>(b.precip + kExactBins);
    unsigned char *hr = static_cast<unsigned char *>(b.h_read);
    const int32_t *off = reinterpret_cast<const int32_t *>(hr);
    const size_t at_pr = (((size_t)nc + 2) * 4 + 7) / 8 * 8;
    const uint32_t *rc = reinterpret_cast<const uint32_t *>(hr + at_pr + 16);
    // on the side stream, beside what follows the new offsets: the refresh of
    // the context's own launch plan (when refreshable: rebuilt on the device for
    // the new layout) and the read-back into the pinned buffer (offsets,
    // precipitated total, class counts)
    auto side_work = [&]() -> sdm_status {
        if (refresh) {
            CTX_CUDA(ctx, plan_refresh(sb->plan, b.cell_off2, nc, ctx->cfg.cell_base, b.side));
            CTX_CUDA(ctx, cudaMemcpyAsync(hr + at_pr + 16, sb->plan.d_refresh, sizeof(uint32_t) * (kNumClass + 1),
                                          cudaMemcpyDeviceToHost, b.side));
        }
        CTX_CUDA(ctx, cudaMemcpyAsync(hr, b.cell_off2, sizeof(int32_t) * (n_groups + 1), cudaMemcpyDeviceToHost, b.side));
        CTX_CUDA(ctx, cudaMemcpyAsync(hr + at_pr, b.precip + kExactBins, 2 * sizeof(double), cudaMemcpyDeviceToHost,
                                      b.side));
        CTX_CUDA(ctx, cudaEventRecord(b.join, b.side));
        return SDM_OK;
    };
    // A few cells leave most of the chip idle while a warp follows a cell's movers
    // and merges them one after the other (us a step, by cells | sorted: 16 to 128 cells of
    // 1000, 5% moving 55 | 50, all moving 75 | 50; of 600 43 | 50 and 95 | 50; of
    // 300 33 | 50 and 67 | 50; 512 cells of 1000 66 | 80 and 103 | 93; 4096 cells: by
    // cells is faster for any share): sorted if the cells are large, or if over a third
    // of the SDs moved a few steps ago.  Any number of cells: sorted for as long when
    // one of them received more than kSedRunKeys SDs (a block that merges a pile works
    // alone: 640 columns of 3 cells of 1000 that all fall into the lowest one 473 us
    // merged in runs, 183 sorted; 10 columns of 64, 120 ms and 0.15).  The step that
    // finds that out is taken twice (257 and 328 us).
    const bool few = nc <= kSedFewCells;
    bool by_cell = ctx->largest_cell <= kSedByCell && !(2 * nc <= kSedFewCells && ctx->largest_cell > kSedFewLargest) &&
                         b.sorted_left == 0;
    auto sorted_step = [&]() -> sdm_status {
        if (!b.group_valid) {
            const int64_t per_block = (int64_t)kSedNT * kSedGroupRun;
            sed_group_kernel<<<(int)((ctx->n_slots + per_block - 1) / per_block), kSedNT, 0, s>>>(ctx->d_cell_off, nc,
                                                                                               ctx->n_slots, b.group);
        }
        CTX_CUDA(ctx, cudaMemsetAsync(b.counts, 0, sizeof(uint32_t) * n_groups, s));
        const int move_blocks = (int)std::max<int64_t>(
            1,
            std::min<int64_t>(kSedMaxBlocks, (ctx->n_slots + (int64_t)kSedNT * kSedU - 1) / ((int64_t)kSedNT * kSedU)));
        sed_move_kernel<<<move_blocks, kSedNT, 0, s>>>(ctx->d_inst, nc, ctx->n_slots, ctx->nx, ctx->dz,
                                                       (float)ctx->cfg.dt, ctx->d_zeta, b.group, ctx->d_id_of_slot,
                                                       b.keys[0], b.vals[0], b.zeta_new, b.counts, b.precip,
                                                       ctx->cfg.cell_base, b.emig);
        // the offset scan, the padding and the rest of the side stream's work
        // beside the radix sort, which needs none of them
        CTX_CUDA(ctx, cudaEventRecord(b.fork, s));
        CTX_CUDA(ctx, cudaStreamWaitEvent(b.side, b.fork, 0));
        sed_scan_kernel<<<1, 1024, 0, b.side>>>(b.counts, n_groups, b.ustart, b.cell_off2, b.precip, precip_sum);
        // the new layout's padding slots (the gather writes only the others)
        sed_pad_kernel<<<(n_groups + 255) / 256, 256, 0, b.side>>>(n_groups, b.ustart, b.cell_off2, b.xi2, b.v2,
                                                                    b.zeta2, b.id2, b.group2);
        const sdm_status sw = side_work();
        if (sw != SDM_OK)
            return sw;
        // stable sort of the new groups, SD-id order in
        const int bits = 32 - __builtin_clz((unsigned)nc | 1u);
        const int cur = radix_sort(b.keys, b.vals, false, n, bits, b.hist, s);
        CTX_CUDA(ctx, cudaStreamWaitEvent(s, b.join, 0));
        sed_gather_kernel<<<1216, 256, 0, s>>>(n, b.keys[cur], b.vals[cur], b.ustart, b.cell_off2, ctx->d_xi, ctx->d_v,
                                               b.zeta_new, ctx->d_id_of_slot, b.xi2, b.v2, b.zeta2, b.id2, b.group2);
        CTX_CUDA(ctx, cudaGetLastError());
        std::swap(b.group, b.group2);
        b.group_valid = true;
        return SDM_OK;
    };
    if (b.sorted_left > 0)
        --b.sorted_left;
    if (by_cell) {
        const size_t st_ = sed_stride(nc);
        SedMoves M{b.keys[0], b.vals[0],      b.keys[1],          b.vals[1],   (uint32_t *)b.group, (uint32_t *)b.group2,
                   b.moves,   b.moves + st_, b.moves + 2 * st_, b.moves + 2 * st_ - 1 - b.parity,
                   b.moves + 2 * st_ - 2 + b.parity, (int32_t *)(b.moves + 3 * st_),
                   (uint32_t *)(b.precip + kExactBins + 1), (uint32_t *)(b.precip + kExactBins + 1) + 1};
        b.parity ^= 1;
        unsigned long long *totals = (unsigned long long *)(b.moves + 4 * st_);
        b.group_valid = false;
        if (ctx->cfg.cell_base > 0) // the emigrants of the step before are none of this one's
            CTX_CUDA(ctx, cudaMemsetAsync(b.emig, 0xFF, sizeof(int32_t) * n, s));
        const int warps = kSedNT / 32;
        const int fall_blocks = std::max(1, std::min((nc + warps - 1) / warps, 152 * 4));
        sed_fall_kernel<<<fall_blocks, kSedNT, 0, s>>>(ctx->d_inst, ctx->d_cell_off, nc, ctx->n_slots, ctx->nx, ctx->dz,
                                                       (float)ctx->cfg.dt, ctx->d_zeta, ctx->d_id_of_slot, b.zeta_new, M,
                                                       b.precip, ctx->cfg.cell_base, b.emig);
        const int blocks = (n_groups + 1023) / 1024;
        if (blocks > 64)
            sed_totals_kernel<<<blocks, 1024, 0, s>>>(M, n_groups, totals);
        sed_offsets_kernel<<<blocks, 1024, 0, s>>>(M, n_groups, blocks > 64 ? totals : nullptr, b.cell_off2, b.precip,
                                                   precip_sum);
        CTX_CUDA(ctx, cudaEventRecord(b.fork, s));
        CTX_CUDA(ctx, cudaStreamWaitEvent(b.side, b.fork, 0));
        st = side_work();
        if (st != SDM_OK)
            return st;
        sed_deal_kernel<<<std::max(1, std::min((nc + warps - 1) / warps, 152 * 8)), kSedNT, 0, s>>>(ctx->d_cell_off, nc, M);
        const int mw = kSedMergeNT / 32;
        const int64_t units = std::max<int64_t>((nc + mw - 1) / mw, (ctx->n_slots - ctx->h_cell_off[nc]) / kSedMergeNT + 1);
        sed_merge_kernel<<<(int)std::min<int64_t>(units, 152 * 9), kSedMergeNT, 0, s>>>(
            ctx->d_cell_off, nc, M, ctx->d_xi, ctx->d_v, b.zeta_new, ctx->d_id_of_slot, b.cell_off2,
            SedLayout{b.xi2, b.v2, b.zeta2, b.id2}, ctx->d_inst, ctx->step);
        CTX_CUDA(ctx, cudaGetLastError());
        CTX_CUDA(ctx, cudaStreamWaitEvent(s, b.join, 0)); // later work may write what the side stream reads
        // the read-back only: what writes the new layout goes on behind it
        CTX_CUDA(ctx, cudaEventSynchronize(b.join));
        uint32_t moved[2]; // movers, whether a cell receives too many
        std::memcpy(moved, hr + at_pr + 8, sizeof moved);
        if (moved[1] || (few && (int64_t)moved[0] * 3 > n))
            b.sorted_left = 16;
        by_cell = moved[1] == 0;
    }
    if (!by_cell) {
        st = sorted_step();
        if (st != SDM_OK)
            return st;
        CTX_CUDA(ctx, cudaEventSynchronize(b.join));
    }
    double precip = 0.0;
    std::memcpy(&precip, hr + at_pr, sizeof precip);
    // the new layout becomes the state; the old one the next scratch
    std::swap(ctx->d_xi, b.xi2);
    std::swap(ctx->d_v, b.v2);
    std::swap(ctx->d_zeta, b.zeta2);
    std::swap(ctx->d_id_of_slot, b.id2);
    std::swap(ctx->d_cell_off, b.cell_off2);
    int32_t largest = 0;
    for (int32_t c = 0; c < nc; ++c)
        largest = std::max(largest, off[c + 1] - off[c]);
    const bool keep_plan = ctx->self_batch && ctx->h_cell_off.size() == (size_t)nc + 1 &&
                           std::equal(ctx->h_cell_off.begin(), ctx->h_cell_off.end(), off) &&
                           same_tuning(ctx->self_batch->plan.tuning, current_tuning());
    ctx->h_cell_off.assign(off, off + nc + 1);
    ctx->n_slots = off[n_groups];
    ctx->largest_cell = largest;
    ctx->layout_version += 1;
    ctx->dev_base = ctx->step;
    if (!by_cell) { // (the merge writes the record itself)
        InstDev inst = make_inst(ctx);
        CTX_CUDA(ctx, cudaMemcpyAsync(ctx->d_inst, &inst, sizeof inst, cudaMemcpyHostToDevice, s));
    }
    const bool refreshed = refresh && !keep_plan && rc[kNumClass] == 0;
    if (refreshed)
        for (int k = 0; k < kNumClass; ++k) {
            Plan &pl = ctx->self_batch->plan;
            pl.n_items[k] = (int)rc[k];
            pl.variant[k] = variant_of_class(k, pl.n_items[k], pl.tuning);
        }
    if (ctx->self_batch && (keep_plan || refreshed))
        ctx->self_batch->versions[0] = ctx->layout_version;
    if (!keep_plan && !refreshed)
        drop_own_plan(ctx);
    if (precipitated)
        *precipitated = precip;
    return SDM_OK;
}

extern "C" sdm_status sdm_get_positions(sdm_ctx *ctx, double *z, int32_t *cell, int on_device)
{
    NvtxRange nvtx_range("sdm_get_positions");
    sdm_status st = ctx_usable(ctx);
    if (st != SDM_OK)
        return st;
    if (!ctx->has_attributes)
        return fail(&ctx->error, SDM_ESTATE, "sdm_set_attributes has not been called");
    if (z && !ctx->has_positions)
        return fail(&ctx->error, SDM_ESTATE, "no positions: sdm_set_positions has not been called");
    if (!z && !cell)
        return SDM_OK;
    cudaStream_t s = ctx->stream;
    const int32_t nc = ctx->cfg.n_cells;
    const int32_t nx = ctx->has_positions ? ctx->nx : 1;
    const int64_t n = ctx->n_sd;
    if (on_device) {
        sed_get_kernel<<<sed_grid(nc + 1), kSedNT, 0, s>>>(ctx->d_cell_off, nc, ctx->n_slots, ctx->d_id_of_slot,
                                                            ctx->d_zeta, nx, ctx->dz, ctx->cfg.cell_base, nullptr, z,
                                                            cell, nullptr, nullptr);
        CTX_CUDA(ctx, cudaGetLastError());
        return SDM_OK;
    }
    const size_t bz = sizeof(double) * n, bc = sizeof(int32_t) * n;
    char *tmp = (char *)ctx->mem.get(bz + bc);
    if (!tmp)
        return fail(&ctx->error, SDM_ENOMEM, "allocation failed");
    sed_get_kernel<<<sed_grid(nc + 1), kSedNT, 0, s>>>(ctx->d_cell_off, nc, ctx->n_slots, ctx->d_id_of_slot,
                                                        ctx->d_zeta, nx, ctx->dz, ctx->cfg.cell_base, nullptr,
                                                        z ? (double *)tmp : nullptr,
                                                        cell ? (int32_t *)(tmp + bz) : nullptr, nullptr, nullptr);
    CTX_CUDA(ctx, cudaGetLastError());
    if (z)
        CTX_CUDA(ctx, cudaMemcpyAsync(z, tmp, bz, cudaMemcpyDeviceToHost, s));
    if (cell)
        CTX_CUDA(ctx, cudaMemcpyAsync(cell, tmp + bz, bc, cudaMemcpyDeviceToHost, s));
    CTX_CUDA(ctx, cudaStreamSynchronize(s));
    ctx->mem.put(tmp, bz + bc);
    return check_device_status(ctx);
}

extern "C" sdm_status sdm_get_heights(sdm_ctx *ctx, double *zeta, int32_t *cell, int on_device)
{
    NvtxRange nvtx_range("sdm_get_heights");
    sdm_status st = ctx_usable(ctx);
    if (st != SDM_OK)
        return st;
    if (!ctx->has_attributes || !ctx->has_positions)
        return fail(&ctx->error, SDM_ESTATE, "no positions: sdm_set_positions has not been called");
    if (!zeta && !cell)
        return SDM_OK;
    cudaStream_t s = ctx->stream;
    const int32_t nc = ctx->cfg.n_cells;
    const int64_t n = ctx->n_sd;
    const int32_t *emig = ctx->cfg.cell_base > 0 ? ctx->sed->emig : nullptr;
    if (on_device) {
        sed_get_kernel<<<sed_grid(nc + 1), kSedNT, 0, s>>>(ctx->d_cell_off, nc, ctx->n_slots, ctx->d_id_of_slot,
                                                            ctx->d_zeta, ctx->nx, ctx->dz, ctx->cfg.cell_base, emig,
                                                            nullptr, nullptr, zeta, cell);
        CTX_CUDA(ctx, cudaGetLastError());
        return SDM_OK;
    }
    const size_t bz = sizeof(double) * n, bc = sizeof(int32_t) * n;
    char *tmp = (char *)ctx->mem.get(bz + bc);
    if (!tmp)
        return fail(&ctx->error, SDM_ENOMEM, "allocation failed");
    sed_get_kernel<<<sed_grid(nc + 1), kSedNT, 0, s>>>(ctx->d_cell_off, nc, ctx->n_slots, ctx->d_id_of_slot,
                                                        ctx->d_zeta, ctx->nx, ctx->dz, ctx->cfg.cell_base, emig, nullptr,
                                                        nullptr, zeta ? (double *)tmp : nullptr,
                                                        cell ? (int32_t *)(tmp + bz) : nullptr);
    CTX_CUDA(ctx, cudaGetLastError());
    if (zeta)
        CTX_CUDA(ctx, cudaMemcpyAsync(zeta, tmp, bz, cudaMemcpyDeviceToHost, s));
    if (cell)
        CTX_CUDA(ctx, cudaMemcpyAsync(cell, tmp + bz, bc, cudaMemcpyDeviceToHost, s));
    CTX_CUDA(ctx, cudaStreamSynchronize(s));
    ctx->mem.put(tmp, bz + bc);
    return check_device_status(ctx);
}

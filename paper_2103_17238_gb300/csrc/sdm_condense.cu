// Condensation step (sdm_condensation_step in include/sdm.h).
//
// The paper lists condensation among the dynamics of its framework and
// prints no formulae.  Reading: the large-drop limit of the diffusional
// growth law, r dr/dt = s G (Rogers & Yau 1989, ch. 7, curvature and solute
// terms dropped), with each cell's supersaturation s and growth coefficient
// G = 1 / (F_k + F_d) held over the step, so r^2 grows by c = 2 G s dt; an
// evaporating SD stops at the floor radius r_min (or at its own radius when
// that is already below it).  The change of volume is evaluated in binary32
// from the binary32 image of the volume and its binary32 radius, in a form
// without cancellation, and added to the binary64 volume (as the fall
// distance of sedimentation is): per SD
//   x = r^2, x' = max(x + c, min(x, r_min^2)), d = c (or floor - x),
//   dV = k43 (d ((x' + a b) + x)) / (a + b), a = sqrt(x'), b = sqrt(x),
//   v' = v + dV.
// Multiplicities do not change.  The per-cell condensed water sum(xi dV) is
// an optional output.
//
// One step on the device (a warp takes up to 256 slots of one cell at a time:
// 16-byte loads of xi and v, the binary32 arithmetic per SD, one binary64 add
// per SD to update v, the sum of xi dV in fixed point):
//   condense_by_cell_kernel one warp per cell, its water at once; or, when
//                         the largest cell is above 1024 slots,
//   condense_kernel       one warp per work item of up to 256 slots, and
//   condense_cells_kernel per cell, its items' partials in item order.
// HBM traffic: 16 B read and 8 B written per live SD.
//
// Compiled as part of the library's single translation unit (included at the
// end of sdm_runtime.cu).

namespace {

constexpr int kCondItem = 256; // slots per work item (a multiple of 2: cells start at even slots)
constexpr int kCondNT = 256;
constexpr int kCondByCell = 1024; // largest cell that one warp takes (4 rounds)
constexpr int kCondFewCells = 1216; // up to here a block takes a cell of more than kCondItem slots
constexpr int kCondStage = 4;     // fields in page-locked memory: the next call's, and those on their way
constexpr float kR3ToVolF = (float)(4.0 * kPi / 3.0); // 4 pi / 3 (binary64 pi) rounded to binary32

struct __align__(16) CondItem {
    int32_t cell;
    int32_t begin; // first slot
    int32_t n;     // slots (<= kCondItem), even
    int32_t pad;
};

struct CondBuffers {
    int64_t layout_version = -1; // the layout the work list was built for
    int32_t n_items = 0;
    CondItem *items = nullptr;
    int32_t *item_start = nullptr; // n_cells + 1, with the first work list
    double *partial = nullptr;     // n_items
    double *cond = nullptr;        // n_cells
    // c of each cell, binary32.  A field other than the last is read by the kernel
    // where it lies in page-locked memory (a copy ahead of it cost more than its
    // reads), which leaves it in cf for the calls that repeat it: those are a
    // launch and nothing else, in a captured graph too.
    float *cf = nullptr;   // n_cells
    float *h_cf = nullptr; // kCondStage fields
    cudaEvent_t cf_done[kCondStage] = {}; // the last kernel that reads each
    int stage = 0;         // the next call's: no kernel reads it
    int last = -1;         // the one that is in cf (-1: none)
};

// f2d_exact (sdm_sediment.cu): the exact widening of a binary32 on the
// integer pipe.

// dV of one live SD (the reading above), binary32.  The binary32 image of
// v is rounded on the integer pipe (d2f_rn): the conversion instruction would
// take the narrow binary64 pipe, which then bounds the kernel.  sqrt(x) is r
// itself: in binary arithmetic rounded to nearest the square root of a
// rounded square is the number again (Boldo 2015; r^2 is far from underflow).
__device__ __forceinline__ float condense_dv(double v, float cf, float xminf)
{
    bool in_range;
    const float r = radius32(d2f_rn(v, in_range)); // volumes lie in [1e-30, 1e30]: always in range
    const float x = __fmul_rn(r, r);
    float xn = __fadd_rn(x, cf);
    const float lo = x < xminf ? x : xminf;
    float d = cf;
    if (xn < lo) {
        xn = lo;
        d = __fsub_rn(lo, x);
    }
    if (d == 0.0f)
        return 0.0f;
    const float a = __fsqrt_rn(xn);
    const float num = __fmul_rn(d, __fadd_rn(__fadd_rn(xn, __fmul_rn(a, r)), x));
    return __fmul_rn(kR3ToVolF, __fdiv_rn(num, __fadd_rn(a, r)));
}

// |dV|'s exponent field (1 for subnormals) and mantissa.
__device__ __forceinline__ uint32_t dv_exponent(float dv) { return max((__float_as_uint(dv) >> 23) & 0xFFu, 1u); }
__device__ __forceinline__ uint32_t dv_mantissa(float dv)
{
    const uint32_t b = __float_as_uint(dv);
    return (b & 0x7FFFFFu) | ((b & 0x7F800000u) ? 0x800000u : 0u);
}

// One warp's round: up to kCondItem slots of one cell (n even) grow, and with
// WATER the sum of xi |dV| is returned (every dV of a cell has the sign of its
// cf).  xi |dV| is exact below xi 2^39 and is cut to 63 bits below the round's
// greatest: FixedSum.
template <bool WATER>
__device__ __forceinline__ double condense_round(const int64_t *__restrict__ xi, double *__restrict__ v, int n, float c,
                                                 float xminf)
{
    constexpr int PAIRS = kCondItem / 64; // SD pairs per lane
    const int lane = threadIdx.x & 31;
    const longlong2 *x2 = reinterpret_cast<const longlong2 *>(xi);
    double2 *v2 = reinterpret_cast<double2 *>(v);
    const int np = n / 2;
    longlong2 xs[PAIRS];
    double2 vs[PAIRS];
#pragma unroll
    for (int k = 0; k < PAIRS; ++k) { // every load of the round first
        const int q = lane + 32 * k;
        xs[k] = q < np ? x2[q] : make_longlong2(0, 0);
        vs[k] = q < np ? v2[q] : make_double2(1.0, 1.0);
    }
    float dv[2 * PAIRS];
    uint32_t emax = 0u;
#pragma unroll
    for (int k = 0; k < PAIRS; ++k) {
        double2 w = vs[k];
        dv[2 * k] = xs[k].x > 0 ? condense_dv(w.x, c, xminf) : 0.0f;
        dv[2 * k + 1] = xs[k].y > 0 ? condense_dv(w.y, c, xminf) : 0.0f;
        if (dv[2 * k] != 0.0f || dv[2 * k + 1] != 0.0f) { // adding 0 changes nothing
            w.x = __dadd_rn(w.x, f2d_exact(dv[2 * k]));
            w.y = __dadd_rn(w.y, f2d_exact(dv[2 * k + 1]));
            v2[lane + 32 * k] = w;
        }
        if constexpr (WATER) {
            if (dv[2 * k] != 0.0f)
                emax = max(emax, 63u - (uint32_t)__clzll(xs[k].x) + dv_exponent(dv[2 * k]));
            if (dv[2 * k + 1] != 0.0f)
                emax = max(emax, 63u - (uint32_t)__clzll(xs[k].y) + dv_exponent(dv[2 * k + 1]));
        }
    }
    if constexpr (!WATER)
        return 0.0;
    emax = __reduce_max_sync(0xFFFFFFFFu, emax);
    FixedSum f;
#pragma unroll
    for (int k = 0; k < 2 * PAIRS; ++k) {
        if (dv[k] == 0.0f)
            continue;
        const uint64_t x = (uint64_t)((k & 1) ? xs[k / 2].y : xs[k / 2].x);
        const uint32_t m = dv_mantissa(dv[k]);
        // the product below 2^63 in units of 2^(emax - 188)
        const int sh = (int)dv_exponent(dv[k]) - (int)emax + 38;
        if (x >> 39) { // xi above 5e11: the product's top 64 bits
            const uint32_t lz = (uint32_t)__clzll((long long)x);
            const uint64_t h = __umul64hi(x << lz, (uint64_t)m << 40); // the product times 2^(lz - 24)
            const int r = sh + 24 - (int)lz;
            f.add(r >= 0 ? h << r : (r > -64 ? h >> -r : 0ull));
        } else {
            const uint64_t pr = x * m;
            f.add(sh >= 0 ? pr << sh : (sh > -64 ? pr >> -sh : 0ull));
        }
    }
    return f.warp_sum((int)emax - 188);
}

// Every cell by one warp: no work list, nothing to rebuild when the layout
// changes, no second pass.  56 + 10 us per call of the 4.19M-SD grid as two
// kernels with binary64 sums (the binary64 pipe 68% busy).  KEEP: the field is
// left in `keep`.
template <bool WATER, bool KEEP>
__global__ void __launch_bounds__(kCondNT) condense_by_cell_kernel(const int32_t *__restrict__ cell_off, int32_t n_cells,
                                                                   const int64_t *__restrict__ xi,
                                                                   double *__restrict__ v, const float *__restrict__ cf,
                                                                   float *__restrict__ keep, float xminf,
                                                                   double *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    // a cell's range and coefficient (page-locked memory) are loaded a cell ahead
    // without the water (31.0 -> 30.3 us with a cold L2; with it 32.0 -> 33.0: not there)
    int32_t next_lo = 0, next_hi = 0;
    float next_c = 0.0f;
    auto ahead = [&](int cell) {
        if (cell < n_cells) {
            next_lo = cell_off[cell];
            next_hi = cell_off[cell + 1];
            next_c = cf[cell];
        }
    };
    ahead(gw);
    for (int cell = gw; cell < n_cells; cell += nw) {
        const int32_t lo = next_lo, hi = next_hi;
        const float c = next_c;
        if constexpr (!WATER)
            ahead(cell + nw);
        double acc = 0.0;
        for (int32_t at = lo; at < hi; at += kCondItem) {
            const double w = condense_round<WATER>(xi + at, v + at, min(kCondItem, hi - at), c, xminf);
            acc = at == lo ? w : __dadd_rn(acc, w);
        }
        if (WATER && lane == 0)
            out[cell] = c < 0.0f ? 0.0 - acc : acc;
        if (KEEP && lane == 0)
            keep[cell] = c;
        if constexpr (WATER)
            ahead(cell + nw);
    }
}

// The same by a block of four warps per cell, a warp per 256 slots (cells of up to
// kCondByCell): where the cells are few and a warp alone would take several rounds
// one after the other.  The rounds' sums are added in the same order.  (us a call, by
// warps | by blocks, without the water: 1 cell of 1000 14.4 | 7.6, 300 of 1000 16.5 | 7.9,
// 1216 of 300 8.7 | 8.5, of 1000 16.6 | 10.3; but 2432 of 300 10.1 | 12.0.)
constexpr int kCondBlockNT = kCondByCell / kCondItem * 32;
template <bool WATER, bool KEEP>
__global__ void __launch_bounds__(kCondBlockNT) condense_block_kernel(const int32_t *__restrict__ cell_off, int32_t n_cells,
                                                                      const int64_t *__restrict__ xi,
                                                                      double *__restrict__ v, const float *__restrict__ cf,
                                                                      float *__restrict__ keep, float xminf,
                                                                      double *__restrict__ out)
{
    __shared__ double s_w[kCondBlockNT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int cell = blockIdx.x; cell < n_cells; cell += gridDim.x) {
        const int32_t lo = cell_off[cell], hi = cell_off[cell + 1];
        const float c = cf[cell];
        const int32_t at = lo + warp * kCondItem;
        const double w = at < hi ? condense_round<WATER>(xi + at, v + at, min(kCondItem, hi - at), c, xminf) : 0.0;
        if (KEEP && threadIdx.x == 0)
            keep[cell] = c;
        if constexpr (WATER) {
            if (lane == 0)
                s_w[warp] = w;
            __syncthreads();
            if (threadIdx.x == 0) {
                double acc = s_w[0];
                for (int k = 1; k < kCondBlockNT / 32 && lo + k * kCondItem < hi; ++k)
                    acc = __dadd_rn(acc, s_w[k]);
                out[cell] = c < 0.0f ? 0.0 - acc : acc;
            }
            __syncthreads();
        }
    }
}

// Cells above kCondByCell slots: work items of up to kCondItem slots.
template <bool WATER>
__global__ void __launch_bounds__(kCondNT) condense_kernel(const CondItem *__restrict__ items, int32_t n_items,
                                                           const int64_t *__restrict__ xi, double *__restrict__ v,
                                                           const float *__restrict__ cf, float *__restrict__ keep,
                                                           int32_t n_cells, float xminf, double *__restrict__ partial)
{
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    if (keep) // (null: not wanted) cells without an item too
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_cells; i += gridDim.x * blockDim.x)
            keep[i] = cf[i];
    for (int it = gw; it < n_items; it += nw) {
        const CondItem I = items[it];
        const float c = cf[I.cell];
        const double w = condense_round<WATER>(xi + I.begin, v + I.begin, I.n, c, xminf);
        if (WATER && lane == 0)
            partial[it] = c < 0.0f ? -w : w;
    }
}

// condensed[c] = the partial sums of cell c's items (one warp per cell)
__global__ void __launch_bounds__(kCondNT) condense_cells_kernel(const int32_t *__restrict__ item_start,
                                                                 int32_t n_cells, const double *__restrict__ partial,
                                                                 double *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int c = gw; c < n_cells; c += nw) {
        double acc = 0.0;
        for (int i = item_start[c] + lane; i < item_start[c + 1]; i += 32)
            acc = __dadd_rn(acc, partial[i]);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1)
            acc = __dadd_rn(acc, __shfl_down_sync(0xFFFFFFFFu, acc, d));
        if (lane == 0)
            out[c] = acc;
    }
}

void cond_release(sdm_ctx *ctx)
{
    if (!ctx->cond)
        return;
    CondBuffers &b = *ctx->cond;
    void *bufs[] = {b.items, b.item_start, b.partial, b.cond, b.cf};
    for (void *p : bufs)
        ctx->mem.put(p, 0);
    for (cudaEvent_t ev : b.cf_done)
        if (ev) {
            cudaEventSynchronize(ev);
            cudaEventDestroy(ev);
        }
    if (b.h_cf)
        cudaFreeHost(b.h_cf);
    delete ctx->cond;
    ctx->cond = nullptr;
}

// The work list of the current layout (rebuilt when the layout changes).
sdm_status cond_prepare(sdm_ctx *ctx)
{
    const int32_t nc = ctx->cfg.n_cells;
    if (!ctx->cond) {
        ctx->cond = new CondBuffers();
        CondBuffers &b = *ctx->cond;
        b.cond = static_cast<double *>(ctx->mem.get(sizeof(double) * nc));
        b.cf = static_cast<float *>(ctx->mem.get(sizeof(float) * nc));
        if (!b.cond || !b.cf) {
            cond_release(ctx);
            return fail(&ctx->error, SDM_ENOMEM, "condensation: device allocation failed");
        }
        cudaError_t e = cudaMallocHost(&b.h_cf, sizeof(float) * nc * kCondStage);
        for (cudaEvent_t &ev : b.cf_done)
            if (e == cudaSuccess)
                e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (e != cudaSuccess) {
            cudaGetLastError();
            cond_release(ctx);
            return fail(&ctx->error, SDM_ENOMEM, "condensation: page-locked staging failed");
        }
    }
    CondBuffers &b = *ctx->cond;
    if (ctx->largest_cell <= kCondByCell || b.layout_version == ctx->layout_version)
        return SDM_OK;
    if (!b.item_start) {
        b.item_start = static_cast<int32_t *>(ctx->mem.get(sizeof(int32_t) * (nc + 1)));
        if (!b.item_start)
            return fail(&ctx->error, SDM_ENOMEM, "condensation: device allocation failed");
    }
    std::vector<CondItem> items;
    std::vector<int32_t> start(nc + 1);
    for (int32_t c = 0; c < nc; ++c) {
        start[c] = (int32_t)items.size();
        const int32_t lo = ctx->h_cell_off[c], hi = ctx->h_cell_off[c + 1];
        for (int32_t o = lo; o < hi; o += kCondItem)
            items.push_back(CondItem{c, o, std::min(kCondItem, hi - o), 0});
    }
    start[nc] = (int32_t)items.size();
    ctx->mem.put(b.items, 0);
    ctx->mem.put(b.partial, 0);
    b.items = nullptr;
    b.partial = nullptr;
    b.n_items = (int32_t)items.size();
    b.layout_version = -1;
    const size_t ni = std::max<size_t>(1, items.size());
    b.items = static_cast<CondItem *>(ctx->mem.get(sizeof(CondItem) * ni));
    b.partial = static_cast<double *>(ctx->mem.get(sizeof(double) * ni));
    if (!b.items || !b.partial)
        return fail(&ctx->error, SDM_ENOMEM, "condensation: device allocation failed");
    cudaStream_t s = ctx->stream;
    CTX_CUDA(ctx, cudaMemcpyAsync(b.items, items.data(), sizeof(CondItem) * items.size(), cudaMemcpyHostToDevice, s));
    CTX_CUDA(ctx, cudaMemcpyAsync(b.item_start, start.data(), sizeof(int32_t) * (nc + 1), cudaMemcpyHostToDevice, s));
    // the host vectors go out of scope: wait for the copies of pageable memory
    CTX_CUDA(ctx, cudaStreamSynchronize(s));
    b.layout_version = ctx->layout_version;
    return SDM_OK;
}

} // namespace

extern "C" sdm_status sdm_condensation_step(sdm_ctx *ctx, const double *G, const double *s, double r_min,
                                            double *condensed, int condensed_on_device)
{
    NvtxRange nvtx_range("sdm_condensation_step");
    sdm_status st = ctx_usable(ctx);
    if (st != SDM_OK)
        return st;
    if (!ctx->has_attributes)
        return fail(&ctx->error, SDM_ESTATE, "sdm_set_attributes has not been called");
    if (!G || !s)
        return fail(&ctx->error, SDM_EINVAL, "G and s (one value per cell) are required");
    if (!(r_min >= 1e-9 && r_min <= 1e-3))
        return fail(&ctx->error, SDM_EINVAL, "r_min = %g outside [1e-9, 1e-3] m", r_min);
    const int32_t nc = ctx->cfg.n_cells;
    const double dt = ctx->cfg.dt;
    st = cond_prepare(ctx);
    if (st != SDM_OK)
        return st;
    CondBuffers &b = *ctx->cond;
    cudaStream_t cs = ctx->stream;
    float *field = b.h_cf + (size_t)b.stage * nc;
    // one pass without branches; what it finds wrong is named by a second
    int bad = 0;
    for (int32_t c = 0; c < nc; ++c) {
        const double g = ((2.0 * G[c]) * s[c]) * dt;
        bad |= (int)!(G[c] >= 0.0) | (int)!(s[c] >= -1.0) | (int)!(s[c] <= 1.0) | (int)!(std::fabs(g) <= 1e-6) |
               (int)!(G[c] <= 1.7976931348623157e308);
        field[c] = (float)g;
    }
    for (int32_t c = 0; bad && c < nc; ++c) {
        if (!(std::isfinite(G[c]) && G[c] >= 0.0) || !(std::isfinite(s[c]) && s[c] >= -1.0 && s[c] <= 1.0))
            return fail(&ctx->error, SDM_EINVAL, "cell %d: G = %g must be finite and >= 0, s = %g in [-1, 1]", c, G[c],
                        s[c]);
        if (!(std::fabs(((2.0 * G[c]) * s[c]) * dt) <= 1e-6))
            return fail(&ctx->error, SDM_EINVAL, "cell %d: |2 G s dt| = %g m^2 above 1e-6 m^2", c,
                        std::fabs(((2.0 * G[c]) * s[c]) * dt));
    }
    const bool changed = b.last < 0 || std::memcmp(field, b.h_cf + (size_t)b.last * nc, sizeof(float) * nc) != 0;
    const float *cf = changed ? field : b.cf;
    float *keep = changed ? b.cf : nullptr;
    const float xminf = (float)(r_min * r_min);
    const int cells_grid = (int)std::min<int64_t>((nc + kCondNT / 32 - 1) / (kCondNT / 32), 152 * 8);
    // the kernels write a device buffer themselves if it lies on eight bytes, else a copy does
    const bool direct = condensed && condensed_on_device && ((uintptr_t)condensed & 7) == 0;
    double *out = direct ? condensed : b.cond;
    if (ctx->largest_cell > kCondItem && ctx->largest_cell <= kCondByCell && nc <= kCondFewCells) {
        const auto kernel = condensed ? (changed ? condense_block_kernel<true, true> : condense_block_kernel<true, false>)
                                      : (changed ? condense_block_kernel<false, true> : condense_block_kernel<false, false>);
        kernel<<<nc, kCondBlockNT, 0, cs>>>(ctx->d_cell_off, nc, ctx->d_xi, ctx->d_v, cf, keep, xminf, out);
    } else if (ctx->largest_cell <= kCondByCell) {
        const auto kernel = condensed ? (changed ? condense_by_cell_kernel<true, true> : condense_by_cell_kernel<true, false>)
                                      : (changed ? condense_by_cell_kernel<false, true>
                                                 : condense_by_cell_kernel<false, false>);
        kernel<<<cells_grid, kCondNT, 0, cs>>>(ctx->d_cell_off, nc, ctx->d_xi, ctx->d_v, cf, keep, xminf, out);
    } else {
        const int grid = (int)std::min<int64_t>((b.n_items + kCondNT / 32 - 1) / (kCondNT / 32), 152 * 8);
        if (condensed) {
            condense_kernel<true><<<grid, kCondNT, 0, cs>>>(b.items, b.n_items, ctx->d_xi, ctx->d_v, cf, keep, nc,
                                                            xminf, b.partial);
            condense_cells_kernel<<<cells_grid, kCondNT, 0, cs>>>(b.item_start, nc, b.partial, out);
        } else {
            condense_kernel<false><<<grid, kCondNT, 0, cs>>>(b.items, b.n_items, ctx->d_xi, ctx->d_v, cf, keep, nc,
                                                             xminf, nullptr);
        }
    }
    CTX_CUDA(ctx, cudaGetLastError());
    if (changed) {
        CTX_CUDA(ctx, cudaEventRecord(b.cf_done[b.stage], cs));
        b.last = b.stage;
        b.stage = (b.stage + 1) % kCondStage;
        CTX_CUDA(ctx, cudaEventSynchronize(b.cf_done[b.stage])); // its kernel, three fields ago
    }
    if (condensed && condensed_on_device && !direct)
        CTX_CUDA(ctx, cudaMemcpyAsync(condensed, b.cond, sizeof(double) * nc, cudaMemcpyDeviceToDevice, cs));
    if (condensed && !condensed_on_device) {
        CTX_CUDA(ctx, cudaMemcpyAsync(condensed, b.cond, sizeof(double) * nc, cudaMemcpyDeviceToHost, cs));
        CTX_CUDA(ctx, cudaStreamSynchronize(cs));
    }
    return SDM_OK;
}

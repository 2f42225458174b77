// The library built for tests/test_gpu_give_up.py: two thirds of the record path's
// buckets wait as ever, every third one's wait gives up at its first look; and a
// way to the allocation-free step's array.
#define SDM_REC_POLLS(bucket) ((bucket) % 3 == 1 ? 0u : kWaitPolls)
#include "../paper_2103_17238_gb300/csrc/sdm_runtime.cu"

// Every byte of the allocation-free step's array set to one value: what no call may rely on.
extern "C" int give_up_fill_noalloc(int value)
{
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess ||
        cudaMemset(p, value, sizeof g_noalloc_scratch) != cudaSuccess)
        return 1;
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}

static __global__ void report_kernel(uint32_t *status, int which)
{
    if (which)
        OneSpread<1>{nullptr, SpreadCell{}, status}.overflow(SpreadCell{});
    else
        OneCell{nullptr, 0, 0, status}.give_up(0);
}

// As a kernel of that step reports a wait that gave up (0) or a full room (1).
extern "C" int give_up_report(int which)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64 || !g_na_wrong_dev[dev])
        return 1;
    report_kernel<<<1, 1>>>(g_na_wrong_dev[dev], which);
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}

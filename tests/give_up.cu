// The library built for tests/test_gpu_give_up.py: two thirds of the record path's
// buckets wait as ever, every third one's wait gives up at its first look.
#define SDM_REC_POLLS(bucket) ((bucket) % 3 == 1 ? 0u : kWaitPolls)
#include "../paper_2103_17238_gb300/csrc/sdm_runtime.cu"

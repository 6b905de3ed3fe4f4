// First kernel of a batch: control block, busy-until, statistics and counters to their state at the start.
#pragma once
#include "device_utils.cuh"

namespace hbf {

struct BeginArgs {
    BatchCtrl *ctrl; const DevState *state; const int64_t *busy; int64_t *busy_stage; hbf_die_stats_t *stats_stage; uint32_t *hist;
    uint32_t n_queues, n_dies; uint32_t *die_claims; const unsigned long long *claim_limit;
};

// 1,024 pairs of neighbouring records (n >= 2; blocks of 1,024 threads): are they out of order, and what span of time does this
// thread's pair show.  A batch that they show to be out of order is not attempted in order (an attempt that finds out by itself
// took 2.7 of the 8.2 ms of 40 M shuffled records).  One pair each: one multiprocessor takes 4 us longer to fetch four.
__device__ __forceinline__ bool begin_samples(const hbf_access_t *acc, uint64_t n, long long *lo, long long *hi) {
    const uint64_t *rec = reinterpret_cast<const uint64_t *>(acc + (uint64_t)threadIdx.x * (n - 1ull) / 1024ull);
    const int64_t v0 = (int64_t)ld_after(rec + 1), v1 = (int64_t)ld_after(rec + 4), up = __shfl_up_sync(0xffffffffu, v0, 1);
    *lo = min(v0, v1); *hi = max(v0, v1);
    return __syncthreads_or(v1 < v0 || ((threadIdx.x & 31) != 0 && v0 < up)) != 0;
}
__device__ __forceinline__ bool begin_refused(const DevState *state) {
    return state->poisoned || state->mode == HBF_MODE_SHUTDOWN || state->mode == HBF_MODE_SEVERE;
}
// one block.  run_sort: the sort path serves the batch; regrouped: the in-order kernels do, on the ordered copy
__device__ __forceinline__ void begin_batch(const BeginArgs &a, int run_sort, uint32_t regrouped) {
    const int tid = threadIdx.x;
    BatchCtrl *ctrl = a.ctrl;
    uint32_t *w = reinterpret_cast<uint32_t *>(ctrl);
    for (int i = tid; i < (int)(sizeof(BatchCtrl) / 4); i += blockDim.x) w[i] = 0u;
    __syncthreads();
    if (tid == 0) {
        int32_t mode = a.state->mode;
        ctrl->mode = mode; ctrl->q_ppm = a.state->q_ppm;
        if (a.state->q_ppm != 1000000) ctrl->div_q = make_div64((uint64_t)a.state->q_ppm);   // (a 128-bit division; nothing looks at it without scaling)
        ctrl->key_and = ~0ull;
        ctrl->run_sort = (uint32_t)run_sort; ctrl->regrouped = regrouped;
        if (a.state->poisoned) { ctrl->code = HBF_E_TIMEOUT; ctrl->skip = 1; }
        else if (mode == HBF_MODE_SHUTDOWN) { ctrl->code = HBF_E_LINK_SHUTDOWN; ctrl->skip = 1; }
        else if (mode == HBF_MODE_SEVERE) { ctrl->code = HBF_E_THROTTLED; ctrl->skip = 1; }
    }
    for (uint32_t r = tid; r < a.n_queues; r += blockDim.x) a.busy_stage[r] = a.busy[r];
    int64_t *s = reinterpret_cast<int64_t *>(a.stats_stage);
    for (uint32_t i = tid; i < a.n_dies * 6u; i += blockDim.x) s[i] = 0;
    for (int i = tid; i < kMaxPasses * kRadix; i += blockDim.x) a.hist[i] = 0u;
    if (a.die_claims)                                        // retention on: an in-order attempt that was handed over counted some
        for (uint32_t d = tid; d < a.n_dies; d += blockDim.x) a.die_claims[d] = 0u;
}

}  // namespace hbf

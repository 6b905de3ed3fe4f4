// First kernel of a batch: control block, busy-until, statistics and counters to their state at the start.
#pragma once
#include "device_utils.cuh"

namespace hbf {

struct BeginArgs {
    BatchCtrl *ctrl; const DevState *state; const int64_t *busy; int64_t *busy_stage; hbf_die_stats_t *stats_stage; uint32_t *hist;
    uint32_t n_queues, n_dies; uint32_t *die_claims; const unsigned long long *claim_limit;
    TileBalance *decides; float twice_from; uint64_t n; uint32_t page_shift; int64_t t_read_ns, t_prog_ns;   // see begin_load (decides: null, not asked)
    const RangeSnap *ranges; uint32_t unit_shift;            // see begin_units (0: not asked)
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

// How much of its span a batch fills, and with that whether its tiles are served twice at once (BatchCtrl::twice): the services of 1,024
// sampled records (a page's time per page they touch, as if all were modeled), the refresh quanta it claims, and what the queues
// are behind when it begins.  twice_from: from this load on it is (see twice_from); below, where the last batch that had to serve half of
// its tiles twice after all had about this load or less (streams that crowd on some queues at a time): a batch whose load is
// lower by a tenth is not, whatever came before it.  (While the choice went by the batches before alone, 200 M records without debt
// behind 200 M with claims took 3,140 us; 2,500 with the fix-up of before that, 2,270 now.)  One block of 1,024 threads, behind
// begin_batch; first, last: the batch's issue times; rec: this thread's sample.
__device__ __forceinline__ void begin_load(const BeginArgs &a, const uint64_t *rec, int64_t first, int64_t last) {
    __shared__ double s_work, s_behind;
    const int tid = threadIdx.x;
    if (tid == 0) s_work = s_behind = 0.0;
    __syncthreads();
    const uint64_t mask = (1ull << a.page_shift) - 1ull, bf = ld_after(rec + 2), pages = ((ld_after(rec) & mask) + (uint32_t)bf + mask) >> a.page_shift;
    double work = (double)pages * (double)(((bf >> 32) & 1u) ? a.t_prog_ns : a.t_read_ns), behind = 0.0;
    for (uint32_t q = tid; q < a.n_queues; q += blockDim.x) behind += (double)max((int64_t)0, a.busy[q] - first);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) { work += __shfl_xor_sync(0xffffffffu, work, o); behind += __shfl_xor_sync(0xffffffffu, behind, o); }
    if ((tid & 31) == 0) { atomicAdd(&s_work, work); atomicAdd(&s_behind, behind); }
    __syncthreads();
    if (tid != 0 || a.ctrl->skip) return;
    double ns = s_work * ((double)a.n / 1024.0);
    if (a.claim_limit) ns += (double)min((unsigned long long)a.n, *a.claim_limit) * (double)(a.t_read_ns + a.t_prog_ns);
    ns = ns * 1e6 / (double)a.ctrl->q_ppm + s_behind;
    const float load = (float)(ns / ((double)a.n_queues * (double)max((int64_t)1, last - first)));
    a.ctrl->load = load;
    if (load >= a.twice_from) a.ctrl->twice = 1u;
    else if (a.decides->twice_left > 0u && load >= 0.9f * a.decides->twice_load) { a.ctrl->twice = 1u; a.decides->twice_left -= 1u; }
}

// Does one of 1,024 sampled records reach over the end of its stripe unit?  Then the first pass is spared (a batch in which only others do is
// noticed by that pass).  One block of 1,024 threads, behind begin_batch; rec: this thread's sample.
__device__ __forceinline__ void begin_units(const BeginArgs &a, const uint64_t *rec) {
    const uint64_t addr = ld_after(rec), bf = ld_after(rec + 2), unit = 1ull << a.unit_shift;
    int g = 0;
    if (classify(*a.ranges, addr, (int64_t)ld_after(rec + 1), (uint32_t)bf, (uint32_t)(bf >> 32), &g) != HBF_ST_READY) return;
    const uint64_t off = a.ranges->media_offset[g] + (addr - a.ranges->base[g]);
    if ((off & (unit - 1ull)) + (uint32_t)bf > unit) a.ctrl->sample_crossed = 1u;
}

}  // namespace hbf

// Channel bus as a second queued stage (an extension; the library's own definition).  After the array stage, a read's data-out
// transfer queues on the bus of its channel in (array-done time, index) order and holds it for the transfer time; the read
// completes when the transfer does.  Programs are unchanged.
//   plan     how the array-done times spread (65,536 samples over 64 stretches): slices of time with about as many reads each,
//            682 per slice and channel
//   scatter  every read becomes a 16-byte entry (time, index, transfer) in the bucket of its slice and channel.  A block takes
//            4,096 records, puts their entries in bucket order in shared memory and writes them in runs: their times lie close
//            together, so that they fall into one or two slices
//   order    a block per bucket puts its entries in order (times spread over bins of shared memory, the place within a bin by
//            comparing), writes the completions and stalls of the reads that wait if the bus was idle before the bucket, and
//            leaves the bucket's map B -> max(B + S, M) and its first 16 entries
//   join     a block per channel: the bus before every bucket, from the maps; where it is busy, the first entries once more, up to
//            the one that ends as before: behind it nothing changes
//   redo     buckets in which the 16 do not reach that far, in full
// A bucket with more than three times the average sends the batch to the radix sort of (channel, time) in submit_kernels.cu.
// Bytes per read: 24 + 8 + 16, then 16 and the results that change.  32 M reads with the array stage: 4,112 us with the radix
// sort (five passes over 12 bytes, two gathers by sorted index), 1,645 in buckets; 20,011 reads 171 and 79.  What bounds it: scatter
// 418 us (memory and instructions in equal parts), order some 650 (instructions: 18 per read and lane; barriers).  A block that
// waited for the bus from the bucket before by look-back instead of assuming it idle: 1,245 us for that kernel; smaller buckets
// of a warp each, with look-back: 3,100.
#include <algorithm>

#include "bus.cuh"
#include "serve_terms.cuh"

namespace hbf {

// a read's channel, array-done time and transfer; false: not a modeled read.  late: the time has no place in 47 bits
struct BusRead { uint32_t channel, x; int64_t done; };
__device__ __forceinline__ bool bus_read(const hbf_access_t *__restrict__ acc, const int64_t *__restrict__ completion, uint64_t i, const RangeSnap &rs, const ModelParams &mp,
                                         const FastRange &fast, bool fast_ok, BusRead *r) {
    const uint64_t *rec = reinterpret_cast<const uint64_t *>(acc + i);
    const uint64_t addr = ld_after(rec), issue = ld_after(rec + 1), bf = ld_after(rec + 2);
    const int64_t comp = ld_after(completion + i);
    uint32_t die;
    if (fast_ok) {
        const Served s = serve_terms_fast(fast, mp, addr, (int64_t)issue, bf);
        if (s.st != HBF_ST_READY || s.op) return false;
        die = s.die; r->x = s.xfer;
        r->channel = die >> mp.die_shift;
    } else {
        int g = 0;
        if (classify(rs, addr, (int64_t)issue, (uint32_t)bf, (uint32_t)(bf >> 32), &g) != HBF_ST_READY || ((bf >> 32) & 1u)) return false;
        const Decoded d = decode(mp, rs.media_offset[g] + (addr - rs.base[g]), (uint32_t)bf);
        const Div64 one = make_div64(1);
        r->x = (uint32_t)service_terms(mp, (uint32_t)bf, d.npages, 0u, 1000000, one).xfer;      // the transfer does not depend on the throttle
        r->channel = d.die / mp.dies;
    }
    r->done = comp - (int64_t)r->x;                          // when the array is done with the read
    return true;
}

__device__ __forceinline__ uint32_t bus_stretch(int64_t t, int64_t lo, uint32_t shift, uint32_t *offset) {
    const uint64_t rel = t <= lo ? 0ull : (uint64_t)(t - lo);
    const uint32_t seg = (uint32_t)min((uint64_t)(kBusSegs - 1), rel >> shift);
    const uint64_t in = min(rel - ((uint64_t)seg << shift), ((uint64_t)1 << shift) - 1u);
    *offset = (uint32_t)(shift > 32u ? in >> (shift - 32u) : in);
    return seg;
}

// state to its start; the span of the array-done times from 2,048 records
__global__ void __launch_bounds__(1024)
k_bus_start(const hbf_access_t *__restrict__ acc, uint64_t n, const int64_t *__restrict__ completion, const RangeSnap *__restrict__ ranges, const __grid_constant__ ModelParams mp,
            const __grid_constant__ FastRange fast, int fast_ok, BatchCtrl *bc, const hbf_batch_result_t *result, const __grid_constant__ BusArgs b) {
    pdl_wait();
    pdl_trigger();
    const int tid = threadIdx.x;
    const uint64_t buckets = (uint64_t)b.slices * b.channels;
    for (uint64_t i = (uint64_t)blockIdx.x * 1024 + tid; i < buckets; i += (uint64_t)gridDim.x * 1024) b.cursor[i] = 0u;
    if (blockIdx.x != 0) return;
    __shared__ long long s_lo, s_hi;
    uint32_t *w = reinterpret_cast<uint32_t *>(bc), *p = reinterpret_cast<uint32_t *>(b.plan);
    for (int i = tid; i < (int)(sizeof(BatchCtrl) / 4); i += 1024) w[i] = 0u;
    for (int i = tid; i < (int)(sizeof(BusPlan) / 4); i += 1024) p[i] = 0u;
    if (tid == 0) { s_lo = INT64_MAX; s_hi = INT64_MIN; }
    __syncthreads();
    const bool refused = result->code != HBF_OK;             // a refused batch has no second stage
    long long lo = INT64_MAX, hi = INT64_MIN;
    if (!refused && b.slices) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            BusRead r;
            const uint64_t i = (uint64_t)(2 * tid + k) * n / 2048u;
            if (bus_read(acc, completion, i, *ranges, mp, fast, fast_ok != 0, &r)) { lo = min(lo, (long long)r.done); hi = max(hi, (long long)r.done); }
        }
    }
    for (int o = 16; o > 0; o >>= 1) { lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
    if ((tid & 31) == 0 && lo <= hi) { atomicMin(&s_lo, lo); atomicMax(&s_hi, hi); }
    __syncthreads();
    if (tid == 0) {
        lo = s_lo; hi = s_hi;
        if (lo > hi) { lo = 0; hi = 1; }
        const int64_t margin = (hi - lo) / 128 + 1;
        const uint64_t span = (uint64_t)(hi - lo + 2 * margin);
        uint32_t shift = 0;
        while (((uint64_t)(kBusSegs - 1) << shift) < span) ++shift;
        b.plan->lo = lo - margin; b.plan->shift = shift;
        b.plan->overflow = b.slices ? 0u : 1u;
        bc->max_completion_ns = INT64_MIN;
        bc->skip = refused ? 1u : 0u;
    }
}

__global__ void __launch_bounds__(1024)
k_bus_plan(const hbf_access_t *__restrict__ acc, uint64_t n, const int64_t *__restrict__ completion, const RangeSnap *__restrict__ ranges, const __grid_constant__ ModelParams mp,
           const __grid_constant__ FastRange fast, int fast_ok, const BatchCtrl *bc, const __grid_constant__ BusArgs b) {
    __shared__ uint32_t s_hist[kBusSegs], s_top[kBusSegs], s_below[kBusSegs], s_last;
    pdl_wait();
    pdl_trigger();
    if (bc->skip || b.slices == 0u) return;
    const int tid = threadIdx.x;
    if (tid < (int)kBusSegs) { s_hist[tid] = 0u; s_top[tid] = 0u; s_below[tid] = 0u; }
    __syncthreads();
    const uint64_t samples = min(n, (uint64_t)kBusSamples), s = (uint64_t)blockIdx.x * 1024 + tid;
    BusRead r;
    if (s < samples && bus_read(acc, completion, s * n / samples, *ranges, mp, fast, fast_ok != 0, &r)) {
        uint32_t off;
        const uint32_t seg = bus_stretch(r.done, b.plan->lo, b.plan->shift, &off);
        atomicAdd(&s_hist[seg], 1u); atomicMax(&s_top[seg], off); atomicMax(&s_below[seg], ~off);
    }
    __syncthreads();
    if (tid < (int)kBusSegs && s_hist[tid]) { atomicAdd(&b.plan->hist[tid], s_hist[tid]); atomicMax(&b.plan->top[tid], s_top[tid]); atomicMax(&b.plan->below[tid], s_below[tid]); }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&b.plan->blocks, 1u) == gridDim.x - 1u ? 1u : 0u;
    __syncthreads();
    if (!s_last || tid >= 32) return;
    __threadfence();
    const uint64_t whole = (uint64_t)1 << min(b.plan->shift, 32u);
    uint32_t h[2] = {__ldcg(&b.plan->hist[2 * tid]), __ldcg(&b.plan->hist[2 * tid + 1])};
    uint32_t inc = h[0] + h[1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (tid >= o) inc += t; }
    const uint64_t total = max(1u, __shfl_sync(0xffffffffu, inc, 31)), parts = (uint64_t)b.slices << 8;
    uint64_t before = inc - h[0] - h[1];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint32_t seg = 2 * tid + k;
        // the part of the stretch that holds its samples, and 16 samples' share more on both sides
        uint64_t a = 0, z = whole - 1u;
        if (h[k]) {
            const uint64_t s0 = (uint32_t)~__ldcg(&b.plan->below[seg]), s1 = __ldcg(&b.plan->top[seg]), more = (s1 - s0) * 16u / h[k] + 1u;
            a = s0 > more ? s0 - more : 0u; z = min(z, s1 + more);
        }
        const uint64_t from = before * parts / total, to = (before + h[k]) * parts / total;
        b.plan->first[seg] = (uint32_t)a; b.plan->last[seg] = (uint32_t)z; b.plan->cum[seg] = from;
        b.plan->mul[seg] = ((to - from) << 32) / (z - a + 1u);
        before += h[k];
    }
}

constexpr int kBsThreads = 512, kBsItems = 8, kBsChunk = kBsThreads * kBsItems;
constexpr uint32_t kBsSlots = 2048;                         // buckets that a block keeps apart at a time
constexpr size_t kBsSmem = (size_t)kBsChunk * 18 + (size_t)kBsSlots * 8;
// an entry: done (47 bits) and the low 17 bits of the transfer; index and the rest of it
__device__ __forceinline__ ulonglong2 bus_pack(int64_t done, uint32_t x, uint32_t idx) {
    return make_ulonglong2((uint64_t)done | ((uint64_t)(x & 0x1ffffu) << 47), (uint64_t)idx | ((uint64_t)(x >> 17) << 32));
}
constexpr uint64_t kBusDoneMask = (1ull << 47) - 1ull;

__global__ void __launch_bounds__(kBsThreads, 2)
k_bus_scatter(const hbf_access_t *__restrict__ acc, uint64_t n, const int64_t *__restrict__ completion, const RangeSnap *__restrict__ ranges, const __grid_constant__ ModelParams mp,
              const __grid_constant__ FastRange fast, int fast_ok, BatchCtrl *bc, const __grid_constant__ BusArgs b) {
    extern __shared__ __align__(16) unsigned char bus_smem[];
    ulonglong2 *s_entry = reinterpret_cast<ulonglong2 *>(bus_smem);           // [kBsChunk] by bucket
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_entry + kBsChunk);       // [kBsSlots] entries of a bucket, then where they begin here
    uint32_t *s_delta = s_cnt + kBsSlots;                                     // [kBsSlots] from the place here to the place in the bucket
    uint16_t *s_slot = reinterpret_cast<uint16_t *>(s_delta + kBsSlots);      // [kBsChunk] an entry's bucket
    __shared__ uint64_t s_cum[kBusSegs], s_mul[kBusSegs];
    __shared__ uint32_t s_first[kBusSegs], s_last[kBusSegs], s_w[kBsThreads / 32], s_min;
    pdl_wait();
    pdl_trigger();
    if (bc->skip || b.slices == 0u) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < (int)kBusSegs) { s_cum[tid] = b.plan->cum[tid]; s_mul[tid] = b.plan->mul[tid]; s_first[tid] = b.plan->first[tid]; s_last[tid] = b.plan->last[tid]; }
    const int64_t lo = b.plan->lo;
    const uint32_t shift = b.plan->shift, channels = b.channels, keep = kBsSlots / channels * channels;
    bool late = false;
    for (uint64_t chunk = blockIdx.x; chunk * kBsChunk < n; chunk += gridDim.x) {
        __syncthreads();                                     // the chunk before is written
        for (uint32_t e = tid; e < kBsSlots; e += kBsThreads) s_cnt[e] = 0u;
        if (tid == 0) s_min = 0xffffffffu;
        int64_t done[kBsItems]; uint32_t x[kBsItems], slot[kBsItems];         // slot: slice and channel first, 0xffffffff: none
        __syncthreads();
        uint32_t least = 0xffffffffu;
#pragma unroll
        for (int k = 0; k < kBsItems; ++k) {
            const uint64_t i = chunk * kBsChunk + (uint64_t)k * kBsThreads + tid;
            BusRead r;
            slot[k] = 0xffffffffu;
            if (i < n && bus_read(acc, completion, i, *ranges, mp, fast, fast_ok != 0, &r)) {
                done[k] = r.done; x[k] = r.x;
                if (r.done < 0 || r.done >= HBF_ISSUE_LIMIT) late = true;
                else {
                    uint32_t off;
                    const uint32_t seg = bus_stretch(r.done, lo, shift, &off), a = s_first[seg];
                    const uint64_t pos = s_cum[seg] + (((uint64_t)(min(max(off, a), s_last[seg]) - a) * s_mul[seg]) >> 32);
                    const uint32_t slice = (uint32_t)min((uint64_t)(b.slices - 1u), pos >> 8);
                    least = min(least, slice);
                    slot[k] = slice * channels + r.channel;  // (below 2^32: there are fewer buckets than records)
                }
            }
        }
        least = __reduce_min_sync(0xffffffffu, least);
        if (lane == 0) atomicMin(&s_min, least);
        __syncthreads();
        const uint32_t base = s_min == 0xffffffffu ? 0u : s_min * channels;
        uint32_t rank[kBsItems];
#pragma unroll
        for (int k = 0; k < kBsItems; ++k) {
            if (slot[k] == 0xffffffffu) continue;
            if (slot[k] - base < keep) rank[k] = atomicAdd(&s_cnt[slot[k] - base], 1u);
            else {                                           // times far apart: by itself
                const uint32_t at = atomicAdd(&b.cursor[slot[k]], 1u);
                if (at < b.cap) b.entries[(uint64_t)slot[k] * b.cap + at] = bus_pack(done[k], x[k], (uint32_t)(chunk * kBsChunk + (uint64_t)k * kBsThreads + tid));
                else b.plan->overflow = 1u;
                slot[k] = 0xffffffffu;
            }
        }
        __syncthreads();
        uint32_t total;
        {                                                    // where every bucket's entries begin here and there
            constexpr int kPer = kBsSlots / kBsThreads;
            uint32_t v[kPer], sum = 0;
#pragma unroll
            for (int k = 0; k < kPer; ++k) { v[k] = s_cnt[tid * kPer + k]; sum += v[k]; }
            uint32_t inc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
            if (lane == 31) s_w[warp] = inc;
            uint32_t at[kPer];
#pragma unroll
            for (int k = 0; k < kPer; ++k) at[k] = v[k] ? atomicAdd(&b.cursor[base + tid * kPer + k], v[k]) : 0u;
            __syncthreads();
            const uint32_t ws = lane < kBsThreads / 32 ? s_w[lane] : 0u;
            uint32_t run = inc - sum + __reduce_add_sync(0xffffffffu, lane < warp ? ws : 0u);
            total = __reduce_add_sync(0xffffffffu, ws);
#pragma unroll
            for (int k = 0; k < kPer; ++k) { s_cnt[tid * kPer + k] = run; s_delta[tid * kPer + k] = at[k] - run; run += v[k]; }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kBsItems; ++k) {
            if (slot[k] == 0xffffffffu) continue;
            const uint32_t q = slot[k] - base, j = s_cnt[q] + rank[k];
            s_entry[j] = bus_pack(done[k], x[k], (uint32_t)(chunk * kBsChunk + (uint64_t)k * kBsThreads + tid));
            s_slot[j] = (uint16_t)q;
        }
        __syncthreads();
        for (uint32_t j = tid; j < total; j += kBsThreads) {
            const uint32_t q = s_slot[j], at = j + s_delta[q];
            if (at < b.cap) b.entries[(uint64_t)(base + q) * b.cap + at] = s_entry[j];
            else b.plan->overflow = 1u;
        }
    }
    if (late) atomicExch(&bc->code, (int)HBF_E_INVAL);      // an array-done time beyond its 47 bits
}

constexpr int kBaThreads = 256, kBaBlocks = 4;               // (512 x 2 and 341 to 1,365 reads per bucket: 3 to 8 % slower at 32 M or at 20,000)
constexpr uint32_t kBaBins = kBusCap;
constexpr int kBaItems = kBusCap / kBaThreads;
constexpr size_t kBaSmem = (size_t)kBusCap * 16 + (size_t)kBaBins * 4;
static_assert(kBaItems == 8, "two words of four bins per thread");
__device__ __forceinline__ int64_t entry_done(const ulonglong2 &e) { return (int64_t)(e.x & kBusDoneMask); }
__device__ __forceinline__ int64_t entry_xfer(const ulonglong2 &e) { return (int64_t)((e.x >> 47) | ((e.y >> 32) << 17)); }

// REDO = false: the shares of the grid, in order.  REDO = true: the buckets of the list, with the bus before them known.
template <bool REDO>
__global__ void __launch_bounds__(kBaThreads, kBaBlocks)
k_bus_order(BatchCtrl *bc, const __grid_constant__ BusArgs b, int64_t *__restrict__ completion, int64_t *__restrict__ stall) {
    extern __shared__ __align__(16) unsigned char bus_smem[];
    ulonglong2 *s_entry = reinterpret_cast<ulonglong2 *>(bus_smem);           // [kBusCap]
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_entry + kBusCap);        // [kBaBins]
    constexpr int kWarps = kBaThreads / 32;
    __shared__ unsigned long long s_min[kWarps], s_max[kWarps];
    __shared__ uint32_t s_w[kWarps];
    __shared__ BusState s_map[kWarps];
    pdl_wait();
    pdl_trigger();
    if (bc->skip || bc->code != HBF_OK || b.plan->overflow) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t count = REDO ? b.plan->redo : b.slices * b.channels;
    long long moved = 0, max_c = INT64_MIN;
    for (uint32_t turn = blockIdx.x; turn < count; turn += gridDim.x) {
        const uint32_t bucket = REDO ? b.redo[turn] : turn;
        const uint32_t m = min(__ldcg(&b.cursor[bucket]), b.cap);
        ulonglong2 v[kBaItems]; uint32_t bin[kBaItems];
        unsigned long long mn = ~0ull, mx = 0ull;
#pragma unroll
        for (int k = 0; k < kBaItems; ++k) {
            if (k * kBaThreads >= m) break;
            if (k * kBaThreads + tid < m) v[k] = __ldcs(b.entries + (uint64_t)bucket * b.cap + k * kBaThreads + tid);
        }
        __syncthreads();                                     // the bucket before is done with
#pragma unroll
        for (uint32_t e = 0; e < kBaBins; e += 4 * kBaThreads) *reinterpret_cast<uint4 *>(s_cnt + e + tid * 4) = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int k = 0; k < kBaItems; ++k) {
            if (k * kBaThreads >= m) break;
            if (k * kBaThreads + tid < m) { const unsigned long long d = v[k].x & kBusDoneMask; mn = min(mn, d); mx = max(mx, d); }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o)); mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o)); }
        if (lane == 0) { s_min[warp] = mn; s_max[warp] = mx; }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kWarps; ++w) { mn = min(mn, s_min[w]); mx = max(mx, s_max[w]); }
        const uint64_t t0 = mn, wide = m ? mx - mn : 0ull;
        const uint32_t sh = wide >> 32 ? 32u - (uint32_t)__clz((int)(wide >> 32)) : 0u;
        const float scale = (float)kBaBins * 0.999f / ((float)(uint32_t)(wide >> sh) + 1.f);   // (where a bin ends need not be exact, only the same for all)
#pragma unroll
        for (int k = 0; k < kBaItems; ++k) {
            if (k * kBaThreads >= m) break;
            if (k * kBaThreads + tid < m) {
                const uint32_t d = min(kBaBins - 1u, (uint32_t)((float)(uint32_t)(((v[k].x & kBusDoneMask) - t0) >> sh) * scale));
                bin[k] = d | (atomicAdd(&s_cnt[d], 1u) << 16);
            }
        }
        __syncthreads();
        {                                                    // exclusive scan of the bins, eight per thread
            constexpr uint32_t kPer = kBaBins / kBaThreads;
            uint32_t c[kPer], sum = 0;
#pragma unroll
            for (uint32_t k = 0; k < kPer; k += 4) {
                const uint4 q = *reinterpret_cast<const uint4 *>(s_cnt + tid * kPer + k);
                c[k] = q.x; c[k + 1] = q.y; c[k + 2] = q.z; c[k + 3] = q.w; sum += q.x + q.y + q.z + q.w;
            }
            uint32_t inc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
            if (lane == 31) s_w[warp] = inc;
            __syncthreads();
            uint32_t run = inc - sum;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) run += w < warp ? s_w[w] : 0u;
#pragma unroll
            for (uint32_t k = 0; k < kPer; k += 4) {
                uint4 q;
                q.x = run; q.y = q.x + c[k]; q.z = q.y + c[k + 1]; q.w = q.z + c[k + 2]; run = q.w + c[k + 3];
                *reinterpret_cast<uint4 *>(s_cnt + tid * kPer + k) = q;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kBaItems; ++k) {
            if (k * kBaThreads >= m) break;
            if (k * kBaThreads + tid < m) s_entry[s_cnt[bin[k] & 0xffffu] + (bin[k] >> 16)] = v[k];
        }
        __syncthreads();
        // an entry's place within its bin: how many of the bin's come before it (rarely more than three in all; reads whose array
        // is done at the very same time share a bin, however many they are)
#pragma unroll
        for (int k = 0; k < kBaItems; ++k) {
            if (k * kBaThreads >= m) break;
            if (k * kBaThreads + tid < m) {
                const uint32_t d = bin[k] & 0xffffu, from = s_cnt[d], to = d + 1u < kBaBins ? s_cnt[d + 1u] : m;
                uint32_t before = 0;
                if (to - from > 1u) {
                    const uint64_t t = v[k].x & kBusDoneMask; const uint32_t idx = (uint32_t)v[k].y;
                    for (uint32_t q = from; q < to; ++q) {
                        const ulonglong2 o = s_entry[q];
                        const uint64_t ot = o.x & kBusDoneMask;
                        before += ot < t || (ot == t && (uint32_t)o.y < idx) ? 1u : 0u;
                    }
                }
                bin[k] = from + before;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kBaItems; ++k) {
            if (k * kBaThreads >= m) break;
            if (k * kBaThreads + tid < m) s_entry[bin[k]] = v[k];
        }
        __syncthreads();
        // every thread's stretch of the ordered entries as one map, and what lies before it in the bucket
        const uint32_t per = (m + kBaThreads - 1u) / kBaThreads, j0 = min(m, tid * per), j1 = min(m, j0 + per);
        int64_t S = 0, M = kNegInf;
        for (uint32_t j = j0; j < j1; ++j) {
            const ulonglong2 e = s_entry[j];
            const int64_t x = entry_xfer(e);
            S += x; M = max(M, entry_done(e)) + x;           // (kNegInf + x stays far below any time)
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t ps = __shfl_up_sync(0xffffffffu, S, o), pm = __shfl_up_sync(0xffffffffu, M, o);
            if (lane >= o) { M = max(pm + S, M); S += ps; }
        }
        if (lane == 31) { s_map[warp].S = S; s_map[warp].M = M; }
        int64_t rs = __shfl_up_sync(0xffffffffu, S, 1), rm = __shfl_up_sync(0xffffffffu, M, 1);
        if (lane == 0) { rs = 0; rm = kNegInf; }
        __syncthreads();
        int64_t ws = 0, wm = kNegInf;                        // the warps before this one
        for (int w = 0; w < warp; ++w) { wm = max(wm + s_map[w].S, s_map[w].M); ws += s_map[w].S; }
        if (!REDO) {
            if (tid == kBaThreads - 1) { BusState t; t.S = ws + S; t.M = max(wm + S, M); b.state[bucket] = t; }
            if (tid < (int)min(m, kBusHead)) b.heads[(uint64_t)bucket * kBusHead + tid] = s_entry[tid];
        }
        int64_t bus = max(wm + rs, rm), real = REDO ? max(b.state[bucket].M + ws + rs, bus) : 0;
        for (uint32_t j = j0; j < j1; ++j) {
            const ulonglong2 e = s_entry[j];
            const int64_t x = entry_xfer(e), done = entry_done(e);
            bus = max(bus, done) + x;
            if (REDO) real = max(real, done) + x;
            const int64_t end = REDO ? real : bus, had = REDO ? bus : done + x;
            if (end != had) {                                // the transfer waits for the bus: completion and stall move by the wait
                const uint32_t idx = (uint32_t)e.y;
                completion[idx] = end;
                atomicAdd(reinterpret_cast<unsigned long long *>(stall + idx), (unsigned long long)(end - had));   // (nothing waits for it)
                moved += end - had; max_c = max(max_c, (long long)end);
            }
        }
    }
    moved = warp_sum(moved); max_c = warp_max(max_c);
    if (lane == 0) {
        if (moved) atomicAdd((unsigned long long *)&bc->modeled_ns, (unsigned long long)moved);
        if (max_c != INT64_MIN) atomicMax(&bc->max_completion_ns, max_c);
    }
}

// a block per channel (see above); what it leaves to be gone over again goes to the list
constexpr int kBjThreads = 512;
__global__ void __launch_bounds__(kBjThreads)
k_bus_join(BatchCtrl *bc, const __grid_constant__ BusArgs b, int64_t *__restrict__ completion, int64_t *__restrict__ stall) {
    __shared__ BusState s_map[kBjThreads / 32];
    pdl_wait();
    pdl_trigger();
    if (bc->skip || bc->code != HBF_OK || b.plan->overflow) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    long long moved = 0, max_c = INT64_MIN;
    for (uint32_t channel = blockIdx.x; channel < b.channels; channel += gridDim.x) {
        const uint32_t per = (b.slices + kBjThreads - 1u) / kBjThreads, lo = min(b.slices, tid * per), hi = min(b.slices, lo + per);
        int64_t S = 0, M = kNegInf;
        for (uint32_t s = lo; s < hi; ++s) { const BusState t = b.state[(uint64_t)s * b.channels + channel]; M = max(M + t.S, t.M); S += t.S; }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t ps = __shfl_up_sync(0xffffffffu, S, o), pm = __shfl_up_sync(0xffffffffu, M, o);
            if (lane >= o) { M = max(pm + S, M); S += ps; }
        }
        __syncthreads();
        if (lane == 31) { s_map[warp].S = S; s_map[warp].M = M; }
        int64_t rs = __shfl_up_sync(0xffffffffu, S, 1), rm = __shfl_up_sync(0xffffffffu, M, 1);
        if (lane == 0) { rs = 0; rm = kNegInf; }
        __syncthreads();
        int64_t bus = b.busy[channel];
        for (int w = 0; w < warp; ++w) bus = max(bus + s_map[w].S, s_map[w].M);
        bus = max(bus + rs, rm);
        for (uint32_t s = lo; s < hi; ++s) {                 // the bus before every bucket of this thread
            const uint32_t bucket = s * b.channels + channel, m = min(b.cursor[bucket], b.cap), h = min(m, kBusHead);
            const BusState t = b.state[bucket];
            const ulonglong2 *head = b.heads + (uint64_t)bucket * kBusHead;
            int64_t real = bus, had = kNegInf;
            uint32_t same = 0;                               // the first entry that ends as if the bus had been idle
            for (; same < h; ++same) {
                const ulonglong2 e = head[same];
                had = max(had, entry_done(e)) + entry_xfer(e); real = max(real, entry_done(e)) + entry_xfer(e);
                if (real == had) break;
            }
            if (same == h && m > h) { b.state[bucket].M = bus; b.redo[atomicAdd(&b.plan->redo, 1u)] = bucket; }
            else {
                real = bus; had = kNegInf;
                for (uint32_t j = 0; j < same; ++j) {
                    const ulonglong2 e = head[j];
                    had = max(had, entry_done(e)) + entry_xfer(e); real = max(real, entry_done(e)) + entry_xfer(e);
                    completion[(uint32_t)e.y] = real; stall[(uint32_t)e.y] += real - had;
                    moved += real - had; max_c = max(max_c, (long long)real);
                }
            }
            bus = max(bus + t.S, t.M);
        }
        __syncthreads();                                     // (every thread has read the bus as the batch found it)
        if (lo < hi && hi == b.slices) b.busy[channel] = bus;
    }
    moved = warp_sum(moved); max_c = warp_max(max_c);
    if (lane == 0) {
        if (moved) atomicAdd((unsigned long long *)&bc->modeled_ns, (unsigned long long)moved);
        if (max_c != INT64_MIN) atomicMax(&bc->max_completion_ns, max_c);
    }
}

cudaError_t launch_bus_buckets(const SubmitArgs &a, BatchCtrl *bc, int64_t *bus_busy, cudaStream_t st) {
    const uint64_t n = a.n;
    const BusArgs b = bus_args(n, a.mp.channels, a.ws, bc, bus_busy);
    const int fast_ok = fast_geom_ok(a.fast, a.mp) ? 1 : 0;
    cudaError_t e = ensure_dyn_smem((const void *)k_bus_scatter, kBsSmem);
    if (e == cudaSuccess) e = ensure_dyn_smem((const void *)k_bus_order<false>, kBaSmem);
    if (e == cudaSuccess) e = ensure_dyn_smem((const void *)k_bus_order<true>, kBaSmem);
    const uint64_t buckets = (uint64_t)b.slices * b.channels;
    const unsigned order_grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(buckets, (uint64_t)a.sm_count * kBaBlocks));
    if (e == cudaSuccess)
        e = launch_first(a.plain_next, k_bus_start, (unsigned)std::min<uint64_t>((buckets + 1023) / 1024 + 1, (uint64_t)a.sm_count), 1024, 0, st, a.acc, n, (const int64_t *)a.completion,
                         a.ranges, a.mp, a.fast, fast_ok, bc, (const hbf_batch_result_t *)a.result, b);
    if (e == cudaSuccess)
        e = launch_pdl(k_bus_plan, (unsigned)((std::min<uint64_t>(n, kBusSamples) + 1023) / 1024), 1024, 0, st, a.acc, n, (const int64_t *)a.completion, a.ranges, a.mp, a.fast, fast_ok,
                       (const BatchCtrl *)bc, b);
    if (e == cudaSuccess)
        e = launch_pdl(k_bus_scatter, (unsigned)std::min<uint64_t>((n + kBsChunk - 1) / kBsChunk, (uint64_t)a.sm_count * 2), kBsThreads, kBsSmem, st, a.acc, n,
                       (const int64_t *)a.completion, a.ranges, a.mp, a.fast, fast_ok, bc, b);
    if (e == cudaSuccess)
        e = launch_pdl(k_bus_order<false>, order_grid, kBaThreads, kBaSmem, st, bc, b, a.completion, a.stall);
    if (e == cudaSuccess) e = launch_pdl(k_bus_join, std::min<unsigned>(std::max(1u, b.channels), (unsigned)a.sm_count), kBjThreads, 0, st, bc, b, a.completion, a.stall);
    if (e == cudaSuccess) e = launch_pdl(k_bus_order<true>, order_grid, kBaThreads, kBaSmem, st, bc, b, a.completion, a.stall);
    g_kernel_launches += 6;
    return e;
}

}  // namespace hbf

// Channel bus as a second queued stage (an extension; the library's own definition).  After the array stage, a read's data-out
// transfer queues on the bus of its channel in (array-done time, index) order and holds it for the transfer time; the read
// completes when the transfer does.  Programs are unchanged.
//   plan     how the array-done times spread (65,536 samples over 64 stretches): slices of time with about as many reads each,
//            1,365 per slice and channel
//   scatter  every read becomes a 16-byte entry (time, index, transfer) in the bucket of its slice and channel.  A block takes
//            4,096 records, puts their entries in bucket order in shared memory and writes them in runs: their times lie close
//            together, so that they fall into one or two slices
//   apply    a block per bucket puts its entries in order (times spread over 4,096 bins of shared memory, the place within a bin
//            by comparing), composes their maps B -> max(B, D) + x, takes the bus as the slice before left it (look-back over the
//            buckets of the channel), and writes the completions and stalls of the reads that waited
// A bucket with more than three times the average sends the batch to the radix sort of (channel, time) in submit_kernels.cu.
// Bytes per read: 24 + 8 + 16, then 16 and the results that change.  32 M reads with the array stage: 4,112 us with the radix
// sort (five passes over 12 bytes, two gathers by sorted index), 2,217 in buckets.
#include <algorithm>

#include "bus.cuh"
#include "serve_terms.cuh"

namespace hbf {

// a read's channel, array-done time and transfer; false: not a modeled read.  late: the time has no place in 47 bits
struct BusRead { uint32_t channel, x; int64_t done; };
__device__ __forceinline__ bool bus_read(const hbf_access_t *__restrict__ acc, const int64_t *__restrict__ completion, uint64_t i, const RangeSnap &rs, const ModelParams &mp,
                                         const FastRange &fast, bool fast_ok, BusRead *r) {
    const uint64_t *rec = reinterpret_cast<const uint64_t *>(acc + i);
    const uint64_t addr = __ldg(rec), issue = __ldg(rec + 1), bf = __ldg(rec + 2);
    const int64_t comp = __ldg(reinterpret_cast<const long long *>(completion + i));
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
    for (uint64_t i = (uint64_t)blockIdx.x * 1024 + tid; i < buckets; i += (uint64_t)gridDim.x * 1024) { b.cursor[i] = 0u; b.state[i].flag = 0u; }
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

constexpr int kBaThreads = 512;
constexpr uint32_t kBaBins = 4096;
constexpr int kBaItems = kBusCap / kBaThreads;
constexpr size_t kBaSmem = (size_t)kBusCap * 16 + (size_t)kBaBins * 4;

__global__ void __launch_bounds__(kBaThreads, 2)
k_bus_buckets(BatchCtrl *bc, const __grid_constant__ BusArgs b, int64_t *__restrict__ completion, int64_t *__restrict__ stall) {
    extern __shared__ __align__(16) unsigned char bus_smem[];
    ulonglong2 *s_entry = reinterpret_cast<ulonglong2 *>(bus_smem);           // [kBusCap]
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_entry + kBusCap);        // [kBaBins]
    __shared__ unsigned long long s_min, s_max;
    __shared__ uint32_t s_w[kBaThreads / 32], s_bucket;
    __shared__ BusMap s_map[kBaThreads / 32];
    __shared__ int64_t s_carry;
    __shared__ int s_ok;
    pdl_wait();
    pdl_trigger();
    if (bc->skip || bc->code != HBF_OK || b.plan->overflow) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t buckets = b.slices * b.channels;
    long long moved = 0, max_c = INT64_MIN;
    for (;;) {
        __syncthreads();
        if (tid == 0) { s_bucket = atomicAdd(&b.plan->ticket, 1u); s_min = ~0ull; s_max = 0ull; s_ok = 1; }
        for (uint32_t e = tid; e < kBaBins; e += kBaThreads) s_cnt[e] = 0u;
        __syncthreads();
        const uint32_t bucket = s_bucket;                    // (in order: what a bucket waits for is in the hands of blocks that run)
        if (bucket >= buckets) break;
        const uint32_t m = min(__ldcg(&b.cursor[bucket]), b.cap);
        ulonglong2 v[kBaItems]; uint32_t bin[kBaItems];
        unsigned long long mn = ~0ull, mx = 0ull;
#pragma unroll
        for (int k = 0; k < kBaItems; ++k) {
            const uint32_t e = k * kBaThreads + tid;
            if (e < m) v[k] = __ldcs(b.entries + (uint64_t)bucket * b.cap + e);
        }
#pragma unroll
        for (int k = 0; k < kBaItems; ++k)
            if (k * kBaThreads + tid < m) { const unsigned long long d = v[k].x & kBusDoneMask; mn = min(mn, d); mx = max(mx, d); }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o)); mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o)); }
        if (lane == 0 && mn <= mx) { atomicMin(&s_min, mn); atomicMax(&s_max, mx); }
        __syncthreads();
        const uint64_t t0 = s_min, wide = m ? s_max - t0 : 0ull;
        const uint32_t sh = wide >> 32 ? 32u - (uint32_t)__clz((int)(wide >> 32)) : 0u;
        const uint64_t mul = ((uint64_t)kBaBins << 32) / ((wide >> sh) + 1ull);
#pragma unroll
        for (int k = 0; k < kBaItems; ++k)
            if (k * kBaThreads + tid < m) {
                const uint32_t d = (uint32_t)(((((v[k].x & kBusDoneMask) - t0) >> sh) * mul) >> 32);
                bin[k] = d | (atomicAdd(&s_cnt[d], 1u) << 16);
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
            uint32_t run = inc - sum + __reduce_add_sync(0xffffffffu, lane < warp ? s_w[lane] : 0u);
#pragma unroll
            for (uint32_t k = 0; k < kPer; k += 4) {
                uint4 q;
                q.x = run; q.y = q.x + c[k]; q.z = q.y + c[k + 1]; q.w = q.z + c[k + 2]; run = q.w + c[k + 3];
                *reinterpret_cast<uint4 *>(s_cnt + tid * kPer + k) = q;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kBaItems; ++k)
            if (k * kBaThreads + tid < m) s_entry[s_cnt[bin[k] & 0xffffu] + (bin[k] >> 16)] = v[k];
        __syncthreads();
        // an entry's place within its bin: how many of the bin's come before it (rarely more than three in all; reads whose array
        // is done at the very same time share a bin, however many they are)
#pragma unroll
        for (int k = 0; k < kBaItems; ++k) {
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
        for (int k = 0; k < kBaItems; ++k)
            if (k * kBaThreads + tid < m) s_entry[bin[k]] = v[k];
        __syncthreads();
        // every thread's stretch of the ordered entries as one map, what lies before it in the bucket, the bucket as a whole
        const uint32_t per = (m + kBaThreads - 1u) / kBaThreads, j0 = min(m, tid * per), j1 = min(m, j0 + per);
        BusMap mine = bus_identity();
        for (uint32_t j = j0; j < j1; ++j) {
            const ulonglong2 e = s_entry[j];
            const int64_t x = (int64_t)((e.x >> 47) | ((e.y >> 32) << 17)), done = (int64_t)(e.x & kBusDoneMask);
            mine.S += x; mine.M = max(mine.M, done) + x;     // (kNegInf + x stays far below any time)
        }
        BusMap incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const BusMap p = bus_shfl_up(incl, o); if (lane >= o) incl = bus_then(p, incl); }
        if (lane == 31) s_map[warp] = incl;
        __syncthreads();
        BusMap run = bus_identity();
        for (int w = 0; w < warp; ++w) run = bus_then(run, s_map[w]);
        BusMap prev = bus_shfl_up(incl, 1);
        if (lane == 0) prev = bus_identity();
        run = bus_then(run, prev);
        if (warp == 0) {
            BusMap all = bus_identity();
            for (int w = 0; w < kBaThreads / 32; ++w) all = bus_then(all, s_map[w]);
            const uint32_t channel = bucket % b.channels;
            if (lane == 0) { b.state[bucket].S = all.S; b.state[bucket].M = all.M; st_release_u32(&b.state[bucket].flag, 1u); }
            // look-back: the buckets of the channel, 32 at a time, the nearest first, as far as one that knows the bus after it
            BusMap near = bus_identity();
            int64_t p = (int64_t)(bucket / b.channels) - 1;
            bool ok = true;
            for (;; p -= 32) {
                BusMap at; at.S = 0; at.f = 1; at.M = 0;
                const int64_t slice = p - lane;
                if (slice < 0) at.M = b.busy[channel];
                else {
                    BusState *st = b.state + ((uint64_t)slice * b.channels + channel);
                    uint32_t polls = 0, flag;
                    while ((flag = ld_acquire_u32(&st->flag)) == 0u) { if (++polls > kSpinLimit) { ok = false; break; } }
                    at.S = ld_relaxed_s64(&st->S); at.M = ld_relaxed_s64(&st->M); at.f = flag == 2u ? 1 : 0;
                }
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    BusMap far;
                    far.S = __shfl_down_sync(0xffffffffu, at.S, o); far.M = __shfl_down_sync(0xffffffffu, at.M, o); far.f = __shfl_down_sync(0xffffffffu, at.f, o);
                    if (lane + o < 32) at = bus_then(far, at);
                }
                at.S = __shfl_sync(0xffffffffu, at.S, 0); at.M = __shfl_sync(0xffffffffu, at.M, 0); at.f = __shfl_sync(0xffffffffu, at.f, 0);
                near = bus_then(at, near);
                ok = __all_sync(0xffffffffu, ok);
                if (near.f || !ok) break;
            }
            if (lane == 0) {
                const int64_t carry = near.M, after = max(carry + all.S, all.M);
                s_carry = carry; s_ok = ok ? 1 : 0;
                if (ok) {
                    // (whoever read "own map" and finds this M already: max(carry + S, after) is the same `after`)
                    BusState *st = b.state + bucket;
                    st_relaxed_s64(&st->M, after);
                    st_release_u32(&st->flag, 2u);
                    if (bucket / b.channels == b.slices - 1u) b.busy[channel] = after;   // (every slice of the channel has read the old one)
                }
            }
        }
        __syncthreads();
        if (!s_ok) { if (tid == 0) atomicExch(&bc->code, (int)HBF_E_TIMEOUT); return; }
        int64_t bus = max(s_carry + run.S, run.M);
        for (uint32_t j = j0; j < j1; ++j) {
            const ulonglong2 e = s_entry[j];
            const int64_t x = (int64_t)((e.x >> 47) | ((e.y >> 32) << 17)), done = (int64_t)(e.x & kBusDoneMask);
            bus = max(bus, done) + x;
            if (bus != done + x) {                           // the transfer waited for the bus: completion and stall move by the wait
                const uint32_t idx = (uint32_t)e.y;
                completion[idx] = bus; stall[idx] += bus - done - x;
                moved += bus - done - x; max_c = max(max_c, (long long)bus);
            }
        }
    }
    moved = warp_sum(moved); max_c = warp_max(max_c);
    if (lane == 0) {
        if (moved) atomicAdd((unsigned long long *)&bc->modeled_ns, (unsigned long long)moved);
        if (max_c != INT64_MIN) atomicMax(&bc->max_completion_ns, max_c);
    }
}

cudaError_t launch_bus_buckets(const SubmitArgs &a, BatchCtrl *bc, int64_t *bus_busy, cudaStream_t st) {
    const uint64_t n = a.n;
    const BusArgs b = bus_args(n, a.mp.channels, a.ws, bus_busy);
    const int fast_ok = fast_geom_ok(a.fast, a.mp) ? 1 : 0;
    cudaError_t e = ensure_dyn_smem((const void *)k_bus_scatter, kBsSmem);
    if (e == cudaSuccess) e = ensure_dyn_smem((const void *)k_bus_buckets, kBaSmem);
    const uint64_t buckets = (uint64_t)b.slices * b.channels;
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
        e = launch_pdl(k_bus_buckets, (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(buckets, (uint64_t)a.sm_count * 2)), kBaThreads, kBaSmem, st, bc, b, a.completion, a.stall);
    g_kernel_launches += 4;
    return e;
}

}  // namespace hbf

// Batches out of issue order: the records are brought into (issue time, batch index) order, the in-order kernels serve them, and
// the results go back to batch order.  (Included by the file whose kernels launch kernels: every launch here is made from the
// device, once a batch has turned out not to be in order.)
//   sample    how the issue times spread: a histogram of 65,536 of them over 64 equal stretches gives every stretch its share
//             of buckets of about 2,560 records
//   scatter   every record goes to its bucket, as a 32-byte slot (record and index; one full sector, one store) at a place that
//             an atomic counter gives out: no order inside a bucket, no second pass.  Statuses are answered here, in batch order
//   offsets   where every bucket begins in the ordered list
//   sort      a block per bucket: the times spread over 4,096 bins of shared memory (about one in two is taken), ranks from the
//             bins' counters, the few bins with several records put in order one by one; records and indices out
//   serve     k_inorder_serve, _scan, _fixstraggle on the ordered list
//   give      completion and index go to the bucket of 8,192 results that they belong to, the same way
//   place     a block per bucket puts them in order through shared memory and writes completions and stalls, whole lines
// A bucket that overflows (times bunched more tightly than the sample shows), or more than 64 records in a bin, sends the batch
// to the radix sort, as do outstanding refresh claims (they go by batch index) and service times the in-order kernels do not hold.
// Bytes per record: 24 + 32 (scatter), 32 + 28 (sort), 28 + 16 (serve), 12 + 16, 16 + 24 + 16 (results): 244, streaming, against
// some 400, a third of them scattered, for six radix passes and a scan that gathers and scatters by sorted index.
#pragma once
#include "inorder_impl.cuh"

namespace hbf {

constexpr uint32_t kRgAvg = 2560, kRgCap = 3840;         // records per bucket: aimed at, and at most (sampling and chance: 1.5 is ten deviations)
constexpr uint32_t kRgSegs = 64, kRgSamples = 65536;
constexpr uint32_t kRgOut = 8192;                        // results per output bucket
constexpr int kRgThreads = 512;
constexpr uint32_t kRgBins = 4096, kRgBinMax = 64;
constexpr int kRgItems = (kRgCap + kRgThreads - 1) / kRgThreads;

struct RegroupCtrl {                                     // cleared before use, with the counters behind it
    uint32_t hist[kRgSegs], done, overflow, shift, segs;
    int64_t lo;
    uint32_t base[kRgSegs + 1], pad;
};
struct __align__(32) RegroupSlot { uint64_t addr; int64_t issue; uint64_t bf; uint64_t idx; };
struct RegroupArgs {
    RegroupCtrl *rg; uint32_t *cursor, *cursor_out, *offset;     // [max_buckets], [out_buckets], [max_buckets]
    RegroupSlot *slots; uint64_t *recs; uint32_t *idx;           // [max_buckets][kRgCap]; [3 n], [n]: the ordered list
    int64_t *comp, *stall; ulonglong2 *entries;                  // inside the slots' memory, once they have been read
    uint32_t max_buckets, out_buckets; uint64_t zero_words;
};
// Where place p of bucket b lies: the buckets' stretches of 32 slots side by side, then their next 32.  All buckets fill at much
// the same pace, so the places in use at a time lie in some 16 MB; with every bucket's slots in one piece each store fell into
// another page (scatter 1,054 us for 40 M records, most of it address translation).
__device__ __forceinline__ uint64_t rg_place(uint32_t buckets, uint32_t b, uint32_t p) { return ((uint64_t)(p >> 5) * buckets + b) * 32u + (p & 31u); }
inline uint32_t regroup_buckets(uint64_t n) { return (uint32_t)(n / kRgAvg) + kRgSegs + 1u; }
inline uint32_t regroup_out_buckets(uint64_t n) { return (uint32_t)((n + kRgOut - 1) / kRgOut); }
inline size_t regroup_slot_bytes(uint64_t n) { return std::max<size_t>((size_t)regroup_buckets(n) * kRgCap * sizeof(RegroupSlot), (size_t)n * 16 + (size_t)regroup_out_buckets(n) * kRgOut * 16 + 512); }
inline size_t regroup_ctrl_bytes(uint64_t n) { return sizeof(RegroupCtrl) + ((size_t)2 * regroup_buckets(n) + regroup_out_buckets(n)) * 4; }
inline RegroupArgs regroup_args(uint64_t n, const Workspace &ws) {
    RegroupArgs r{};
    r.max_buckets = regroup_buckets(n); r.out_buckets = regroup_out_buckets(n);
    r.rg = static_cast<RegroupCtrl *>(ws.rg_ctrl);
    r.cursor = reinterpret_cast<uint32_t *>(r.rg + 1); r.cursor_out = r.cursor + r.max_buckets; r.offset = r.cursor_out + r.out_buckets;
    r.zero_words = (sizeof(RegroupCtrl) + ((size_t)r.max_buckets + r.out_buckets) * 4) / 4;
    r.slots = static_cast<RegroupSlot *>(ws.rg_slots); r.recs = static_cast<uint64_t *>(ws.rg_recs); r.idx = static_cast<uint32_t *>(ws.rg_idx);
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    char *b = static_cast<char *>(ws.rg_slots);
    r.comp = reinterpret_cast<int64_t *>(b); r.stall = reinterpret_cast<int64_t *>(b + up(n * 8)); r.entries = reinterpret_cast<ulonglong2 *>(b + 2 * up(n * 8));
    return r;
}

__global__ void __launch_bounds__(1024)
k_regroup_sample(const hbf_access_t *__restrict__ acc, uint64_t n, const BatchCtrl *ctrl, RegroupArgs r) {
    __shared__ uint32_t sh[kRgSegs];
    __shared__ uint32_t s_last;
    const int tid = threadIdx.x;
    if (tid < (int)kRgSegs) sh[tid] = 0u;
    // the span that the begin kernel's samples showed, with a margin; stretches of a power of two of nanoseconds
    const int64_t first = ctrl->issue_lo, last = ctrl->issue_hi, margin = (last - first) / 128 + 1, lo = first - margin;
    const uint64_t span = (uint64_t)(last - first + 2 * margin);
    uint32_t shift = 0;
    while (((uint64_t)(kRgSegs - 1) << shift) < span) ++shift;
    __syncthreads();
    const uint64_t samples = min(n, (uint64_t)kRgSamples), s = (uint64_t)blockIdx.x * 1024 + tid;
    if (s < samples) {
        const int64_t t = (int64_t)__ldg(reinterpret_cast<const uint64_t *>(acc + s * n / samples) + 1);
        const uint64_t rel = t <= lo ? 0ull : (uint64_t)(t - lo);
        atomicAdd(&sh[min((uint64_t)(kRgSegs - 1), rel >> shift)], 1u);
    }
    __syncthreads();
    if (tid < (int)kRgSegs && sh[tid]) atomicAdd(&r.rg->hist[tid], sh[tid]);
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&r.rg->done, 1u) == gridDim.x - 1u ? 1u : 0u;
    __syncthreads();
    if (!s_last || tid != 0) return;
    const uint64_t want = n / kRgAvg;
    uint32_t at = 0;
    for (uint32_t k = 0; k < kRgSegs; ++k) {               // at least one bucket each; the sum stays within max_buckets
        r.rg->base[k] = at;
        at += (uint32_t)max(1ull, (unsigned long long)(want * __ldcg(&r.rg->hist[k]) / samples));
    }
    r.rg->base[kRgSegs] = at; r.rg->lo = lo; r.rg->shift = shift;
}

constexpr int kRgScatterItems = 4;
__global__ void __launch_bounds__(256)
k_regroup_scatter(const hbf_access_t *__restrict__ acc, uint64_t n, const RangeSnap *__restrict__ ranges, const __grid_constant__ FastRange fast, RegroupArgs r, uint8_t *status) {
    __shared__ uint32_t s_base[kRgSegs + 1];
    for (uint32_t k = threadIdx.x; k <= kRgSegs; k += blockDim.x) s_base[k] = r.rg->base[k];
    __syncthreads();
    const int64_t lo = r.rg->lo;
    const uint32_t shift = r.rg->shift, buckets = r.rg->base[kRgSegs];
    for (uint64_t i0 = (uint64_t)blockIdx.x * (256 * kRgScatterItems) + threadIdx.x; i0 < n; i0 += (uint64_t)gridDim.x * (256 * kRgScatterItems)) {
        uint64_t addr[kRgScatterItems], issue[kRgScatterItems], bf[kRgScatterItems];
        uint32_t at[kRgScatterItems], bucket[kRgScatterItems];
#pragma unroll
        for (int k = 0; k < kRgScatterItems; ++k) {
            const uint64_t i = i0 + (uint64_t)k * 256;
            addr[k] = issue[k] = bf[k] = 0ull;
            if (i < n) { const uint64_t *rec = reinterpret_cast<const uint64_t *>(acc + i); addr[k] = __ldcs(rec); issue[k] = __ldcs(rec + 1); bf[k] = __ldcs(rec + 2); }
        }
#pragma unroll
        for (int k = 0; k < kRgScatterItems; ++k) {
            const uint64_t i = i0 + (uint64_t)k * 256;
            if (i < n) {
                const uint64_t rel = (int64_t)issue[k] <= lo ? 0ull : (uint64_t)((int64_t)issue[k] - lo);
                const uint32_t seg = (uint32_t)min((uint64_t)(kRgSegs - 1), rel >> shift);
                const uint64_t in = min(rel - ((uint64_t)seg << shift), ((uint64_t)1 << shift) - 1u);
                const uint32_t b0 = s_base[seg], nb = s_base[seg + 1] - b0;
                // (the offset is cut to 32 bits first: the product has to fit, and a bucket's edge need not be exact)
                bucket[k] = b0 + (uint32_t)(((shift > 32u ? in >> (shift - 32u) : in) * nb) >> min(shift, 32u));
                at[k] = atomicAdd(&r.cursor[bucket[k]], 1u);
            }
        }
#pragma unroll
        for (int k = 0; k < kRgScatterItems; ++k) {
            const uint64_t i = i0 + (uint64_t)k * 256;
            if (i < n) {
                if (at[k] < kRgCap)
                    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(r.slots + rg_place(buckets, bucket[k], at[k])), "l"(addr[k]), "l"(issue[k]), "l"(bf[k]), "l"(i) : "memory");
                else r.rg->overflow = 1u;
                if (status) {
                    const uint32_t bytes = (uint32_t)bf[k], flags = (uint32_t)(bf[k] >> 32);
                    int st, g = 0;
                    if (fast.on) {
                        const uint64_t rel = addr[k] - fast.base;
                        st = ((fast.perms >> (flags & 1u)) & 1u) ? HBF_ST_READY : HBF_ST_FAULT_PERM;
                        if ((uint64_t)bytes > fast.length - rel) st = HBF_ST_FAULT_PARTIAL;
                        if (rel >= fast.length) st = HBF_ST_NATIVE;
                        if (bytes == 0u || flags > 1u || (issue[k] >> kIssueBits) != 0ull) st = HBF_ST_UNSUPPORTED;
                    } else {
                        st = classify(*ranges, addr[k], (int64_t)issue[k], bytes, flags, &g);
                    }
                    status[i] = (uint8_t)st;
                }
            }
        }
    }
}

__global__ void __launch_bounds__(1024) k_regroup_offsets(uint64_t n, RegroupArgs r) {
    __shared__ uint32_t s_w[32];
    if (r.rg->overflow) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t buckets = r.rg->base[kRgSegs], per = (buckets + 1023u) / 1024u, lo = min(buckets, tid * per), hi = min(buckets, lo + per);
    uint32_t sum = 0;
    for (uint32_t b = lo; b < hi; ++b) sum += r.cursor[b];
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    uint32_t run = inc - sum;
    for (int w = 0; w < warp; ++w) run += s_w[w];
    for (uint32_t b = lo; b < hi; ++b) { r.offset[b] = run; run += r.cursor[b]; }
}

constexpr size_t kRgSortSmem = (size_t)kRgCap * (8 + 2) + (size_t)kRgBins * 4;
__global__ void __launch_bounds__(kRgThreads, 3) k_regroup_sort(RegroupArgs r) {
    extern __shared__ __align__(16) unsigned char rg_smem[];
    uint64_t *s_key = reinterpret_cast<uint64_t *>(rg_smem);                 // [kRgCap] time from the bucket's first << 32 | index
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_key + kRgCap);          // [kRgBins]
    uint16_t *s_slot = reinterpret_cast<uint16_t *>(s_cnt + kRgBins);        // [kRgCap]
    __shared__ long long s_min, s_max;
    __shared__ uint32_t s_w[kRgThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t buckets = r.rg->base[kRgSegs];
    if (r.rg->overflow) return;
    for (uint32_t b = blockIdx.x; b < buckets; b += gridDim.x) {
        const uint32_t m = min(r.cursor[b], kRgCap), off = r.offset[b];
        auto slot = [&](uint32_t e) { return r.slots + rg_place(buckets, b, e); };
        __syncthreads();                                     // shared memory of the bucket before is no longer read
        if (tid == 0) { s_min = INT64_MAX; s_max = INT64_MIN; }
        for (uint32_t e = tid; e < kRgBins; e += kRgThreads) s_cnt[e] = 0u;
        int64_t issue[kRgItems]; uint32_t idx[kRgItems], bin[kRgItems];
        long long lo = INT64_MAX, hi = INT64_MIN;
#pragma unroll
        for (int k = 0; k < kRgItems; ++k) {
            const uint32_t e = k * kRgThreads + tid;
            if (e < m) { issue[k] = slot(e)->issue; idx[k] = (uint32_t)slot(e)->idx; lo = min(lo, (long long)issue[k]); hi = max(hi, (long long)issue[k]); }
        }
        for (int o = 16; o > 0; o >>= 1) { lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
        __syncthreads();
        if (lane == 0 && lo <= hi) { atomicMin(&s_min, lo); atomicMax(&s_max, hi); }
        __syncthreads();
        const int64_t first = s_min;
        const uint64_t span = m ? (uint64_t)(s_max - first) : 0ull;
        if (span >> 32) { if (tid == 0) r.rg->overflow = 1u; return; }      // (the same for the whole block)
        const uint64_t mul = ((uint64_t)kRgBins << 32) / (span + 1ull);
#pragma unroll
        for (int k = 0; k < kRgItems; ++k) {
            const uint32_t e = k * kRgThreads + tid;
            if (e < m) { const uint32_t d = (uint32_t)(((uint64_t)(issue[k] - first) * mul) >> 32); bin[k] = d | (atomicAdd(&s_cnt[d], 1u) << 16); }
        }
        __syncthreads();
        {                                                    // exclusive scan of the bins, eight per thread
            uint32_t v[kRgBins / kRgThreads], sum = 0;
#pragma unroll
            for (uint32_t k = 0; k < kRgBins / kRgThreads; ++k) { v[k] = s_cnt[tid * (kRgBins / kRgThreads) + k]; sum += v[k]; }
            uint32_t inc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
            if (lane == 31) s_w[warp] = inc;
            __syncthreads();
            uint32_t run = inc - sum;
            for (int w = 0; w < warp; ++w) run += s_w[w];
#pragma unroll
            for (uint32_t k = 0; k < kRgBins / kRgThreads; ++k) { s_cnt[tid * (kRgBins / kRgThreads) + k] = run; run += v[k]; }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kRgItems; ++k) {
            const uint32_t e = k * kRgThreads + tid;
            if (e < m) s_key[s_cnt[bin[k] & 0xffffu] + (bin[k] >> 16)] = ((uint64_t)(issue[k] - first) << 32) | idx[k];
        }
        __syncthreads();
        bool over = false;
        // a record's place within its bin: how many of the bin's keys are smaller (a bin rarely has more than four)
#pragma unroll
        for (int k = 0; k < kRgItems; ++k) {
            const uint32_t e = k * kRgThreads + tid;
            if (e < m) {
                const uint32_t d = bin[k] & 0xffffu, from = s_cnt[d], to = d + 1u < kRgBins ? s_cnt[d + 1u] : m;
                uint32_t before = 0;
                if (to - from > kRgBinMax) over = true;
                else if (to - from > 1u) {
                    const uint64_t key = ((uint64_t)(issue[k] - first) << 32) | idx[k];
                    for (uint32_t q = from; q < to; ++q) before += s_key[q] < key ? 1u : 0u;
                }
                s_slot[from + before] = (uint16_t)e;
            }
        }
        if (__syncthreads_or(over)) { if (tid == 0) r.rg->overflow = 1u; return; }
        for (uint32_t j = tid; j < m; j += kRgThreads) {
            const RegroupSlot *p = slot(s_slot[j]);
            uint64_t w0, w1, w2, w3;
            asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(w0), "=l"(w1), "=l"(w2), "=l"(w3) : "l"(p));
            uint64_t *o = r.recs + (uint64_t)(off + j) * 3;
            o[0] = w0; o[1] = w1; o[2] = w2;
            r.idx[off + j] = (uint32_t)w3;
        }
    }
}

__global__ void __launch_bounds__(256) k_regroup_give(uint64_t n, const BatchCtrl *ctrl, RegroupArgs r) {
    if (!ctrl->inorder_used) return;
    for (uint64_t i0 = (uint64_t)blockIdx.x * 1024 + threadIdx.x; i0 < n; i0 += (uint64_t)gridDim.x * 1024) {
        uint64_t comp[4]; uint32_t idx[4], at[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint64_t i = i0 + (uint64_t)k * 256;
            if (i < n) { comp[k] = (uint64_t)__ldcs(reinterpret_cast<const long long *>(r.comp + i)); idx[k] = __ldg(r.idx + i); }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) if (i0 + (uint64_t)k * 256 < n) at[k] = atomicAdd(&r.cursor_out[idx[k] / kRgOut], 1u);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i0 + (uint64_t)k * 256 < n) r.entries[rg_place(r.out_buckets, idx[k] / kRgOut, at[k])] = make_ulonglong2(comp[k], idx[k] % kRgOut);   // (a permutation: no more than kRgOut each)
    }
}

__global__ void __launch_bounds__(1024) k_regroup_place(const hbf_access_t *__restrict__ acc, uint64_t n, BatchCtrl *ctrl, RegroupArgs r,
                                                        int64_t *__restrict__ completion, int64_t *__restrict__ stall) {
    extern __shared__ __align__(16) unsigned char rg_smem[];
    int64_t *s_comp = reinterpret_cast<int64_t *>(rg_smem);
    if (!ctrl->inorder_used) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->regrouped = 1u;
    for (uint32_t b = blockIdx.x; b < r.out_buckets; b += gridDim.x) {
        const uint64_t base = (uint64_t)b * kRgOut;
        const uint32_t m = (uint32_t)min((uint64_t)kRgOut, n - base);
        __syncthreads();
        for (uint32_t e = threadIdx.x; e < m; e += 1024u) { const ulonglong2 v = __ldcs(r.entries + rg_place(r.out_buckets, b, e)); s_comp[v.y] = (int64_t)v.x; }
        __syncthreads();
        for (uint32_t e = threadIdx.x; e < m; e += 1024u) {
            const int64_t c = s_comp[e], issue = (int64_t)__ldcs(reinterpret_cast<const uint64_t *>(acc + base + e) + 1);
            __stcs(reinterpret_cast<long long *>(completion + base + e), (long long)c);
            __stcs(reinterpret_cast<long long *>(stall + base + e), (long long)(c - issue));
        }
    }
}
constexpr size_t kRgPlaceSmem = (size_t)kRgOut * 8;

}  // namespace hbf

// The begin kernel of batches that may turn out to be out of issue order, with the phases that bring the records into order
// (regroup.cuh has the whole of it).  A block per multiprocessor; where the batch is in order all but the first leave at once
// (65,536 records in order: 57.1 -> 58.2 us with reset, 1.2 M 72.0 -> 72.9; 65,536 shuffled 328 -> 172, 1.2 M 517 -> 332).
// 40 M shuffled records take 2,810 us, 4,600 as ten kernels launched from the device: such launches take some 9 us each, and the
// kernels get no more shared memory than one block of theirs needs, so that one ran per multiprocessor where two or three fit.
// scatter 620 us and give 690: bound by the rate of single atomics and stores all over the L2 (60 per ns; the number of buckets,
// the counters' spacing and the warps in flight do not change it).
#include <algorithm>

#include "begin.cuh"
#include "regroup.cuh"

namespace hbf {

size_t regroup_slot_bytes(uint64_t n) { return std::max<size_t>((size_t)regroup_buckets(n) * kRgCap * sizeof(RegroupSlot), (size_t)n * 16 + (size_t)regroup_out_buckets(n) * kRgOut * 16 + 512); }
size_t regroup_ctrl_bytes(uint64_t n) { return ((size_t)(kRgPad + 1) * regroup_buckets(n) + (size_t)kRgPad * regroup_out_buckets(n) + regroup_buckets(n) / kRgChunk + 1) * 4; }
OrderedCopy ordered_copy(uint64_t n, const Workspace &ws) {
    const RegroupArgs r = regroup_args(n, ws, nullptr);
    return OrderedCopy{reinterpret_cast<const hbf_access_t *>(r.recs), r.comp, r.stall};
}

constexpr int kRgThreads = 1024, kRgGroup = 512, kRgGroups = kRgThreads / kRgGroup;
constexpr uint32_t kRgBins = 4096;
constexpr int kRgItems = kRgCap / kRgGroup;
static_assert(kRgCap % kRgGroup == 0 && kRgBins % kRgGroup == 0, "whole rounds");
constexpr uint32_t kRgParts = 4096;                      // chunks of buckets at most: 2^32 records
constexpr size_t kRgGroupSmem = (size_t)kRgCap * 28 + (size_t)kRgBins * 4;
constexpr size_t kRgSmem = kRgGroups * kRgGroupSmem + (size_t)kRgParts * 4;

__device__ __forceinline__ void group_sync(int group) { asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kRgGroup) : "memory"); }

// A time's stretch, and its offset in it (32 bits of it: a bucket's edge need not be exact).
__device__ __forceinline__ uint32_t rg_stretch(int64_t t, int64_t lo, uint32_t shift, uint32_t *offset) {
    const uint64_t rel = t <= lo ? 0ull : (uint64_t)(t - lo);
    const uint32_t seg = (uint32_t)min((uint64_t)(kRgSegs - 1), rel >> shift);
    const uint64_t in = min(rel - ((uint64_t)seg << shift), ((uint64_t)1 << shift) - 1u);
    *offset = (uint32_t)(shift > 32u ? in >> (shift - 32u) : in);
    return seg;
}

// Do so many records share their issue times that buckets would overflow, or spend their time on telling equal times apart?  1,024
// samples, one per thread, and a table of the distinct ones; where few are equal, pairs of equal ones tell (of m samples of D times
// about m^2 / 2D), else the distinct ones are nearly all there are.  The buckets' time depends on how the few times fall into their bins as well,
// so no line by the number alone is right everywhere.  us, shuffled records, in buckets with 1, 20, 60, 120, 250, 400 and 600 per time, and by
// the radix sort: 40 M 2,780, 3,690, 4,910, 7,990, 5,030, 14,700, 10,000, and 6,340; 12 M 970, 1,270, 1,630, 2,570, 1,690, 4,670, 3,310, and 1,880;
// 4 M 444, 552, 667, 982, 690, 1,750, 1,290, and 645; 1 M 299, 343, 338, 422, 334, 677, 550, and 300 (small batches lose 4 to 15 % up to 300 per
// time, and 40 to 50 % where the times fall badly; from 900 on the buckets overflow, and the attempt is lost besides).
constexpr uint32_t kRgCrowd = 300, kRgSeen = 4096;
__device__ __forceinline__ bool rg_crowded(long long time, uint64_t n, unsigned long long *seen) {
    for (uint32_t e = threadIdx.x; e < kRgSeen; e += kRgThreads) seen[e] = 0ull;
    __syncthreads();
    const unsigned long long key = (unsigned long long)time + 1ull;
    uint32_t at = (uint32_t)((key * 0x9e3779b97f4a7c15ull) >> 52);
    bool fresh = false;
    for (;;) {                                               // (a quarter full at most)
        const unsigned long long had = atomicCAS(seen + at, 0ull, key);
        fresh = had == 0ull;
        if (fresh || had == key) break;
        at = (at + 1u) % kRgSeen;
    }
    const uint64_t distinct = (uint64_t)__syncthreads_count(fresh), equal = kRgThreads - distinct;
    return equal != 0ull && n > kRgCrowd * (2u * distinct <= (uint64_t)kRgThreads ? distinct : (uint64_t)kRgThreads * kRgThreads / (2u * equal));
}

__global__ void __launch_bounds__(kRgThreads, 1)
k_begin_regroup(const __grid_constant__ BeginArgs b, const hbf_access_t *__restrict__ acc, uint64_t n, const RangeSnap *__restrict__ ranges,
                const __grid_constant__ FastRange fast, const __grid_constant__ RegroupArgs r, uint8_t *status) {
    extern __shared__ __align__(16) unsigned char rg_smem[];
    __shared__ long long s_lo, s_hi;
    __shared__ uint32_t s_base[kRgSegs], s_first[kRgSegs], s_last[kRgSegs], s_buckets, s_w[kRgThreads / 32], s_next[kRgGroups];
    __shared__ uint64_t s_mul[kRgSegs];
    __shared__ long long s_min[kRgGroups], s_max[kRgGroups];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_wait();
    pdl_trigger();
    // pairs of neighbouring records show whether the batch is in order (every block asks the same ones)
    if (tid == 0) { s_lo = INT64_MAX; s_hi = INT64_MIN; }
    long long first, last;
    bool bad = begin_samples(acc, n, &first, &last);
    const long long one = first;
    if (bad) {
        for (int o = 16; o > 0; o >>= 1) { first = min(first, __shfl_xor_sync(0xffffffffu, first, o)); last = max(last, __shfl_xor_sync(0xffffffffu, last, o)); }
        if (lane == 0) { atomicMin(&s_lo, first); atomicMax(&s_hi, last); }
        __syncthreads();
        first = s_lo; last = s_hi;
    }
    // (refresh claims go by batch index: a batch that has to pay some is sorted, and one whose workspace has no room, or with few
    // distinct times; so is one whose samples lie outside the limits of
    // issue times, which the sort path refuses: spans up to 2^48 ns are all that the stretches below are made for)
    const bool outside = first < 0 || last >= HBF_ISSUE_LIMIT;
    const bool sorted = bad && (first >= last || outside || !r.cursor || rg_crowded(one, n, reinterpret_cast<unsigned long long *>(rg_smem)) || (b.claim_limit && *b.claim_limit > 0ull)), go = bad && !sorted && !begin_refused(b.state);
    RegroupSync *sync = r.sync;
    BatchCtrl *ctrl = b.ctrl;
    const uint32_t limit = b.state->spin_limit;
    if (blockIdx.x == 0) {
        begin_batch(b, sorted ? 1 : 0, go ? 1u : 0u);
        if (b.decides && !sorted) begin_load(b, reinterpret_cast<const uint64_t *>(acc + (uint64_t)tid * (n - 1ull) / 1024ull), bad ? first : ld_after(&acc[0].issue_ns), bad ? last : ld_after(&acc[n - 1].issue_ns));
        if (tid < 2) sync->claim[3 + tid] = 0u;              // (those of the last kernel)
        if (tid == 2) sync->claim[6] = 0u;
        if (tid < 3) sync->done[3 + tid] = 0u;
        __threadfence();
        __syncthreads();
        if (tid == 0 && go) atomicAdd(&sync->done[0], 1u);
    }
    if (!go) return;

    // ---- sample: how the issue times spread.  The span that the pairs showed, with a margin; stretches of a power of two of ns
    const int64_t margin = (last - first) / 128 + 1, lo = first - margin;
    const uint64_t span = (uint64_t)(last - first + 2 * margin);
    uint32_t shift = 0;
    while (((uint64_t)(kRgSegs - 1) << shift) < span) ++shift;
    const uint64_t samples = min(n, (uint64_t)kRgSamples);
    constexpr uint32_t kShare = 256, kZero = 8192;
    const uint32_t sample_shares = (uint32_t)((samples + kShare - 1) / kShare);
    const uint64_t zeros = ((uint64_t)r.max_buckets + r.out_buckets) * kRgPad;
    const uint32_t zero_shares = (uint32_t)((zeros + kZero - 1) / kZero);
    rg_shares(sync, 0, sample_shares + zero_shares, kRgNone, [&](uint32_t k) {
        if (k < zero_shares) {
            for (uint64_t i = (uint64_t)k * kZero + lane; i < min(zeros, (uint64_t)(k + 1) * kZero); i += 32) r.cursor[i] = 0u;
            return;
        }
        for (uint64_t s = (uint64_t)(k - zero_shares) * kShare + lane; s < min(samples, (uint64_t)(k - zero_shares + 1) * kShare); s += 32) {
            uint32_t off;
            const uint32_t seg = rg_stretch((int64_t)ld_after(reinterpret_cast<const uint64_t *>(acc + s * n / samples) + 1), lo, shift, &off);
            atomicAdd(&sync->hist[seg], 1u); atomicMax(&sync->top[seg], off); atomicMax(&sync->below[seg], ~off);
        }
    });
    __syncthreads();
    if (!rg_wait_or_give_up(sync, 0, sample_shares + zero_shares + 1u, limit, ctrl)) return;
    if (warp == 0) {
        const uint64_t want = n / kRgAvg, whole = (uint64_t)1 << min(shift, 32u);
        uint32_t nb[2], sum = 0;
#pragma unroll
        for (int k = 0; k < 2; ++k) {                        // at least one bucket each; the sum stays within max_buckets
            nb[k] = (uint32_t)max(1ull, (unsigned long long)((want * __ldcg(&sync->hist[2 * lane + k]) + samples - 1u) / samples));
            sum += nb[k];
        }
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
        uint32_t at = inc - sum;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint32_t seg = 2 * lane + k, count = __ldcg(&sync->hist[seg]);
            // the part of the stretch that holds its samples, and 16 samples' share more on both sides (a record beyond it is one
            // in e^16): the first and the last stretch are rarely full, and equal parts of them would be filled twice over
            uint64_t a = 0, z = whole - 1u;
            if (count) {
                const uint64_t s0 = (uint32_t)~__ldcg(&sync->below[seg]), s1 = __ldcg(&sync->top[seg]), more = (s1 - s0) * 16u / count + 1u;
                a = s0 > more ? s0 - more : 0u; z = min(z, s1 + more);
            }
            s_base[seg] = at; s_first[seg] = (uint32_t)a; s_last[seg] = (uint32_t)z;
            s_mul[seg] = ((uint64_t)nb[k] << 32) / (z - a + 1u);
            at += nb[k];
        }
        if (lane == 31) s_buckets = at;
    }
    __syncthreads();
    const uint32_t buckets = s_buckets;

    // ---- scatter: a warp takes 1,024 records, 128 at a time
    constexpr uint32_t kScatter = 1024;
    const uint32_t scatters = (uint32_t)((n + kScatter - 1) / kScatter);
    rg_shares(sync, 1, scatters, b.state->test_stage == 1u ? b.state->test_tile : kRgNone, [&](uint32_t g) {
        if (ld_relaxed_u32(&ctrl->run_sort)) return;         // a bucket has overflowed: the rest is not worth sending
        for (uint32_t at0 = 0; at0 < kScatter; at0 += 128u) {
            uint64_t addr[4], issue[4], bf[4];
            uint32_t at[4], bucket[4];
            const uint64_t i0 = (uint64_t)g * kScatter + at0 + lane;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint64_t i = i0 + 32u * k;
                addr[k] = issue[k] = bf[k] = 0ull;
                if (i < n) { const uint64_t *rec = reinterpret_cast<const uint64_t *>(acc + i); addr[k] = __ldcs(rec); issue[k] = __ldcs(rec + 1); bf[k] = __ldcs(rec + 2); }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (i0 + 32u * k < n) {
                    uint32_t off;
                    const uint32_t seg = rg_stretch((int64_t)issue[k], lo, shift, &off), a = s_first[seg];
                    bucket[k] = s_base[seg] + (uint32_t)(((uint64_t)(min(max(off, a), s_last[seg]) - a) * s_mul[seg]) >> 32);
                    at[k] = atomicAdd(&r.cursor[(size_t)bucket[k] * kRgPad], 1u);
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint64_t i = i0 + 32u * k;
                if (i < n) {
                    if (at[k] < kRgCap)
                        asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(r.slots + rg_place(buckets, bucket[k], at[k])), "l"(addr[k]), "l"(issue[k]), "l"(bf[k]), "l"(i) : "memory");
                    else ctrl->run_sort = 1u;
                    if (status) {
                        const uint32_t bytes = (uint32_t)bf[k], flags = (uint32_t)(bf[k] >> 32);
                        int st, gi = 0;
                        if (fast.on) {
                            const uint64_t rel = addr[k] - fast.base;
                            st = ((fast.perms >> (flags & 1u)) & 1u) ? HBF_ST_READY : HBF_ST_FAULT_PERM;
                            if ((uint64_t)bytes > fast.length - rel) st = HBF_ST_FAULT_PARTIAL;
                            if (rel >= fast.length) st = HBF_ST_NATIVE;
                            if (bytes == 0u || flags > 1u || (issue[k] >> kIssueBits) != 0ull) st = HBF_ST_UNSUPPORTED;
                        } else {
                            st = classify(*ranges, addr[k], (int64_t)issue[k], bytes, flags, &gi);
                        }
                        status[i] = (uint8_t)st;
                    }
                }
            }
        }
    });
    __syncthreads();
    if (!rg_wait_or_give_up(sync, 1, scatters, limit, ctrl)) return;
    if (ld_relaxed_u32(&ctrl->run_sort)) return;             // a bucket overflowed (settled: the same for every block)

    // ---- offsets: where a bucket begins among its chunk of 1,024, and the chunks' sums
    const uint32_t chunks = (buckets + kRgChunk - 1u) / kRgChunk;
    rg_shares(sync, 2, chunks, kRgNone, [&](uint32_t c) {
        uint32_t run = 0;
        for (uint32_t k = 0; k < kRgChunk; k += 256u) {
            uint32_t v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) { const uint32_t q = c * kRgChunk + k + 32u * j + lane; v[j] = q < buckets ? __ldcg(&r.cursor[(size_t)q * kRgPad]) : 0u; }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                uint32_t inc = v[j];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
                const uint32_t q = c * kRgChunk + k + 32u * j + lane;
                if (q < buckets) r.offset[q] = run + inc - v[j];
                run += __shfl_sync(0xffffffffu, inc, 31);
            }
        }
        if (lane == 0) r.part[c] = run;
    });
    __syncthreads();
    if (!rg_wait_or_give_up(sync, 2, chunks, limit, ctrl)) return;
    uint32_t *s_part = reinterpret_cast<uint32_t *>(rg_smem + kRgGroups * kRgGroupSmem);
    if (warp == 0) {
        uint32_t run = 0;
        for (uint32_t c = 0; c < chunks; c += 32u) {
            const uint32_t v = c + lane < chunks ? __ldcg(&r.part[c + lane]) : 0u;
            uint32_t inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
            if (c + lane < chunks) s_part[c + lane] = run + inc - v;
            run += __shfl_sync(0xffffffffu, inc, 31);
        }
    }
    __syncthreads();

    // ---- sort: each half of the block on buckets of its own, the next one taken while one is at work
    const int group = tid / kRgGroup, gtid = tid % kRgGroup, gwarp = gtid >> 5;
    uint64_t *s_rec = reinterpret_cast<uint64_t *>(rg_smem + group * kRgGroupSmem);   // [3 kRgCap] the ordered records
    uint64_t *s_key = s_rec;                                                          // [kRgCap] before that: time from the bucket's first << 32 | index
    uint32_t *s_idx = reinterpret_cast<uint32_t *>(s_rec + 3 * kRgCap);               // [kRgCap]
    uint32_t *s_cnt = s_idx + kRgCap;                                                 // [kRgBins]
    uint32_t *s_sum = s_w + group * (kRgGroup / 32);
    if (gtid == 0) s_next[group] = atomicAdd(&sync->claim[5], 1u);
    group_sync(group);
    uint32_t at = s_next[group];
    while (at < buckets) {
        const uint32_t m = min(__ldcg(&r.cursor[(size_t)at * kRgPad]), kRgCap), off = s_part[at / kRgChunk] + __ldcg(&r.offset[at]);
        uint64_t addr[kRgItems], bf[kRgItems]; int64_t issue[kRgItems]; uint32_t idx[kRgItems], bin[kRgItems];
#pragma unroll
        for (int k = 0; k < kRgItems; ++k) {
            const uint32_t e = k * kRgGroup + gtid;
            if (e < m) {
                uint64_t w;
                asm volatile("ld.global.cs.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(addr[k]), "=l"(issue[k]), "=l"(bf[k]), "=l"(w) : "l"(r.slots + rg_place(buckets, at, e)));
                idx[k] = (uint32_t)w;
            }
        }
        group_sync(group);                                   // shared memory of the bucket before is no longer read
        if (gtid == 0) { s_min[group] = INT64_MAX; s_max[group] = INT64_MIN; s_next[group] = atomicAdd(&sync->claim[5], 1u); }
        for (uint32_t e = gtid; e < kRgBins; e += kRgGroup) s_cnt[e] = 0u;
        long long mn = INT64_MAX, mx = INT64_MIN;
#pragma unroll
        for (int k = 0; k < kRgItems; ++k) if (k * kRgGroup + gtid < m) { mn = min(mn, (long long)issue[k]); mx = max(mx, (long long)issue[k]); }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o)); mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o)); }
        group_sync(group);
        if (lane == 0 && mn <= mx) { atomicMin(&s_min[group], mn); atomicMax(&s_max[group], mx); }
        group_sync(group);
        const uint32_t next = s_next[group];
        if (next < buckets) {                                // the next bucket is called into the L2 meanwhile
#pragma unroll
            for (int k = 0; k < kRgItems; ++k) {
                const uint32_t e = k * kRgGroup + gtid;
                if ((e & 3u) == 0u && e < kRgAvg) asm volatile("prefetch.global.L2 [%0];" ::"l"(r.slots + rg_place(buckets, next, e)));
            }
        }
        const int64_t t0 = s_min[group];
        const uint64_t wide = m ? (uint64_t)(s_max[group] - t0) : 0ull;
        if (wide >> 32) { if (gtid == 0) ctrl->run_sort = 1u; return; }               // (the same for the whole group, which no one waits for)
        const uint64_t mul = ((uint64_t)kRgBins << 32) / (wide + 1ull);
#pragma unroll
        for (int k = 0; k < kRgItems; ++k)
            if (k * kRgGroup + gtid < m) { const uint32_t d = (uint32_t)(((uint64_t)(issue[k] - t0) * mul) >> 32); bin[k] = d | (atomicAdd(&s_cnt[d], 1u) << 16); }
        group_sync(group);
        {                                                    // exclusive scan of the bins, eight per thread
            constexpr uint32_t kPer = kRgBins / kRgGroup;
            uint32_t v[kPer], sum = 0;
#pragma unroll
            for (uint32_t k = 0; k < kPer; k += 4) {
                const uint4 q = *reinterpret_cast<const uint4 *>(s_cnt + gtid * kPer + k);
                v[k] = q.x; v[k + 1] = q.y; v[k + 2] = q.z; v[k + 3] = q.w; sum += q.x + q.y + q.z + q.w;
            }
            uint32_t inc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
            if (lane == 31) s_sum[gwarp] = inc;
            group_sync(group);
            uint32_t run = inc - sum + __reduce_add_sync(0xffffffffu, lane < gwarp ? s_sum[lane] : 0u);
#pragma unroll
            for (uint32_t k = 0; k < kPer; k += 4) {
                uint4 q;
                q.x = run; q.y = q.x + v[k]; q.z = q.y + v[k + 1]; q.w = q.z + v[k + 2]; run = q.w + v[k + 3];
                *reinterpret_cast<uint4 *>(s_cnt + gtid * kPer + k) = q;
            }
        }
        group_sync(group);
#pragma unroll
        for (int k = 0; k < kRgItems; ++k)
            if (k * kRgGroup + gtid < m) s_key[s_cnt[bin[k] & 0xffffu] + (bin[k] >> 16)] = ((uint64_t)(issue[k] - t0) << 32) | idx[k];
        group_sync(group);
        // a record's place within its bin: how many of the bin's keys are smaller (rarely more than three in all; records issued at the
        // same time share a bin, however many they are)
#pragma unroll
        for (int k = 0; k < kRgItems; ++k) {
            if (k * kRgGroup + gtid < m) {
                const uint32_t d = bin[k] & 0xffffu, from = s_cnt[d], to = d + 1u < kRgBins ? s_cnt[d + 1u] : m;
                uint32_t before = 0;
                if (to - from > 1u) {
                    const uint64_t key = ((uint64_t)(issue[k] - t0) << 32) | idx[k];
                    for (uint32_t q = from; q < to; ++q) before += s_key[q] < key ? 1u : 0u;
                }
                bin[k] = from + before;
            }
        }
        group_sync(group);
#pragma unroll
        for (int k = 0; k < kRgItems; ++k)
            if (k * kRgGroup + gtid < m) { uint64_t *o = s_rec + bin[k] * 3u; o[0] = addr[k]; o[1] = (uint64_t)issue[k]; o[2] = bf[k]; s_idx[bin[k]] = idx[k]; }
        group_sync(group);
        uint64_t *out = r.recs + (uint64_t)off * 3;
        for (uint32_t j = gtid; j < 3u * m; j += kRgGroup) out[j] = s_rec[j];
        for (uint32_t j = gtid; j < m; j += kRgGroup) r.idx[off + j] = s_idx[j];
        at = next;
    }
}

cudaError_t launch_begin_regroup(const SubmitArgs &a, const BeginArgs &b, cudaStream_t st) {
    const cudaError_t e = ensure_dyn_smem((const void *)k_begin_regroup, kRgSmem);
    if (e != cudaSuccess) return e;
    return launch_first(a.plain_next, k_begin_regroup, (unsigned)std::min<uint64_t>((uint64_t)a.sm_count, a.n / 2048 + 1), kRgThreads, kRgSmem, st, b, a.acc, a.n, a.ranges, a.fast, regroup_args(a.n, a.ws, a.rg_sync), a.status);
}

}  // namespace hbf

// Batches out of issue order: the records are brought into (issue time, batch index) order, the in-order kernels serve that copy,
// and the results go back to batch order.  Two kernels of the in-order path do that when the samples of the first one showed a
// batch out of order, each in several phases: the begin kernel, and the last one.
//   sample    how the issue times spread: a histogram of 65,536 of them over 64 equal stretches gives every stretch its share
//             of buckets of about 1,365 records
//   scatter   every record goes to its bucket, as a 32-byte slot (record and index; one full sector, one store) at a place that
//             an atomic counter gives out: no order inside a bucket, no second pass.  Statuses are answered here, in batch order
//   offsets   where every bucket begins in the ordered list
//   sort      512 threads per bucket: the times spread over 4,096 bins of shared memory (about one in three is taken); a record's
//             place within its bin is the number of smaller (time, index) in it; the ordered records leave through shared memory
//   (the in-order kernels)
//   give      completion, issue time and index go to the bucket of 2,048 results that they belong to, the same way
//   place     a block per bucket puts them in order through shared memory and writes completions and stalls, whole lines
// A bucket that overflows (times bunched more tightly than the sample shows) sends the batch
// to the radix sort, as do few distinct times (rg_crowded), outstanding refresh claims (they go by batch index) and service times the in-order kernels do not hold.
// Bytes per record: 24 + 32 (scatter), 32 + 28 (sort), 28 + 16 (serve), 20 + 16, 16 + 16 (results): 228, streaming, against
// some 400, a third of them scattered, for six radix passes and a scan that gathers and scatters by sorted index.
// The work of a phase is dealt out in shares, in order, by a counter, and a block that finds none left waits until all are done:
// what it waits for is in the hands of blocks that run, so it does not matter how many of the grid run at a time.
#pragma once
#include "device_utils.cuh"

namespace hbf {

constexpr uint32_t kRgAvg = 1365, kRgCap = 2048;         // records per bucket: aimed at, and at most (sampling and chance: 1.5 is ten deviations)
constexpr uint32_t kRgSegs = 64, kRgSamples = 65536;
constexpr uint32_t kRgOut = 2048;                        // results per output bucket
constexpr uint32_t kRgChunk = 1024;                      // buckets of a share of the offsets phase
constexpr uint32_t kRgPad = 8;                           // words from counter to counter: one to a sector (eight in one: give 1,200 us for 40 M, now 690)

struct __align__(32) RegroupSlot { uint64_t addr; int64_t issue; uint64_t bf; uint64_t idx; };
struct RegroupArgs {
    RegroupSync *sync;
    uint32_t *cursor, *cursor_out, *offset, *part;       // [max_buckets][kRgPad], [out_buckets][kRgPad], [max_buckets], [chunks]
    RegroupSlot *slots; uint64_t *recs; uint32_t *idx;   // slots; [3 n], [n]: the ordered list
    int64_t *comp, *stall; ulonglong2 *entries;          // inside the slots' memory, once they have been read
    uint32_t max_buckets, out_buckets;
};
inline uint32_t regroup_buckets(uint64_t n) { return (uint32_t)(n / kRgAvg) + kRgSegs + 1u; }
inline uint32_t regroup_out_buckets(uint64_t n) { return (uint32_t)((n + kRgOut - 1) / kRgOut); }
inline RegroupArgs regroup_args(uint64_t n, const Workspace &ws, RegroupSync *sync) {
    RegroupArgs r{};
    r.sync = sync;
    if (!ws.rg_ctrl) return r;                               // (no room: the radix sort serves what is out of order)
    r.max_buckets = regroup_buckets(n); r.out_buckets = regroup_out_buckets(n);
    r.cursor = static_cast<uint32_t *>(ws.rg_ctrl); r.cursor_out = r.cursor + (size_t)kRgPad * r.max_buckets;
    r.offset = r.cursor_out + (size_t)kRgPad * r.out_buckets; r.part = r.offset + r.max_buckets;
    r.slots = static_cast<RegroupSlot *>(ws.rg_slots); r.recs = static_cast<uint64_t *>(ws.rg_recs); r.idx = static_cast<uint32_t *>(ws.rg_idx);
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    char *b = static_cast<char *>(ws.rg_slots);
    r.comp = reinterpret_cast<int64_t *>(b); r.stall = reinterpret_cast<int64_t *>(b + up(n * 8)); r.entries = reinterpret_cast<ulonglong2 *>(b + 2 * up(n * 8));
    return r;
}

// Where place p of bucket b lies: the buckets' stretches of 32 slots side by side, then their next 32.  All buckets fill at much
// the same pace, so the places in use at a time lie close together; with every bucket's slots in one piece each store fell into
// another page (scatter 1,054 us for 40 M records, most of it address translation).
__device__ __forceinline__ uint64_t rg_place(uint32_t buckets, uint32_t b, uint32_t p) { return ((uint64_t)(p >> 5) * buckets + b) * 32u + (p & 31u); }

// the shares of a phase, taken by warps.  silent: a share that is not reported as done (test support: see hbf_debug_wait_test)
template <class F>
__device__ __forceinline__ void rg_shares(RegroupSync *s, int phase, uint32_t shares, uint32_t silent, F &&f) {
    const int lane = threadIdx.x & 31;
    uint32_t done = 0;
    for (;;) {
        uint32_t k = 0;
        if (lane == 0) k = atomicAdd(&s->claim[phase], 1u);
        k = __shfl_sync(0xffffffffu, k, 0);
        if (k >= shares) break;
        f(k);
        if (k != silent) ++done;
    }
    if (done) {
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicAdd(&s->done[phase], done);
    }
}
constexpr uint32_t kRgNone = 0xffffffffu;
// all shares of a phase are done; false: the wait ran out
__device__ __forceinline__ bool rg_wait(RegroupSync *s, int phase, uint32_t shares, uint32_t limit) {
    bool ok = true;
    if (threadIdx.x == 0) {
        uint32_t polls = 0;
        while (ld_acquire_u32(&s->done[phase]) < shares) {
            if (++polls > limit) { ok = false; break; }
            __nanosleep(64);
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}
// the same in the begin kernel: a wait that runs out gives the batch up (its last kernel poisons the context)
__device__ __forceinline__ bool rg_wait_or_give_up(RegroupSync *s, int phase, uint32_t shares, uint32_t limit, BatchCtrl *ctrl) {
    const bool ok = rg_wait(s, phase, shares, limit);
    if (!ok && threadIdx.x == 0) { atomicExch(&ctrl->code, (int)HBF_E_TIMEOUT); ctrl->skip = 1; }
    return ok;
}

// The results of a regrouped batch back to batch order (blocks of the last kernel, in groups of 256 threads: a bucket each).  Behind the one
// wait nothing can fail any more: the first block that is past it calls commit() then, beside the others' work.  A block whose wait runs out leaves the rest
// to those that got past it; true: this block is the last to leave, and none did (nothing was committed, no result given back).
template <class Commit>
__device__ __forceinline__ bool rg_give_back(const RegroupArgs &r, uint64_t n, const DevState *state, int64_t *__restrict__ completion, int64_t *__restrict__ stall, ulonglong2 *s_out, Commit &&commit) {      // s_out: [kRgOut] of shared memory per group
    constexpr int kGroup = 256;
    __shared__ uint32_t s_b, s_bucket[4];
    constexpr uint32_t kGive = 1024;                         // records of a share
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t gives = (uint32_t)((n + kGive - 1) / kGive);
    rg_shares(r.sync, 3, gives, state->test_stage == 2u ? state->test_tile : kRgNone, [&](uint32_t g) {
        for (uint32_t at0 = 0; at0 < kGive; at0 += 128u) {
            uint64_t comp[4], issue[4]; uint32_t idx[4], at[4];
            const uint64_t i0 = (uint64_t)g * kGive + at0 + lane;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint64_t i = i0 + 32u * k;
                if (i < n) {
                    comp[k] = (uint64_t)__ldcs(reinterpret_cast<const long long *>(r.comp + i)); idx[k] = __ldcs(r.idx + i);
                    issue[k] = comp[k] - (uint64_t)__ldcs(reinterpret_cast<const long long *>(r.stall + i));
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) if (i0 + 32u * k < n) at[k] = atomicAdd(&r.cursor_out[(size_t)(idx[k] / kRgOut) * kRgPad], 1u);
#pragma unroll
            for (int k = 0; k < 4; ++k)                      // (a permutation: no bucket gets more than kRgOut; issue times have 47 bits)
                if (i0 + 32u * k < n) r.entries[rg_place(r.out_buckets, idx[k] / kRgOut, at[k])] = make_ulonglong2(comp[k], (issue[k] << 16) | (idx[k] % kRgOut));
        }
    });
    __syncthreads();
    if (!rg_wait(r.sync, 3, gives, state->spin_limit)) {
        if (tid == 0) { __threadfence(); s_b = atomicAdd(&r.sync->done[5], 1u); __threadfence(); }
        __syncthreads();
        return s_b == gridDim.x - 1u;
    }
    if (tid == 0) s_b = atomicAdd(&r.sync->claim[6], 1u);
    __syncthreads();
    if (s_b == 0u) commit();
    const int group = tid / kGroup, gtid = tid % kGroup;
    auto group_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kGroup) : "memory"); };
    s_out += (size_t)group * kRgOut;
    for (;;) {
        group_sync();                                        // the results of the bucket before have been read
        if (gtid == 0) s_bucket[group] = atomicAdd(&r.sync->claim[4], 1u);
        group_sync();
        const uint32_t b = s_bucket[group];
        if (b >= r.out_buckets) return false;
        const uint64_t base = (uint64_t)b * kRgOut;
        const uint32_t m = (uint32_t)min((uint64_t)kRgOut, n - base);
#pragma unroll 8
        for (uint32_t e = gtid; e < m; e += kGroup) {
            const ulonglong2 v = __ldcg(r.entries + rg_place(r.out_buckets, b, e));
            s_out[(uint32_t)v.y & 0xffffu] = make_ulonglong2(v.x, v.x - (v.y >> 16));
        }
        group_sync();
#pragma unroll 4
        for (uint32_t e = gtid; e < m; e += kGroup) {
            const ulonglong2 v = s_out[e];
            __stcs(reinterpret_cast<long long *>(completion + base + e), (long long)v.x);
            __stcs(reinterpret_cast<long long *>(stall + base + e), (long long)v.y);
        }
    }
}

}  // namespace hbf

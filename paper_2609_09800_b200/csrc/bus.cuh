// The channel-bus stage: sizes and arrays (bus_kernels.cu: the stage; submit_kernels.cu: its form by radix sort).
#pragma once
#include "device_utils.cuh"

namespace hbf {

struct BusMap { int64_t S, M; int f; };                    // B -> max(B + S, M); f: B does not matter
__device__ __forceinline__ BusMap bus_then(const BusMap &a, const BusMap &b) {       // a first, then b
    if (b.f) return b;
    BusMap r; r.S = a.S + b.S; r.M = max((int64_t)(a.M + b.S), b.M); r.f = a.f; return r;
}
__device__ __forceinline__ BusMap bus_identity() { BusMap r; r.S = 0; r.M = kNegInf; r.f = 0; return r; }
__device__ __forceinline__ BusMap bus_shfl_up(const BusMap &v, int o) {
    BusMap r; r.S = __shfl_up_sync(0xffffffffu, v.S, o); r.M = __shfl_up_sync(0xffffffffu, v.M, o); r.f = __shfl_up_sync(0xffffffffu, v.f, o);
    return r;
}

constexpr uint32_t kBusSegs = 64, kBusSamples = 65536;
constexpr uint32_t kBusAvg = 682, kBusCap = 2048;          // reads per bucket: aimed at, and at most (three times the average: channels and times differ)
constexpr uint32_t kBusMaxChannels = 2048;
constexpr uint32_t kBusHead = 16;                          // first entries of a bucket, kept in order
struct BusPlan {
    uint32_t hist[kBusSegs], top[kBusSegs], below[kBusSegs];  // samples of a stretch of time, their largest offset, 2^32 - 1 less their smallest
    uint32_t blocks, overflow, redo, shift;                 // redo: buckets on the list of those to be gone over again
    int64_t lo;
    uint32_t first[kBusSegs], last[kBusSegs];               // the part of a stretch that its share of the slices is spread over
    uint64_t cum[kBusSegs], mul[kBusSegs];                  // in 1/256 slices
};
struct BusState { int64_t S, M; };                          // a bucket as one map; then M: the bus before it
struct BusArgs {
    BusPlan *plan; uint32_t *cursor, *redo; BusState *state; ulonglong2 *entries, *heads;
    uint32_t channels, slices, cap; int64_t *busy;
};
inline uint32_t bus_slices(uint64_t n, uint32_t channels) { return (uint32_t)((n + (uint64_t)kBusAvg * channels - 1) / ((uint64_t)kBusAvg * channels)); }
inline uint32_t bus_cap(uint64_t n, uint32_t channels) {
    const uint64_t buckets = (uint64_t)bus_slices(n, channels) * channels, cap = 3 * (n / buckets) + 96;
    return (uint32_t)(cap < kBusCap ? cap : kBusCap);
}
inline size_t bus_entry_bytes(uint64_t n, uint32_t channels) {
    if (channels > kBusMaxChannels) return 0;
    const size_t buckets = (size_t)bus_slices(n, channels) * channels, a = (size_t)3 * n + 96 * buckets, b = (size_t)kBusCap * buckets;
    return (a < b ? a : b) * sizeof(ulonglong2);             // (at least buckets times places, and never less for more records)
}
inline size_t bus_head_bytes(uint64_t n, uint32_t channels) {
    return channels > kBusMaxChannels ? 0 : (size_t)bus_slices(n, channels) * channels * (kBusHead * sizeof(ulonglong2) + sizeof(BusState) + 8);
}
static_assert(sizeof(BatchCtrl) <= kBusPlanAt && sizeof(BusPlan) <= kBusPlanBytes && sizeof(BusPlan) % 4 == 0, "the plan's place");
inline BusPlan *bus_plan_of(BatchCtrl *bc) { return reinterpret_cast<BusPlan *>(reinterpret_cast<char *>(bc) + kBusPlanAt); }
inline BusArgs bus_args(uint64_t n, uint32_t channels, const Workspace &ws, BatchCtrl *bc, int64_t *busy) {
    BusArgs b{};
    b.plan = bus_plan_of(bc); b.channels = channels; b.busy = busy;
    if (!ws.bus_heads) return b;                            // slices = 0: the radix sort serves the batch
    b.slices = bus_slices(n, channels); b.cap = bus_cap(n, channels);
    const size_t buckets = (size_t)b.slices * channels;
    b.heads = static_cast<ulonglong2 *>(ws.bus_heads);
    b.state = reinterpret_cast<BusState *>(b.heads + kBusHead * buckets);
    b.cursor = reinterpret_cast<uint32_t *>(b.state + buckets); b.redo = b.cursor + buckets;
    b.entries = static_cast<ulonglong2 *>(ws.rg_slots);
    return b;
}

}  // namespace hbf

// The time-bin energy ledger: how one event is booked (see energy_bins.cu for the definition).
#pragma once
#include "device_utils.cuh"

namespace hbf {

__device__ __forceinline__ void ledger_add(unsigned long long *ledger, uint32_t n_dies, uint32_t n_bins, int64_t cur_bin,
                                           uint32_t die, int64_t bin, int64_t pj) {
    bin = max(bin, cur_bin);
    bin = min(bin, cur_bin + (int64_t)n_bins - 1);
    if (pj) atomicAdd(&ledger[(size_t)(bin % (int64_t)n_bins) * n_dies + die], (unsigned long long)pj);
}

// one event: energy pj over [start, start + s), split over the bins it overlaps.  Every bin before the event's last one
// gets floor(pj * overlap / s); the overlap is a whole bin for all of them but the first, so the bins that the ring clamps
// into its first or last slot are booked in one step each and the loop only walks bins inside the ring: at most n_bins
// turns, whatever the ratio of service time to bin width.
__device__ __forceinline__ void ledger_event(unsigned long long *ledger, uint32_t n_dies, uint32_t n_bins, int64_t cur_bin, int64_t bin_ns,
                                             uint32_t die, int64_t start, int64_t s, int64_t pj) {
    const int64_t end = start + s;
    const int64_t b0 = start / bin_ns, b1 = (end - 1) / bin_ns;
    if (b0 == b1) { ledger_add(ledger, n_dies, n_bins, cur_bin, die, b0, pj); return; }
    const int64_t ring_hi = cur_bin + (int64_t)n_bins - 1;
    const int64_t first = (int64_t)(((unsigned __int128)(uint64_t)pj * (uint64_t)((b0 + 1) * bin_ns - start)) / (uint64_t)s);
    const int64_t full = (int64_t)(((unsigned __int128)(uint64_t)pj * (uint64_t)bin_ns) / (uint64_t)s);
    auto run = [&](int64_t from, int64_t to) {               // shares of the bins [from, to), from >= b0, to <= b1
        return to <= from ? (int64_t)0 : (from == b0 ? first + (to - from - 1) * full : (to - from) * full);
    };
    const int64_t below_end = min(b1, max(b0, cur_bin));     // bins [b0, below_end) lie before the ring
    const int64_t above_begin = min(b1, max(below_end, ring_hi));   // bins [above_begin, b1) lie at or past its last slot
    int64_t given = 0;
    const int64_t below = run(b0, below_end);
    ledger_add(ledger, n_dies, n_bins, cur_bin, die, cur_bin, below); given += below;
    for (int64_t b = below_end; b < above_begin; ++b) {
        const int64_t share = b == b0 ? first : full;
        ledger_add(ledger, n_dies, n_bins, cur_bin, die, b, share); given += share;
    }
    const int64_t above = run(above_begin, b1);
    ledger_add(ledger, n_dies, n_bins, cur_bin, die, ring_hi, above); given += above;
    ledger_add(ledger, n_dies, n_bins, cur_bin, die, b1, pj - given);
}

}  // namespace hbf

// The time-bin energy ledger: how one event is booked (see energy_bins.cu for the definition).
#pragma once
#include "device_utils.cuh"

namespace hbf {

// Divisions are what an event costs: one by the bin width, none by the ring's size (cur_slot: where the ring's first bin, cur_bin,
// lies), and a share's product is divided in 64 bits where it fits them, nearly always (in 128 bits that is a call of some
// hundred instructions, which one event in five, over a bin's end, took a whole warp through twice).  A coupled window of 1 ms 77 -> 76 us.
struct Ledger { unsigned long long *at; int64_t bin_ns, cur_bin; uint32_t n_dies, n_bins, cur_slot; };
__device__ __forceinline__ Ledger make_ledger(unsigned long long *at, uint32_t n_dies, uint32_t n_bins, int64_t cur_bin, int64_t bin_ns) {
    Ledger l; l.at = at; l.bin_ns = bin_ns; l.cur_bin = cur_bin; l.n_dies = n_dies; l.n_bins = n_bins; l.cur_slot = n_bins ? (uint32_t)(cur_bin % (int64_t)n_bins) : 0u;
    return l;
}
__device__ __forceinline__ void ledger_add(const Ledger &l, uint32_t die, int64_t bin, int64_t pj) {
    const int64_t ahead = min(max(bin - l.cur_bin, (int64_t)0), (int64_t)l.n_bins - 1);
    const uint64_t slot = (uint64_t)l.cur_slot + (uint64_t)ahead;
    if (pj) atomicAdd(&l.at[(slot >= l.n_bins ? slot - l.n_bins : slot) * l.n_dies + die], (unsigned long long)pj);
}
__device__ __forceinline__ int64_t ledger_share(int64_t pj, int64_t overlap, int64_t s) {     // floor(pj * overlap / s)
    if (__umul64hi((uint64_t)pj, (uint64_t)overlap) == 0ull) return (int64_t)(((uint64_t)pj * (uint64_t)overlap) / (uint64_t)s);
    return (int64_t)(((unsigned __int128)(uint64_t)pj * (uint64_t)overlap) / (uint64_t)s);
}

// one event: energy pj over [start, start + s), split over the bins it overlaps.  Every bin before the event's last one
// gets floor(pj * overlap / s); the overlap is a whole bin for all of them but the first, so the bins that the ring clamps
// into its first or last slot are booked in one step each and the loop only walks bins inside the ring: at most n_bins
// turns, whatever the ratio of service time to bin width.
__device__ __forceinline__ void ledger_event(const Ledger &l, uint32_t die, int64_t start, int64_t s, int64_t pj) {
    const int64_t b0 = start / l.bin_ns, within = start - b0 * l.bin_ns;
    if (s <= l.bin_ns - within) { ledger_add(l, die, b0, pj); return; }
    const int64_t b1 = b0 + (within + s - 1) / l.bin_ns;
    const int64_t ring_hi = l.cur_bin + (int64_t)l.n_bins - 1;
    const int64_t first = ledger_share(pj, l.bin_ns - within, s);
    const int64_t full = b1 - b0 > 1 ? ledger_share(pj, l.bin_ns, s) : 0;   // (no whole bin between the first and the last)
    auto run = [&](int64_t from, int64_t to) {               // shares of the bins [from, to), from >= b0, to <= b1
        return to <= from ? (int64_t)0 : (from == b0 ? first + (to - from - 1) * full : (to - from) * full);
    };
    const int64_t below_end = min(b1, max(b0, l.cur_bin));     // bins [b0, below_end) lie before the ring
    const int64_t above_begin = min(b1, max(below_end, ring_hi));   // bins [above_begin, b1) lie at or past its last slot
    int64_t given = 0;
    const int64_t below = run(b0, below_end);
    ledger_add(l, die, l.cur_bin, below); given += below;
    for (int64_t b = below_end; b < above_begin; ++b) {
        const int64_t share = b == b0 ? first : full;
        ledger_add(l, die, b, share); given += share;
    }
    const int64_t above = run(above_begin, b1);
    ledger_add(l, die, ring_hi, above); given += above;
    ledger_add(l, die, b1, pj - given);
}

}  // namespace hbf

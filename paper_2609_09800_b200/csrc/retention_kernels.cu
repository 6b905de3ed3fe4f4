// Retention, refresh and wear (Design D4) as data-parallel kernels.
//   per epoch (hbf_retention_advance): region temperatures -> Arrhenius damage rate per region -> damage and
//     eligibility per block -> the refresh plan.  The paper's emission order (eligibility epoch, channel round
//     robin, die round robin, zone, block, page) is not walked: every quantum computes its own place in it.  With
//     r_die the quantum's rank in its die's (zone, plane, block, page) list, the dies of a channel served in turn
//     put it at r_ch = sum over the channel's dies d' of min(len[d'], r_die), plus the dies before its own that
//     still have a quantum of that rank; the channels served in turn put it at the same expression over channels
//     with r_ch.  The ranks come from one scan per die; the rest is arithmetic on the per-die lengths.  (k_ret_plan runs the
//     other way: it lays the plan out round by round, a lane per channel, from where the dies stand at a warp's first round.)
//   per batch (hbf_submit_batch): the claim window finds the batch index below which the modeled accesses claim
//     one outstanding quantum each (they claim in index order), before the batch is served; after it, the reads
//     are counted into their blocks' disturb counters, blocks whose last quantum is now claimed commit, and the
//     claimed energy is booked on the claimants' dies.
//   idle time (hbf_retention_decay) drains quanta on an account of its own and commits likewise.
#include <algorithm>

#include "device_utils.cuh"

namespace hbf {

__device__ __forceinline__ bool ret_ready(const RangeSnap &rs, const hbf_access_t *acc, uint64_t i, uint64_t *off, uint32_t *bytes, uint32_t *op) {
    const uint64_t *rec = reinterpret_cast<const uint64_t *>(acc + i);
    const uint64_t addr = ld_after(rec), bf = ld_after(rec + 2);
    const int64_t issue = (int64_t)ld_after(rec + 1);
    int g = 0;
    if (classify(rs, addr, issue, (uint32_t)bf, (uint32_t)(bf >> 32), &g) != HBF_ST_READY) return false;
    if (off) *off = rs.media_offset[g] + (addr - rs.base[g]);
    if (bytes) *bytes = (uint32_t)bf;
    if (op) *op = (uint32_t)(bf >> 32) & 1u;
    return true;
}

__device__ __forceinline__ void load_ranges(RangeSnap *dst, const RangeSnap *src) {
    for (int i = threadIdx.x; i < (int)(sizeof(RangeSnap) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t *>(dst)[i] = reinterpret_cast<const uint32_t *>(src)[i];
}

// inclusive scan of one value per thread over the block; *total (nullable) receives the sum
template <int THREADS>
__device__ __forceinline__ uint32_t block_scan_incl(uint32_t v, uint32_t *total) {
    __shared__ uint32_t s_w[THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const uint32_t y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
    __syncthreads();                                          // the previous use of s_w is over
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    uint32_t before = 0, sum = 0;
    for (int w = 0; w < THREADS / 32; ++w) { const uint32_t t = s_w[w]; if (w < warp) before += t; sum += t; }
    if (total) *total = sum;
    return x + before;
}

// whether this block is the last of the grid to come here: every other one's writes are visible then (the counter is 0 between kernels)
__device__ __forceinline__ bool ret_last_block(RetState *st) {
    __shared__ uint32_t s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) { s_last = atomicAdd(&st->epoch_blocks, 1ull) == gridDim.x - 1u ? 1u : 0u; __threadfence(); if (s_last) st->epoch_blocks = 0ull; }
    __syncthreads();
    return s_last != 0u;
}

// =====================================================================================================
// claim window: how far into the batch do the outstanding quanta reach?
// =====================================================================================================
constexpr int kRetTile = 1024;
// Tiles are handed out in order from a counter, eight at a time; a block stops taking tiles once the tiles already finished hold at
// least as many modeled accesses as there is debt (the tiles in flight only add to that).  Work is proportional to the reach of the
// debt, not to the batch.  A debt of as many quanta as the batch has records reaches past its end whatever they are: nothing is
// counted then, and what the batch claims is the number of its modeled accesses (kRetAll).
// (a tile of 1,024 at a time, 256 threads: 164 us for 20.6 M of 24 M records, and 37 for the search; now 106, 4.7 TB/s,
// and 14.  The search is the last block's, commits and accounts behind the batch are one kernel, and all overlap their starts: two batches of 500,000
// with an epoch between 259 -> 237 us, of 24 M 1,204 -> 1,176)
constexpr int kRetWinThreads = 1024, kRetWinTiles = 8;
constexpr unsigned long long kRetAll = ~0ull;
__global__ void __launch_bounds__(kRetWinThreads)
k_ret_window(const hbf_access_t *acc, uint64_t n, const RangeSnap *__restrict__ ranges_g, const __grid_constant__ RetDev r) {
    __shared__ RangeSnap rs;
    __shared__ uint32_t s_first, s_cnt[2][kRetWinTiles];
    pdl_wait();
    pdl_trigger();
    RetState *st = r.st;
    const unsigned long long debt = st->planned - st->claimed - st->decayed;
    if (debt == 0ull || debt >= n) {
        if (blockIdx.x == 0 && threadIdx.x == 0) { st->claim_limit = debt ? n : 0ull; st->claims_now = debt && n ? kRetAll : 0ull; }
        return;
    }
    load_ranges(&rs, ranges_g);
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < 2 * kRetWinTiles) (&s_cnt[0][0])[tid] = 0u;
    const uint64_t n_tiles = (n + kRetTile - 1) / kRetTile;
    for (uint32_t turn = 0;; turn ^= 1u) {
        __syncthreads();                                     // (the counts of the turn before have been read, the tables are there)
        if (tid == 0) s_first = *reinterpret_cast<volatile unsigned long long *>(&st->counted) >= debt ? 0xffffffffu : (uint32_t)min(atomicAdd(&st->tickets, (unsigned long long)kRetWinTiles), 0xffffffffull);
        if (tid < kRetWinTiles) s_cnt[turn ^ 1u][tid] = 0u;
        __syncthreads();
        const uint64_t first = s_first;
        if (first >= n_tiles) break;
        bool is[kRetWinTiles];
#pragma unroll
        for (int k = 0; k < kRetWinTiles; ++k) { const uint64_t i = (first + k) * kRetTile + tid; is[k] = i < n && ret_ready(rs, acc, i, nullptr, nullptr, nullptr); }
#pragma unroll
        for (int k = 0; k < kRetWinTiles; ++k) { const uint32_t c = (uint32_t)__popc(__ballot_sync(0xffffffffu, is[k])); if (lane == k && c) atomicAdd(&s_cnt[turn][k], c); }
        __syncthreads();
        if (tid == 0) {
            unsigned long long sum = 0;
            for (int k = 0; k < kRetWinTiles; ++k) if (first + k < n_tiles) { r.tile_count[first + k] = s_cnt[turn][k]; sum += s_cnt[turn][k]; }
            __threadfence();
            atomicAdd(&st->counted, sum);
        }
    }
    // the last block: the tile in which the running count reaches the debt, then the record inside it
    if (!ret_last_block(st)) return;
    __shared__ unsigned long long s_base, s_before;
    __shared__ uint32_t s_found;
    const uint64_t T = min((uint64_t)__ldcg(&st->tickets), n_tiles);
    if (tid == 0) { s_base = 0ull; s_found = 0xffffffffu; }
    __syncthreads();
    constexpr int kPer = 8;
    for (uint64_t chunk = 0; chunk < T; chunk += kRetTile * kPer) {
        const uint64_t t0 = chunk + (uint64_t)tid * kPer;
        uint32_t v[kPer], mine = 0, sum = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) { v[k] = t0 + k < T ? __ldcg(r.tile_count + t0 + k) : 0u; mine += v[k]; }
        const uint32_t incl = block_scan_incl<kRetTile>(mine, &sum);
        unsigned long long at = s_base + incl - mine;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            if (at < debt && at + v[k] >= debt) { s_found = (uint32_t)(t0 + k); s_before = at; }
            at += v[k];
        }
        __syncthreads();
        if (s_found != 0xffffffffu) break;
        if (tid == 0) s_base += sum;
        __syncthreads();
    }
    const uint32_t found = s_found;
    if (found == 0xffffffffu) {                               // the whole batch claims and debt remains
        if (tid == 0) { st->claim_limit = n; st->claims_now = s_base; }
    } else {
        const uint32_t need = (uint32_t)(debt - s_before);    // 1 .. the tile's count
        const uint64_t i = (uint64_t)found * kRetTile + (uint64_t)tid;
        const uint32_t flag = (i < n && ret_ready(rs, acc, i, nullptr, nullptr, nullptr)) ? 1u : 0u;
        const uint32_t incl = block_scan_incl<kRetTile>(flag, nullptr);
        if (flag && incl == need) { st->claim_limit = i + 1ull; st->claims_now = debt; }
    }
    if (tid == 0) { st->tickets = 0ull; st->counted = 0ull; }
}

cudaError_t launch_ret_window(const hbf_access_t *acc, uint64_t n, const RangeSnap *ranges, const RetDev &r, int sm_count, bool *plain_next, cudaStream_t st) {
    const uint64_t tiles = (n + kRetTile - 1) / kRetTile;
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((tiles + kRetWinTiles - 1) / kRetWinTiles, (uint64_t)sm_count * 2));
    g_kernel_launches += 1;
    return launch_first(plain_next, k_ret_window, grid, kRetWinThreads, 0, st, acc, n, ranges, r);
}

// =====================================================================================================
// after the batch: read disturb, commits, bookkeeping
// =====================================================================================================
// The in-order serve pass counts the reads into the disturb counters as it streams the batch (observed_inline).  This
// pass covers the other cases: the batch was served without that pass (count now), or the pass ran and the batch was
// then refused (take the counts back: the same reads, the same amounts).
__global__ void __launch_bounds__(256)
k_ret_observe(const hbf_access_t *__restrict__ acc, uint64_t n, const RangeSnap *__restrict__ ranges_g,
              const ModelParams *__restrict__ mp_g, const hbf_batch_result_t *result, const __grid_constant__ RetDev r) {
    __shared__ RangeSnap rs;
    __shared__ ModelParams mp;
    pdl_wait();
    pdl_trigger();
    const bool ok = result->code == HBF_OK, inline_done = r.st->observed_inline != 0u;
    if (ok == inline_done) return;                           // counted and accepted, or neither
    const bool undo = inline_done;
    load_ranges(&rs, ranges_g);
    for (int i = threadIdx.x; i < (int)(sizeof(ModelParams) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t *>(&mp)[i] = reinterpret_cast<const uint32_t *>(mp_g)[i];
    __syncthreads();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        uint64_t off; uint32_t bytes, op;
        if (!ret_ready(rs, acc, i, &off, &bytes, &op) || op) continue;
        const uint64_t in_page = off & ((1ull << mp.page_shift) - 1ull);
        const uint32_t npages = (uint32_t)((in_page + bytes + (1ull << mp.page_shift) - 1ull) >> mp.page_shift);
        atomicAdd(&r.disturb[ret_block_of(mp, r, off)], undo ? 0u - npages : npages);
    }
}

// a block whose last quantum lies below the watermark commits one cycle and clears its counters
__device__ __forceinline__ void ret_commit_due(const RetDev &r, unsigned long long mark) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b < r.n_blocks; b += stride) {
        if (r.epoch_of[b] == 0u || r.last_pos[b] >= mark) continue;
        ret_commit_block(r, b);
    }
}
__global__ void __launch_bounds__(256) k_ret_commit(RetDev r) { ret_commit_due(r, r.st->claimed + r.st->decayed); }

// the same behind a batch; the last block books what the batch claimed
__global__ void __launch_bounds__(256) k_ret_close(const hbf_batch_result_t *result, int64_t *pending, int64_t quantum_pj, uint32_t n_dies, const __grid_constant__ RetDev r) {
    pdl_wait();
    pdl_trigger();
    RetState *st = r.st;
    const bool ok = result->code == HBF_OK;
    const unsigned long long claims = !ok ? 0ull : st->claims_now == kRetAll ? (unsigned long long)result->n_modeled : st->claims_now;
    if (ok) ret_commit_due(r, st->claimed + st->decayed + claims);
    if (!ret_last_block(st)) return;
    for (uint32_t d = threadIdx.x; d < n_dies; d += blockDim.x) {
        const uint32_t c = r.die_claims[d];
        if (ok && c) pending[d] += (int64_t)c * quantum_pj;
        r.die_claims[d] = 0u;
    }
    if (threadIdx.x == 0) {
        st->claimed += claims;
        st->claims_now = 0ull; st->claim_limit = 0ull; st->observed_inline = 0u;
    }
}

static unsigned ret_grid(uint64_t items, int sm_count) {
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((items + 255) / 256, (uint64_t)sm_count * 8));
}

cudaError_t launch_ret_close(const hbf_access_t *acc, uint64_t n, const RangeSnap *ranges, const ModelParams *mp_dev, const ModelParams &mp,
                             const hbf_batch_result_t *result, int64_t *pending, int binned, const RetDev &r, int sm_count, bool *plain_next, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    if (n) e = launch_first(plain_next, k_ret_observe, ret_grid(n, sm_count), 256, 0, st, acc, n, ranges, mp_dev, result, r);
    if (e != cudaSuccess) return e;
    const int64_t page = (int64_t)1 << mp.page_shift;
    const int64_t quantum_pj = mp.e_cmd_read_pj + mp.e_byte_read_pj * page + mp.e_cmd_prog_pj + mp.e_byte_prog_pj * page;
    // (with the time bins on, the ledger has the energy)
    e = launch_first(plain_next, k_ret_close, ret_grid(r.n_blocks, sm_count), 256, 0, st, result, pending, binned ? (int64_t)0 : quantum_pj, mp.n_dies, r);
    g_kernel_launches += n ? 2 : 1;
    return e;
}

// =====================================================================================================
// one epoch: temperatures -> damage -> eligibility -> plan.  Three launches that overlap their starts (two when the caller gives
// the temperatures): the regions' hottest cells; a block per die for rate, damage, eligibility and ranks; the plan, whose last
// block closes the epoch.  65,536 blocks on a 128 x 128 field: 36 us of kernels and 8 gaps as eight
// launches, 17 us and 3 overlapped starts now (a coupled window of 1 ms: 106 -> 76 us).
// Between epochs region_max holds nothing and chan_len zeros: the last block of the plan kernel leaves them so.
// =====================================================================================================
__device__ __forceinline__ int ordered_int(float f) { const int k = __float_as_int(f); return k >= 0 ? k : k ^ 0x7fffffff; }
__device__ __forceinline__ float ordered_float(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff); }

__global__ void __launch_bounds__(256)
k_ret_region_max(const float *__restrict__ theta, const int32_t *__restrict__ cell_region, uint64_t n_cells, RetDev r) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x, first = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int32_t g = first < n_cells ? cell_region[first] : -1;   // (the floorplan does not change: read before the field is there)
    pdl_wait();
    pdl_trigger();
    for (uint64_t i = first; i - threadIdx.x % 32u < n_cells; i += stride) {     // (whole warps)
        if (i != first) g = i < n_cells ? cell_region[i] : -1;
        const int v = g >= 0 ? ordered_int(ld_after(theta + i)) : 0;
        int32_t same;
        __match_all_sync(0xffffffffu, g, &same);             // cells side by side mostly lie in one region
        if (same) {
            const int m = __reduce_max_sync(0xffffffffu, v);
            if (g >= 0 && lane_id() == 0) atomicMax(&r.region_max[g], m);
        } else if (g >= 0) {
            atomicMax(&r.region_max[g], v);
        }
    }
}

// a block per die: Arrhenius lifetime at its region's temperature (first equation of D4) and the damage it adds per block in
// this epoch (second equation of D4); eligibility; the list of the newly eligible blocks in the die's (zone, plane, block) order
constexpr int kRetDieThreads = 256;
__global__ void __launch_bounds__(kRetDieThreads)
k_ret_die(RetDev r, const int32_t *__restrict__ die_region, uint32_t planes, uint32_t dies, int from_field, float ambient_c, double dt_s) {
    __shared__ double s_rate;
    pdl_wait();
    pdl_trigger();
    const uint32_t epoch = r.st->epoch + 1u, die = blockIdx.x;
    const uint32_t per_die = planes * r.bpp, zone_span = planes * r.bpz;
    if (threadIdx.x == 0) {
        const uint32_t g = die_region ? (uint32_t)die_region[die] : 0u;
        double temp_c;
        if (from_field) {
            const float rise = ordered_float(r.region_max[g]);
            temp_c = rise == -INFINITY ? (double)ambient_c : (double)(ambient_c + rise);
        } else {
            temp_c = r.region_temp[g];
        }
        const double life = r.l_ref_s * exp(r.ea_over_kb * (1.0 / (temp_c + 273.15) - 1.0 / r.t_ref_k));
        s_rate = r.accel * dt_s / life;
    }
    uint32_t running = 0;
    for (uint32_t o0 = 0; o0 < per_die; o0 += kRetDieThreads) {
        const uint32_t o = o0 + threadIdx.x;
        uint64_t b = 0; uint32_t flag = 0, was = 0, hits = 0; double d = 0.0; bool worn = true;
        if (o < per_die) {
            const uint32_t zone = o / zone_span, rem = o % zone_span, pl = rem / r.bpz, kk = rem % r.bpz;
            b = ((uint64_t)die * planes + pl) * r.bpp + zone * r.bpz + kk;
            worn = r.worn[b] != 0; d = r.damage[b]; was = r.epoch_of[b];
            if (r.disturb_limit) hits = r.disturb[b];
        }
        if (o0 == 0u) __syncthreads();                       // (the rate)
        if (!worn) {
            d += s_rate;
            r.damage[b] = d;
            if (was == 0u && (d >= r.lead || (r.disturb_limit && hits >= r.disturb_limit))) { r.epoch_of[b] = epoch; flag = 1u; }
        }
        uint32_t sum = 0;
        const uint32_t incl = block_scan_incl<kRetDieThreads>(flag, &sum);
        if (flag) r.list[(uint64_t)die * per_die + running + incl - 1u] = (uint32_t)b;
        running += sum;
    }
    if (threadIdx.x == 0) {
        const unsigned long long len = (unsigned long long)running * r.ppb;
        r.die_len[die] = len;
        if (len) atomicAdd(&r.chan_len[die / dies], len);
    }
}

// the last block of the plan kernel: every other one has read what changes here
__device__ __forceinline__ void ret_close_epoch(const RetDev &r, uint32_t channels) {
    __shared__ uint32_t s_last;
    RetState *st = r.st;
    __syncthreads();
    if (threadIdx.x == 0) { __threadfence(); s_last = atomicAdd(&st->epoch_blocks, 1ull) == gridDim.x - 1u ? 1u : 0u; }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    unsigned long long total = 0;
    for (uint32_t c = threadIdx.x; c < channels; c += blockDim.x) { total += __ldcg(r.chan_len + c); r.chan_len[c] = 0ull; }
    total = (unsigned long long)warp_sum((long long)total);
    if (lane_id() == 0 && total) atomicAdd(&st->planned, total);
    for (uint32_t g = threadIdx.x; g < r.n_regions; g += blockDim.x) r.region_max[g] = ordered_int(-INFINITY);
    if (threadIdx.x == 0) { st->epoch += 1u; st->epoch_blocks = 0ull; }
}

// The plan, in the order it is laid out: a round takes a quantum from every channel that has one left, so the places of a round
// lie side by side.  A lane of a warp is a channel (up to four of them), the warp takes a run of consecutive rounds: it finds where
// the channels' dies stand at its first round and steps from there, the die's next page or the channel's next die.  Every
// length of an epoch is below 2^32 (a quantum id is 32 bits and a block is planned at most once at a time).
// 20.6 M quanta: a warp per eligible block that worked out the place of every page by itself (300 instructions per 32, a store of
// 4 bytes all over the plan each) took 284 us, this 73.
constexpr int kRetPlanThreads = 256, kRetPlanWarps = kRetPlanThreads / 32;
constexpr uint32_t kRetPlanCells = 2048;                  // channels x dies: nine tables of that many words in shared memory
template <int G>
__global__ void __launch_bounds__(kRetPlanThreads)
k_ret_plan(RetDev r, uint32_t channels, uint32_t dies, uint32_t planes) {
    extern __shared__ uint32_t ret_smem[];
    const uint32_t cells = channels * dies;
    uint32_t *s_len = ret_smem;                              // [dies][channels] quanta of the die
    uint32_t *s_blk = ret_smem + (1u + threadIdx.x / 32u) * cells;   // [dies][channels] per warp: the block that the die's next page lies in
    const int tid = threadIdx.x, lane = tid & 31;
    pdl_wait();
    pdl_trigger();
    const RetState *st = r.st;
    const unsigned long long base = st->planned;
    const uint64_t base_mod = base % r.plan_cap;
    const uint32_t per_die = planes * r.bpp, ppb = r.ppb;
    uint32_t len[G], most = 0;
#pragma unroll
    for (int g = 0; g < G; ++g) { const uint32_t c = g * 32u + lane; len[g] = c < channels ? (uint32_t)r.chan_len[c] : 0u; most = max(most, len[g]); }
    most = __reduce_max_sync(0xffffffffu, most);             // rounds (the same for every warp)
    if (most) for (uint32_t k = tid; k < cells; k += kRetPlanThreads) s_len[(k % dies) * channels + k / dies] = (uint32_t)r.die_len[k];
    __syncthreads();
    const uint32_t warps = gridDim.x * kRetPlanWarps, run = max(32u, (most + warps - 1u) / warps);
    const uint64_t first = (uint64_t)(blockIdx.x * kRetPlanWarps + tid / 32) * run;
    if (first < most) {
        const uint32_t r0 = (uint32_t)first, r1 = (uint32_t)min((uint64_t)most, first + run);
        uint32_t pos = 0, turn[G], page[G], at[G], mask[G], die[G], next[G];   // turn: quanta that each of the channel's dies has given, as page and place in the list
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const uint32_t c = g * 32u + lane;
            pos += min(len[g], r0);
            turn[g] = 0u; mask[g] = 0u; next[g] = 0u; die[g] = 0u; page[g] = 0u; at[g] = 0u;
            if (c >= channels || len[g] <= r0) continue;
            uint32_t left = r0;
            for (;;) {                                       // the stretch between two ends of dies that the round falls into
                mask[g] = 0u; next[g] = 0xffffffffu;
                for (uint32_t d = 0; d < dies; ++d) { const uint32_t l = s_len[d * channels + c]; if (l > turn[g]) { mask[g] |= 1u << d; next[g] = min(next[g], l); } }
                const uint32_t a = (uint32_t)__popc(mask[g]);
                const uint64_t here = (uint64_t)(next[g] - turn[g]) * a;
                if (left < here) {
                    turn[g] += left / a;
                    uint32_t m = mask[g];
                    for (uint32_t k = left % a; k > 0u; --k) m &= m - 1u;
                    die[g] = (uint32_t)__ffs((int)m) - 1u;
                    break;
                }
                left -= (uint32_t)here; turn[g] = next[g];
            }
            at[g] = turn[g] / ppb; page[g] = turn[g] % ppb;
            for (uint32_t d = 0; d < dies; ++d) if ((mask[g] >> d) & 1u) s_blk[d * channels + c] = r.list[(uint64_t)(c * dies + d) * per_die + at[g]];
        }
        pos = __reduce_add_sync(0xffffffffu, pos);           // quanta of the rounds before
        const unsigned lt = lanemask_lt();
        for (uint32_t round = r0; round < r1; ++round) {
            uint32_t before = 0;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const bool on = len[g] > round;
                const unsigned who = __ballot_sync(0xffffffffu, on);
                if (on) {
                    const uint32_t c = g * 32u + lane, p = pos + before + (uint32_t)__popc(who & lt), b = s_blk[die[g] * channels + c];
                    uint64_t slot = base_mod + p;
                    if (slot >= r.plan_cap) slot -= r.plan_cap;
                    r.plan[slot] = b * ppb + page[g];
                    if (page[g] + 1u == ppb) r.last_pos[b] = base + p;   // the last page's place: a block's pages go out in order
                    const uint32_t later = mask[g] & ~((2u << die[g]) - 1u);
                    if (later) die[g] = (uint32_t)__ffs((int)later) - 1u;
                    else {
                        turn[g] += 1u; page[g] += 1u;
                        const bool turned = page[g] == ppb;
                        if (turned) { page[g] = 0u; at[g] += 1u; }
                        if (turn[g] == next[g]) {            // some of the dies have given all they had
                            mask[g] = 0u; next[g] = 0xffffffffu;
                            for (uint32_t d = 0; d < dies; ++d) { const uint32_t l = s_len[d * channels + c]; if (l > turn[g]) { mask[g] |= 1u << d; next[g] = min(next[g], l); } }
                        }
                        if (turned) for (uint32_t d = 0; d < dies; ++d) if ((mask[g] >> d) & 1u) s_blk[d * channels + c] = r.list[(uint64_t)(c * dies + d) * per_die + at[g]];
                        die[g] = mask[g] ? (uint32_t)__ffs((int)mask[g]) - 1u : 0u;
                    }
                }
                before += (uint32_t)__popc(who);
            }
            pos += before;
        }
    }
    ret_close_epoch(r, channels);
}

// The same plan for any number of channels and dies: `split` blocks per die, one warp per eligible block, its lanes over the
// block's pages, every page's place by itself (the sums at the head of this file).
__global__ void __launch_bounds__(256)
k_ret_emit(RetDev r, uint32_t channels, uint32_t dies, uint32_t planes, uint32_t split) {
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t die = blockIdx.x / split, part = blockIdx.x % split, ch = die / dies, di = die % dies;
    const unsigned long long base = r.st->planned;
    const uint64_t base_mod = base % r.plan_cap;
    const uint32_t blocks = (uint32_t)(r.die_len[die] / r.ppb);
    const unsigned long long *dlen = r.die_len + (size_t)ch * dies;
    for (uint32_t k = part * 8u + warp; k < blocks; k += split * 8u) {
        const uint64_t b = r.list[(uint64_t)die * planes * r.bpp + k];
        for (uint32_t pg = (uint32_t)lane; pg < r.ppb; pg += 32u) {
            const uint32_t r_die = k * r.ppb + pg;
            uint32_t r_ch = 0, pos = 0;
            for (uint32_t d = 0; d < dies; ++d) { const uint32_t len = (uint32_t)dlen[d]; r_ch += min(len, r_die) + ((d < di && len > r_die) ? 1u : 0u); }
            for (uint32_t c = 0; c < channels; ++c) { const uint32_t len = (uint32_t)r.chan_len[c]; pos += min(len, r_ch) + ((c < ch && len > r_ch) ? 1u : 0u); }
            uint64_t slot = base_mod + pos;
            if (slot >= r.plan_cap) slot -= r.plan_cap;
            r.plan[slot] = (uint32_t)(b * r.ppb + pg);
            if (pg + 1u == r.ppb) r.last_pos[b] = base + pos;
        }
    }
    ret_close_epoch(r, channels);
}

cudaError_t launch_ret_advance(const RetDev &r, const ModelParams &mp, const ThermalDev *field, const float *theta, const int32_t *die_region,
                               int have_temps, int64_t dt_ns, int sm_count, bool *plain_next, cudaStream_t st) {
    const int from_field = have_temps ? 0 : 1;
    const float ambient = from_field ? field->ambient_c : 0.0f;
    cudaError_t e = cudaSuccess;
    if (from_field) {
        const uint64_t cells = (uint64_t)field->H * field->W;
        e = launch_first(plain_next, k_ret_region_max, ret_grid(cells, sm_count), 256, 0, st, theta, field->cell_region, cells, r);
        g_kernel_launches += 1;
    }
    if (e == cudaSuccess) e = launch_first(plain_next, k_ret_die, mp.n_dies, kRetDieThreads, 0, st, r, die_region, mp.planes, mp.dies, from_field, ambient, (double)dt_ns * 1e-9);
    if (e == cudaSuccess) {
        const uint32_t cells = mp.channels * mp.dies;
        if (mp.channels <= 128u && mp.dies <= 32u && cells <= kRetPlanCells) {      // (a lane holds four channels, a word the dies of one)
            const size_t smem = (size_t)(1 + kRetPlanWarps) * cells * sizeof(uint32_t);
            auto k = mp.channels <= 32u ? k_ret_plan<1> : mp.channels <= 64u ? k_ret_plan<2> : k_ret_plan<4>;
            e = ensure_dyn_smem((const void *)k, smem);
            // a warp has 32 rounds at least: no more of them than the longest epoch there can be fills
            const uint64_t rounds = r.plan_cap / mp.channels, blocks = (rounds + 32 * kRetPlanWarps - 1) / (32 * kRetPlanWarps);
            if (e == cudaSuccess)
                e = launch_pdl(k, (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(blocks, (uint64_t)sm_count * (smem > 50u * 1024u ? 2 : 4))), kRetPlanThreads, smem, st, r, mp.channels, mp.dies, mp.planes);
        } else {
            const uint32_t split = std::max<uint32_t>(1u, std::min<uint32_t>((uint32_t)(sm_count * 8) / mp.n_dies, (mp.planes * r.bpp + 7u) / 8u));   // eight blocks per multiprocessor where the dies are fewer
            e = launch_pdl(k_ret_emit, mp.n_dies * split, 256, 0, st, r, mp.channels, mp.dies, mp.planes, split);
        }
    }
    g_kernel_launches += 2;
    return e;
}

// =====================================================================================================
// idle time drains debt: one quantum per scaled quantum time (Eq. 3), on an account of its own
// =====================================================================================================
__global__ void k_ret_decay(RetDev r, const DevState *state, int64_t quantum_ns, int64_t idle_ns) {
    RetState *st = r.st;
    const int64_t q = state->q_ppm;
    const int64_t scaled = q == 1000000 ? quantum_ns : (quantum_ns * 1000000 + q - 1) / q;
    unsigned long long drained = (unsigned long long)(idle_ns / scaled);
    const unsigned long long debt = st->planned - st->claimed - st->decayed;
    st->decayed += min(drained, debt);
}

// the totals, and how many blocks wait for their refresh, counted here (every block's epoch on its way to the host took 139 us for
// 65,536 blocks, this 24)
__global__ void __launch_bounds__(256)
k_ret_totals(RetDev r, RetState *h_state, unsigned long long *h_waiting) {
    RetState *st = r.st;
    uint32_t c = 0;
    const uint64_t quads = r.n_blocks / 4, stride = (uint64_t)gridDim.x * 256;
    for (uint64_t q = (uint64_t)blockIdx.x * 256 + threadIdx.x; q < quads; q += stride) {
        const uint4 e = reinterpret_cast<const uint4 *>(r.epoch_of)[q];
        c += (e.x != 0u) + (e.y != 0u) + (e.z != 0u) + (e.w != 0u);
    }
    if (blockIdx.x == 0 && threadIdx.x < r.n_blocks % 4) c += r.epoch_of[quads * 4 + threadIdx.x] != 0u;
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane_id() == 0 && c) atomicAdd(&st->counted, (unsigned long long)c);
    __shared__ uint32_t s_last;
    __syncthreads();
    if (threadIdx.x == 0) { __threadfence(); s_last = atomicAdd(&st->epoch_blocks, 1ull) == gridDim.x - 1u ? 1u : 0u; }
    __syncthreads();
    if (!s_last || threadIdx.x != 0) return;
    __threadfence();
    *h_waiting = atomicExch(&st->counted, 0ull);             // (both counters are zero between launches)
    atomicExch(&st->epoch_blocks, 0ull);
    RetState now = *st;
    now.counted = 0ull; now.epoch_blocks = 0ull;
    *h_state = now;
}
cudaError_t launch_ret_totals(const RetDev &r, int sm_count, RetState *h_state, unsigned long long *h_waiting, cudaStream_t st) {
    k_ret_totals<<<ret_grid(r.n_blocks / 4 + 1, sm_count), 256, 0, st>>>(r, h_state, h_waiting);
    g_kernel_launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_ret_decay(const RetDev &r, const ModelParams &mp, const DevState *state, int64_t idle_ns, int sm_count, cudaStream_t st) {
    k_ret_decay<<<1, 1, 0, st>>>(r, state, mp.t_read_ns + mp.t_prog_ns, idle_ns);
    k_ret_commit<<<ret_grid(r.n_blocks, sm_count), 256, 0, st>>>(r);
    g_kernel_launches += 2;
    return cudaGetLastError();
}

}  // namespace hbf

// Small batches (at most kInSmallMax records) in one launch of one thread-block cluster, instead of tiles, a scan, a fix-up and a
// straggle pass whose fixed costs a few thousand records cannot pay for.  A block looks at a share of the records, and serves and
// commits a share of the queues (whole dies); queues do not interact, so nothing waits but for two cluster barriers and the totals at the end.
//   look    a thread per record: status, queue, service terms; counts per destination block, stable ranks.  The blocks
//           exchange their counts (barrier 1), so every block knows the whole batch's statuses, order and claims, takes the
//           same decision about it, and knows where its records go
//   send    every record becomes an entry in the list of the block that owns its queue, in batch order, through distributed
//           shared memory (barrier 2)
//   serve   a list in issue order: a warp takes a row of 32 entries, composes the maps of the lanes that hold the same queue, and the
//           queues' busy-until in shared memory are moved on row after row, handed from warp to warp through named barriers (as in
//           inorder_kernels.cu); results, ledger events, busy-until and per-die totals go out
//   sort    a list that is not in issue order is sorted by issue time, 8 bits a pass over the bits that differ, then by queue, stable, in
//           shared memory (a row of 32 ranks itself with match_any), and served by a segmented max-plus scan (a queue's run is a
//           segment): a thread composes the maps of its entries, the block scans the threads' maps, the thread walks its entries
//           again from the busy-until that reaches it.  (Lists in issue order went this way too: a window of 1 ms 23.3 us with its thermal step, now 20.2.)
//   close   the first block adds up the batch's totals and writes the summary: they are sent to its shared memory, and the others are done.  With the channel-bus stage on the
//           batch may still be refused once its largest completion is known: the blocks then stage what they commit, and the
//           first one commits it
// Bound by the latency of some thirty dependent steps.  Every block looking at all the records (no exchange) took 57,000 warp
// instructions per block, half of them classification: 18 us for 5,900 records.
#include <algorithm>
#include <mutex>
#include <vector>

#include <cooperative_groups.h>

#include "ledger.cuh"
#include "serve_terms.cuh"

namespace cg = cooperative_groups;

namespace hbf {

constexpr int kSmThreads = 512, kSmWarps = kSmThreads / 32;
constexpr int kSmCluster = 16, kSmPortable = 8;          // blocks: 16 where the device can place them (not a portable size), else 8
constexpr uint32_t kSmSlice = 256;                       // queues per block, at most: the bins of the sort
constexpr int kSmChain = 15;                               // warps that serve rows: a hardware barrier each
constexpr int kSmMaxRows = 32;                           // rows of 32 records a block looks at, at most
constexpr uint32_t kSmIdxBits = 13;
static_assert((1u << kSmIdxBits) == kInSmallMax && kInSmallMax / kSmPortable <= kSmMaxRows * 32, "index bits of an entry; rows of a block");

struct SmallArgs {
    const hbf_access_t *acc; uint32_t n, chunk, slice, forced, bus_on;    // chunk: records a block looks at (a multiple of 32)
    const RangeSnap *ranges; FastRange fast; ModelParams mp;
    DevState *state; BatchCtrl *ctrl; hbf_batch_result_t *result;
    int64_t *busy, *busy_stage, *pending; hbf_die_stats_t *stats_stage, *die_stats;
    int64_t *completion, *stall; uint8_t *status; uint32_t *order;
    unsigned long long *ledger; int64_t bin_ns, cur_bin; uint32_t n_bins, ret_on;     // ledger == null: energy to the pending totals
    RetDev ret;
};

static uint32_t small_padded(uint32_t n) { return (n + 255u) / 256u * 256u; }
static size_t small_smem(uint32_t n) { return (size_t)small_padded(n) * (8 + 8 + 4 + 2 + 2 + 1); }
static uint32_t small_slice(const ModelParams &mp, int blocks) {        // whole dies; 0: more queues than a block takes
    const uint32_t per_die = mp.queue_level == 0u ? mp.planes : 1u, slice = (mp.n_dies + blocks - 1) / blocks * per_die;
    return slice > kSmSlice ? 0u : slice;
}

// one stable pass over m places: src -> dst by digit(place) < bins <= 256
template <class Digit>
__device__ __forceinline__ void small_sort_pass(const uint16_t *src, uint16_t *dst, uint32_t m, uint32_t bins, uint16_t (*hist)[kSmSlice + 2], uint32_t *dbase,
                                                uint32_t *wsum, Digit digit) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rows = (m + 31u) / 32u, per_warp = (rows + kSmWarps - 1) / kSmWarps, first = warp * per_warp * 32u;
    for (uint32_t d = lane; d < bins; d += 32u) hist[warp][d] = 0;
    __syncwarp();
    for (uint32_t r = 0; r < per_warp; ++r) {                // counts per (warp, digit)
        const uint32_t at = first + r * 32u + lane;
        if (first + r * 32u >= m) break;
        const uint32_t d = at < m ? digit(src[at]) : 0xffffu;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        if (lane == __ffs(peers) - 1 && at < m) hist[warp][d] = (uint16_t)(hist[warp][d] + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    uint32_t total = 0, inc = 0;                             // a thread per digit: where every warp's keys of it begin, then where the digits begin
    if (tid < (int)kSmSlice) {
        if ((uint32_t)tid < bins) {
#pragma unroll
            for (int w = 0; w < kSmWarps; ++w) { const uint32_t c = hist[w][tid]; hist[w][tid] = (uint16_t)total; total += c; }
        }
        inc = total;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
        if (lane == 31) wsum[warp] = inc;
    }
    __syncthreads();
    if (tid < (int)kSmSlice) {
        uint32_t before = 0;
#pragma unroll
        for (int w = 0; w < (int)kSmSlice / 32; ++w) before += w < warp ? wsum[w] : 0u;
        if ((uint32_t)tid < bins) dbase[tid] = before + inc - total;
    }
    __syncthreads();
    for (uint32_t r = 0; r < per_warp; ++r) {
        const uint32_t at = first + r * 32u + lane;
        if (first + r * 32u >= m) break;
        const uint32_t p = at < m ? src[at] : 0u, d = at < m ? digit(p) : 0xffffu;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        uint32_t before = 0;
        if (at < m) { before = hist[warp][d]; dst[dbase[d] + before + __popc(peers & lanemask_lt())] = (uint16_t)p; }
        __syncwarp();
        if (lane == __ffs(peers) - 1 && at < m) hist[warp][d] = (uint16_t)(before + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
}

struct SmMap { int64_t S, M; int f; };                     // B -> max(B + S, M); f: holds the head of a run, so B no longer matters
__device__ __forceinline__ SmMap sm_then(const SmMap &x, const SmMap &y) {        // x first, then y
    SmMap r; r.S = y.f ? y.S : x.S + y.S; r.M = y.f ? y.M : max((int64_t)(x.M + y.S), y.M); r.f = x.f | y.f; return r;
}
__device__ __forceinline__ SmMap sm_shfl_up(const SmMap &v, int o) {
    SmMap u; u.S = __shfl_up_sync(0xffffffffu, v.S, o); u.M = __shfl_up_sync(0xffffffffu, v.M, o); u.f = __shfl_up_sync(0xffffffffu, v.f, o); return u;
}

__device__ __noinline__ Served small_terms_general(const RangeSnap &rs, const ModelParams &mp, uint64_t addr, int64_t issue, uint64_t bf, int64_t q_ppm, Div64 div_q) {
    unsigned ignored = 0;                                    // (services are 64 bits here)
    return serve_terms(rs, mp, addr, issue, bf, q_ppm, div_q, ignored, 63);
}

// R: records a thread looks at; EXTRA: with the ledger or retention
template <int R, bool EXTRA>
__global__ void __launch_bounds__(kSmThreads, 1)
k_small_serve(const __grid_constant__ SmallArgs a) {
    extern __shared__ __align__(16) unsigned char sm_small[];
    constexpr int kCols = kSmCluster + 1;                    // destinations, and the modeled accesses as a column of their own
    __shared__ uint32_t s_row[kSmMaxRows][kCols];            // per row of 32: entries per destination, then those before the row
    __shared__ uint32_t s_tab[kSmCluster][kSmCluster + 4];   // from every block: entries per destination; ready, native, failing, out of order
    __shared__ uint32_t s_base[kSmCluster];                  // where this block's entries begin in every destination's list
    __shared__ uint32_t s_total[kSmCluster];                 // entries of every destination's list
    __shared__ uint32_t s_all[6];                            // of the batch: (-), modeled before this block's records, modeled, native, failing, out of order
    __shared__ uint32_t s_flags[3];                          // this block: native, failing, out of order
    __shared__ unsigned long long s_lo, s_hi;                // smallest and largest issue time of the list (batches out of order)
    __shared__ int64_t s_busy[kSmSlice];
    __shared__ uint32_t s_nr[kSmSlice], s_np[kSmSlice], s_br[2][kSmSlice], s_bp[2][kSmSlice], s_work[2][kSmSlice];
    __shared__ uint32_t s_claims[EXTRA ? kSmSlice : 1];
    __shared__ uint16_t s_hist[kSmWarps][kSmSlice + 2];
    __shared__ uint32_t s_dbase[kSmSlice], s_wsum[kSmWarps];
    __shared__ int64_t w_S[kSmWarps], w_M[kSmWarps];
    __shared__ int w_f[kSmWarps];
    __shared__ long long w_stall[kSmWarps], w_max[kSmWarps];
    __shared__ long long s_tot[kSmCluster][3];               // (first block) every block's stalls, services, largest completion
    __shared__ Div64 s_div;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ __align__(8) uint64_t s_bar;                  // (first block) every block's totals have come
    const uint32_t rank = cluster.block_rank(), blocks = cluster.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&s_bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&s_bar)), "r"(blocks * 24u) : "memory");
    }
    cluster.barrier_arrive();                                // (waited for below: every block runs before one writes into another)
    const ModelParams &mp = a.mp;
    const RangeSnap &rs = *a.ranges;
    const uint32_t n = a.n, padded = (n + 255u) / 256u * 256u;
    const uint32_t q_lo = min(mp.n_queues, rank * a.slice), q_n = min(a.slice, mp.n_queues - q_lo);
    const uint32_t per_die = mp.queue_level == 0u ? mp.planes : 1u, d_lo = q_lo / per_die, d_n = q_n / per_die;
    int64_t *s_s = reinterpret_cast<int64_t *>(sm_small);                     // by place in the list: service time
    uint64_t *s_key = reinterpret_cast<uint64_t *>(s_s + padded);             //   issue time << 16 | program << 13 | batch index
    uint32_t *s_px = reinterpret_cast<uint32_t *>(s_key + padded);            //   transfer | claim << 31
    uint16_t *perm0 = reinterpret_cast<uint16_t *>(s_px + padded), *perm1 = perm0 + padded;
    uint8_t *s_lq = reinterpret_cast<uint8_t *>(perm1 + padded);              //   queue in the slice
    const uint64_t *rec0 = reinterpret_cast<const uint64_t *>(a.acc);
    const uint32_t begin = min(n, rank * a.chunk), end = min(n, begin + a.chunk);
    if (tid < (int)kSmSlice) {
        s_nr[tid] = s_np[tid] = s_br[0][tid] = s_br[1][tid] = s_bp[0][tid] = s_bp[1][tid] = s_work[0][tid] = s_work[1][tid] = 0u;
        if (EXTRA) s_claims[tid] = 0u;
    }
    for (int e = tid; e < kSmMaxRows * kCols; e += kSmThreads) (&s_row[0][0])[e] = 0u;
    if (tid < 3) s_flags[tid] = 0u;
    if (tid == 0) { s_lo = ~0ull; s_hi = 0ull; }
    // what the kernels before may still be writing is only called into the L2 here
    if (begin + (uint32_t)tid * 4u < end) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.acc + begin + tid * 4));
    __syncthreads();
    pdl_wait();                                              // everything above reads kernel arguments only
    pdl_trigger();

    // ---- look
    uint64_t addr[R], bf[R]; int64_t issue[R], prev[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint32_t i = begin + r * kSmThreads + tid;
        addr[r] = bf[r] = 0ull; issue[r] = 0; prev[r] = INT64_MIN;
        if (i < end) {
            const uint64_t *rec = rec0 + (size_t)i * 3;
            addr[r] = ld_after(rec); issue[r] = (int64_t)ld_after(rec + 1); bf[r] = ld_after(rec + 2);
            if (lane == 0 && i > 0u) prev[r] = (int64_t)ld_after(rec - 2);
        }
    }
    int code = HBF_OK;
    const int32_t mode = a.state->mode, poisoned = a.state->poisoned;
    const int64_t q_ppm = a.state->q_ppm;
    unsigned long long debt = 0ull;
    if (EXTRA && a.ret_on) debt = a.ret.st->planned - a.ret.st->claimed - a.ret.st->decayed;
    if ((uint32_t)tid < q_n) s_busy[tid] = a.busy[q_lo + tid];
    if (poisoned) code = HBF_E_TIMEOUT;
    else if (mode == HBF_MODE_SHUTDOWN) code = HBF_E_LINK_SHUTDOWN;
    else if (mode == HBF_MODE_SEVERE) code = HBF_E_THROTTLED;
    if (q_ppm != 1000000) {                                  // (a 128-bit division: one thread makes it)
        if (tid == 0) s_div = make_div64((uint64_t)q_ppm);
        __syncthreads();
    }
    const Div64 div_q = s_div;                               // (not looked at without thermal scaling)
    const bool fast = a.fast.on != 0u && mp.pow2_geom != 0u && mp.xfer_tab_max_cb != 0u && q_ppm == 1000000;
    const int64_t quantum_ns = !EXTRA ? 0 : q_ppm == 1000000 ? mp.t_read_ns + mp.t_prog_ns
        : (int64_t)div64((uint64_t)(mp.t_read_ns + mp.t_prog_ns) * 1000000ull + (uint64_t)q_ppm - 1ull, div_q);
    uint32_t m = 0, n_ready = 0, n_native = 0, n_fault = 0;
    bool unsorted = false;
    unsigned long long claims = 0ull;
    long long sum_stall = 0, max_c = INT64_MIN;
    cluster.barrier_wait();
    if (code == HBF_OK) {                                    // (the same for every block)
        Served v[R];
        uint32_t dest[R], at[R], rr[R];                      // destination; rank among its entries of the row; rank among the row's modeled accesses
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t i = begin + r * kSmThreads + tid;
            const bool have = i < end;
            int64_t before = __shfl_up_sync(0xffffffffu, issue[r], 1);
            if (lane == 0) before = prev[r];
            v[r].st = -1;
            if (have) v[r] = fast ? serve_terms_fast<false>(a.fast, mp, addr[r], issue[r], bf[r]) : small_terms_general(rs, mp, addr[r], issue[r], bf[r], q_ppm, div_q);
            if (have && a.status) a.status[i] = (uint8_t)v[r].st;
            const bool ready = v[r].st == HBF_ST_READY;
            dest[r] = ready ? v[r].queue / a.slice : 0xffffu;
            const unsigned peers = __match_any_sync(0xffffffffu, dest[r]), br = __ballot_sync(0xffffffffu, ready);
            at[r] = (uint32_t)__popc(peers & lanemask_lt()); rr[r] = (uint32_t)__popc(br & lanemask_lt());
            const uint32_t row = r * kSmWarps + warp;
            if (ready && at[r] == 0u) s_row[row][dest[r]] = (uint32_t)__popc(peers);
            const unsigned bn = __ballot_sync(0xffffffffu, v[r].st == HBF_ST_NATIVE), bv = __ballot_sync(0xffffffffu, have);
            const bool uns = __any_sync(0xffffffffu, have && issue[r] < before);
            if (lane == 0) {
                s_row[row][kSmCluster] = (uint32_t)__popc(br);
                if (bn) atomicAdd(&s_flags[0], (uint32_t)__popc(bn));
                const uint32_t bad = (uint32_t)__popc(bv) - (uint32_t)__popc(br) - (uint32_t)__popc(bn);     // every other status is a fault
                if (bad) atomicAdd(&s_flags[1], bad);
                if (uns) s_flags[2] = 1u;
            }
        }
        __syncthreads();
        for (int col = warp; col < kCols; col += kSmWarps) { // a warp per column, a lane per row: the entries before every row; the total goes to every block
            const uint32_t c = s_row[lane][col];
            uint32_t inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
            s_row[lane][col] = inc - c;
            const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
            if ((uint32_t)lane < blocks) {
                uint32_t *t = cluster.map_shared_rank(&s_tab[0][0], lane) + rank * (kSmCluster + 4);
                t[col] = total;
                if (col == kSmCluster) { t[kSmCluster + 1] = s_flags[0]; t[kSmCluster + 2] = s_flags[1]; t[kSmCluster + 3] = s_flags[2]; }
            }
        }
        cluster.sync();
        for (int col = warp; col < kSmCluster + 4; col += kSmWarps) {        // a warp per column, lane = the block the counts come from
            const uint32_t c = (uint32_t)lane < blocks ? s_tab[lane][col] : 0u;
            uint32_t inc = c;
#pragma unroll
            for (int o = 1; o < kSmCluster; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
            const uint32_t all = __shfl_sync(0xffffffffu, inc, kSmCluster - 1), before = __shfl_sync(0xffffffffu, inc - c, (int)rank);
            if (lane == 0) {
                if (col < kSmCluster) { s_base[col] = before; s_total[col] = all; }
                else if (col == kSmCluster) { s_all[1] = before; s_all[2] = all; }
                else s_all[2 + col - kSmCluster] = all;      // native, failing, blocks that saw records out of order
            }
        }
        __syncthreads();
        m = s_total[rank]; n_ready = s_all[2]; n_native = s_all[3]; n_fault = s_all[4]; unsorted = s_all[5] != 0u;
        if (n_fault) code = HBF_E_ACCESS_FAULT;              // fail closed: refuse the batch
        else if (unsorted && a.forced) code = HBF_E_INVAL;
        if (code == HBF_OK) {
            // ---- send
            claims = min(debt, (unsigned long long)n_ready);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const uint32_t i = begin + r * kSmThreads + tid, row = r * kSmWarps + warp;
                if (v[r].st == HBF_ST_READY) {
                    const uint32_t among = s_all[1] + s_row[row][kSmCluster] + rr[r];            // place among the batch's modeled accesses
                    const bool claim = EXTRA && among < claims;
                    const uint32_t p = s_base[dest[r]] + s_row[row][dest[r]] + at[r];
                    cluster.map_shared_rank(s_s, dest[r])[p] = v[r].s + (claim ? quantum_ns : 0);
                    cluster.map_shared_rank(s_key, dest[r])[p] = ((uint64_t)issue[r] << 16) | (v[r].op << kSmIdxBits) | i;
                    cluster.map_shared_rank(s_px, dest[r])[p] = v[r].xfer | (claim ? 0x80000000u : 0u);
                    cluster.map_shared_rank(s_lq, dest[r])[p] = (uint8_t)(v[r].queue - dest[r] * a.slice);
                    if (EXTRA && a.bus_on && claim && among + 1u == claims) { a.ret.st->claim_limit = claims == debt ? i + 1u : n; a.ret.st->claims_now = claims; }
                    if (EXTRA && a.ret_on && !a.bus_on && !v[r].op) {    // read disturb: the read's pages, on the block of its first page
                        uint64_t off;
                        if (a.fast.on) off = a.fast.media_offset + (addr[r] - a.fast.base);
                        else { int g = 0; classify(rs, addr[r], issue[r], (uint32_t)bf[r], 0u, &g); off = rs.media_offset[g] + (addr[r] - rs.base[g]); }
                        const uint64_t page = 1ull << mp.page_shift;
                        atomicAdd(&a.ret.disturb[ret_block_of(mp, a.ret, off)], (uint32_t)(((off & (page - 1ull)) + (uint32_t)bf[r] + page - 1ull) >> mp.page_shift));
                    }
                } else if (v[r].st == HBF_ST_NATIVE) {
                    a.completion[i] = issue[r]; a.stall[i] = 0;
                }
            }
            cluster.sync();
        }
    }
    if (code == HBF_OK) {
        // (the sizes come from the records again; they are needed once the list is served)
        uint64_t bf0 = 0ull;
        if ((uint32_t)tid < m) bf0 = ld_after(rec0 + (size_t)((uint32_t)s_key[tid] & (kInSmallMax - 1u)) * 3 + 2);
        const Ledger book = EXTRA && a.ledger ? make_ledger(a.ledger, mp.n_dies, a.n_bins, a.cur_bin, a.bin_ns) : Ledger{};
        auto ledger_of = [&](uint32_t lq, uint32_t i, uint32_t op, bool claim, int64_t s, int64_t end) {        // the access's events
            const int64_t own = s - (claim ? quantum_ns : 0), page = (int64_t)1 << mp.page_shift;
            const uint64_t gm = (1ull << (op ? mp.prog_gran_shift : mp.read_gran_shift)) - 1ull, cb = ((uint64_t)(uint32_t)ld_after(rec0 + (size_t)i * 3 + 2) + gm) & ~gm;
            const uint32_t die = d_lo + lq / per_die;
            const int64_t pj = op ? mp.e_cmd_prog_pj + mp.e_byte_prog_pj * (int64_t)cb : mp.e_cmd_read_pj + mp.e_byte_read_pj * (int64_t)cb;
            if (claim) ledger_event(book, die, end - s, quantum_ns,
                                    mp.e_cmd_read_pj + mp.e_byte_read_pj * page + mp.e_cmd_prog_pj + mp.e_byte_prog_pj * page);
            ledger_event(book, die, end - own, own, pj);
        };
        if (!unsorted) {
            // ---- serve, row after row
            const uint32_t rows = (m + 31u) / 32u;
            if (warp < kSmChain) {
                for (uint32_t r = (uint32_t)warp; r < rows; r += kSmChain) {
                    const uint32_t p = r * 32u + lane;
                    const bool have = p < m;
                    const uint64_t key = have ? s_key[p] : 0ull;
                    const int64_t s = have ? s_s[p] : 0;
                    const uint32_t lq = have ? s_lq[p] : 0u, px = have ? s_px[p] : 0u, i = (uint32_t)key & (kInSmallMax - 1u), op = (uint32_t)(key >> kSmIdxBits) & 1u;
                    const int64_t t = (int64_t)(key >> 16), x = (int64_t)(px & 0x7fffffffu);
                    const unsigned peers = __match_any_sync(0xffffffffu, have ? lq : 0x100u + lane), le = peers & (lanemask_lt() | (1u << lane));
                    int64_t S = s, M = t + (op ? x : 0) + s;                    // of the lanes of this queue up to this one, by doubling
                    const unsigned before = le & ~(1u << lane);
                    int prev_l = before ? 31 - __clz((int)before) : -1;
                    const uint32_t most = __reduce_max_sync(0xffffffffu, (uint32_t)__popc(le));
                    for (uint32_t span = 1; span < most; span <<= 1) {
                        const int src = prev_l >= 0 ? prev_l : lane;
                        const int64_t Se = __shfl_sync(0xffffffffu, S, src), Me = __shfl_sync(0xffffffffu, M, src);
                        const int pe = __shfl_sync(0xffffffffu, prev_l, src);
                        if (prev_l >= 0) { M = max(Me + S, M); S += Se; prev_l = pe; }
                    }
                    const bool last = have && (peers >> lane) == 1u;
                    if (r > 0u) asm volatile("barrier.cta.sync.aligned %0, 64;" ::"r"(1 + warp), "l"(S), "l"(M), "r"(lq), "r"((int)last) : "memory");
                    const int64_t B = max(s_busy[lq] + S, M);
                    if (last) s_busy[lq] = B;
                    __syncwarp();
                    if (r + 1u < rows) asm volatile("barrier.cta.arrive.aligned %0, 64;" ::"r"(1 + (warp + 1) % kSmChain) : "memory");
                    if (have) {
                        const int64_t c = B + (op ? 0 : x), waited = c - t;
                        a.completion[i] = c; a.stall[i] = waited;
                        sum_stall += waited; max_c = max(max_c, (long long)c);
                        if (EXTRA && a.ledger && !a.bus_on) ledger_of(lq, i, op, (px >> 31) != 0u, s, B);
                    }
                }
                sum_stall = warp_sum(sum_stall); max_c = warp_max(max_c);
            }
        } else {
        // ---- sort
        if (a.bus_on && (uint32_t)tid < q_n) a.busy_stage[q_lo + tid] = s_busy[tid];      // (of queues without an access)
        for (uint32_t p = (uint32_t)tid; p < m; p += kSmThreads) perm0[p] = (uint16_t)p;
        {
            unsigned long long lo = ~0ull, hi = 0ull;
            for (uint32_t p = (uint32_t)tid; p < m; p += kSmThreads) { const unsigned long long t = s_key[p] >> 16; lo = min(lo, t); hi = max(hi, t); }
            for (int o = 16; o > 0; o >>= 1) { lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
            if (lane == 0 && lo <= hi) { atomicMin(&s_lo, lo); atomicMax(&s_hi, hi); }
        }
        __syncthreads();
        uint16_t *src = perm0, *dst = perm1;
        if (m > 1u) {
            const unsigned long long first = s_lo, span = s_hi - first;
            for (uint32_t sh = 0; sh < 48u && (span >> sh) != 0ull; sh += 8u) {
                small_sort_pass(src, dst, m, 256u, s_hist, s_dbase, s_wsum, [&](uint32_t p) { return (uint32_t)(((s_key[p] >> 16) - first) >> sh) & 255u; });
                uint16_t *t = src; src = dst; dst = t;
            }
        }
        small_sort_pass(src, dst, m, a.slice, s_hist, s_dbase, s_wsum, [&](uint32_t p) { return (uint32_t)s_lq[p]; });
        const uint16_t *sorted = dst;
        uint32_t below = 0;                                  // entries of the lists before this one (for hbf_queue_order)
        for (uint32_t d = 0; d < rank; ++d) below += s_total[d];
        // ---- serve
        const uint32_t per = (m + kSmThreads - 1u) / kSmThreads, p0 = (uint32_t)tid * per, p1 = min(m, p0 + per);   // this thread's entries
        const uint32_t prev_q = p0 > 0u && p0 < m ? s_lq[sorted[p0 - 1u]] : 0xffffffffu;
        SmMap agg; agg.S = 0; agg.M = kNegInf; agg.f = 0;
        {
            uint32_t pq = prev_q;
            for (uint32_t p = p0; p < p1; ++p) {
                const uint32_t e = sorted[p], lq = s_lq[e], px = s_px[e];
                const uint64_t key = s_key[e];
                const int64_t s = s_s[e], t = (int64_t)(key >> 16) + ((key >> kSmIdxBits) & 1u ? (int64_t)(px & 0x7fffffffu) : 0);
                SmMap x; x.S = s; x.f = lq != pq; x.M = (x.f ? max(t, s_busy[lq]) : t) + s;
                agg = sm_then(agg, x);
                pq = lq;
            }
        }
        SmMap inc = agg;
        if (warp * 32u * per < m) {                          // (warps without entries hold identities)
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const SmMap u = sm_shfl_up(inc, o); if (lane >= o) inc = sm_then(u, inc); }
        }
        if (lane == 31) { w_S[warp] = inc.S; w_M[warp] = inc.M; w_f[warp] = inc.f; }
        __syncthreads();
        if (warp * 32u * per < m) {
            SmMap ex; ex.S = 0; ex.M = kNegInf; ex.f = 0;     // everything before this thread's entries
            if (warp > 0) {                                   // every warp scans the warps' maps for itself
                SmMap wm; wm.S = w_S[lane & (kSmWarps - 1)]; wm.M = w_M[lane & (kSmWarps - 1)]; wm.f = w_f[lane & (kSmWarps - 1)];
#pragma unroll
                for (int o = 1; o < kSmWarps; o <<= 1) { const SmMap u = sm_shfl_up(wm, o); if (lane >= o) wm = sm_then(u, wm); }
                ex.S = __shfl_sync(0xffffffffu, wm.S, warp - 1); ex.M = __shfl_sync(0xffffffffu, wm.M, warp - 1); ex.f = __shfl_sync(0xffffffffu, wm.f, warp - 1);
            }
            const SmMap u = sm_shfl_up(inc, 1);
            if (lane > 0) ex = sm_then(ex, u);
            // (the first entry of the list is a head, so a map without a head never reaches an entry that needs its input)
            int64_t B = ex.M;
            uint32_t pq = prev_q;
            for (uint32_t p = p0; p < p1; ++p) {
                const uint32_t e = sorted[p], lq = s_lq[e], px = s_px[e], i = (uint32_t)s_key[e] & (kInSmallMax - 1u), op = (uint32_t)(s_key[e] >> kSmIdxBits) & 1u;
                const int64_t t = (int64_t)(s_key[e] >> 16), s = s_s[e], x = (int64_t)(px & 0x7fffffffu);
                if (lq != pq) B = s_busy[lq];
                B = max(t + (op ? x : 0), B) + s;
                const int64_t c = B + (op ? 0 : x), waited = c - t;
                a.completion[i] = c; a.stall[i] = waited;
                sum_stall += waited; max_c = max(max_c, (long long)c);
                if (p + 1u == m || s_lq[sorted[p + 1u]] != lq)   // last access of its queue in this batch
                    (a.bus_on ? a.busy_stage : a.busy)[q_lo + lq] = B;
                a.order[below + p] = i;
                if (EXTRA && a.ledger && !a.bus_on) ledger_of(lq, i, op, (px >> 31) != 0u, s, B);
                pq = lq;
            }
            sum_stall = warp_sum(sum_stall); max_c = warp_max(max_c);
        }
        }
        if (lane == 0) { w_stall[warp] = sum_stall; w_max[warp] = max_c; }
        // ---- per-die totals (32-bit adds with a carry: a 64-bit one in shared memory is a loop)
        for (uint32_t p = (uint32_t)tid; p < m; p += kSmThreads) {
            const uint64_t key = s_key[p], bfp = p < (uint32_t)kSmThreads ? bf0 : ld_after(rec0 + (size_t)((uint32_t)key & (kInSmallMax - 1u)) * 3 + 2);
            const uint32_t op = (uint32_t)(key >> kSmIdxBits) & 1u, ld = s_lq[p] / per_die;
            const uint64_t gm = (1ull << (op ? mp.prog_gran_shift : mp.read_gran_shift)) - 1ull, cb = ((uint64_t)(uint32_t)bfp + gm) & ~gm, s = (uint64_t)s_s[p];
            auto add = [](uint32_t *lo, uint32_t *hi, uint64_t x) {
                const uint32_t l = (uint32_t)x, old = atomicAdd(lo, l), c = (uint32_t)(x >> 32) + (old + l < old ? 1u : 0u);
                if (c) atomicAdd(hi, c);
            };
            atomicAdd(op ? &s_np[ld] : &s_nr[ld], 1u);
            add(op ? &s_bp[0][ld] : &s_br[0][ld], op ? &s_bp[1][ld] : &s_br[1][ld], cb);
            add(&s_work[0][ld], &s_work[1][ld], s);
            if (EXTRA && (s_px[p] >> 31)) atomicAdd(&s_claims[ld], 1u);
        }
        __syncthreads();
        if (!unsorted && (uint32_t)tid < q_n) (a.bus_on ? a.busy_stage : a.busy)[q_lo + tid] = s_busy[tid];
        const int64_t page = (int64_t)1 << mp.page_shift;
        const int64_t quantum_pj = mp.e_cmd_read_pj + mp.e_byte_read_pj * page + mp.e_cmd_prog_pj + mp.e_byte_prog_pj * page;
        if ((uint32_t)tid < d_n) {
            hbf_die_stats_t ds;
            ds.busy_ns = (int64_t)(((uint64_t)s_work[1][tid] << 32) | s_work[0][tid]);
            ds.bytes_read = (int64_t)(((uint64_t)s_br[1][tid] << 32) | s_br[0][tid]); ds.bytes_prog = (int64_t)(((uint64_t)s_bp[1][tid] << 32) | s_bp[0][tid]);
            ds.n_read = s_nr[tid]; ds.n_prog = s_np[tid];
            ds.energy_pj = mp.e_cmd_read_pj * ds.n_read + mp.e_byte_read_pj * ds.bytes_read + mp.e_cmd_prog_pj * ds.n_prog + mp.e_byte_prog_pj * ds.bytes_prog;
            const uint32_t d = d_lo + tid;
            if (a.bus_on) {
                a.stats_stage[d] = ds;
                if (EXTRA && a.ret_on) a.ret.die_claims[d] = s_claims[tid];
            } else {
                if (a.die_stats) a.die_stats[d] = ds;
                const int64_t pj = ds.energy_pj + (EXTRA ? (int64_t)s_claims[tid] * quantum_pj : 0);
                if (!a.ledger && pj) atomicAdd(reinterpret_cast<unsigned long long *>(a.pending + d), (unsigned long long)pj);   // (no wait for the old value)
            }
        }
        if (EXTRA && a.ret_on && !a.bus_on && claims) {      // blocks whose last quantum is now claimed commit one cycle
            const unsigned long long mark = a.ret.st->planned - debt + claims;
            for (uint64_t b = ((uint64_t)rank * kSmThreads + tid) * 4u; b < a.ret.n_blocks; b += (uint64_t)blocks * kSmThreads * 4u) {
                uint32_t e[4] = {0u, 0u, 0u, 0u};            // (four at a time: most blocks wait for nothing)
                if (b + 4u <= a.ret.n_blocks) *reinterpret_cast<uint4 *>(e) = *reinterpret_cast<const uint4 *>(a.ret.epoch_of + b);
                else for (uint32_t k = 0; b + k < a.ret.n_blocks; ++k) e[k] = a.ret.epoch_of[b + k];
#pragma unroll
                for (uint32_t k = 0; k < 4u; ++k) if (e[k] != 0u && a.ret.last_pos[b + k] < mark) ret_commit_block(a.ret, b + k);
            }
        }
        if (warp == kSmWarps - 1) {
            const long long stall = warp_sum(lane < kSmWarps ? w_stall[lane] : 0), latest = warp_max(lane < kSmWarps ? w_max[lane] : INT64_MIN);
            long long work = 0;
            for (uint32_t d = (uint32_t)lane; d < d_n; d += 32u) work += (long long)(((uint64_t)s_work[1][d] << 32) | s_work[0][d]);
            work = warp_sum(work);
            if (lane < 3) {
                const long long v = lane == 0 ? stall : lane == 1 ? work : latest;
                if (a.bus_on) cluster.map_shared_rank(&s_tot[0][0], 0)[rank * 3u + lane] = v;        // (the barrier below comes behind it)
                else smem_send(smem_remote(smem_addr(&s_tot[rank][lane]), 0u), v, smem_remote(smem_addr(&s_bar), 0u));
            }
        }
    } else if (code != HBF_E_LINK_SHUTDOWN && code != HBF_E_THROTTLED) {              // refused: zeroed outputs, nothing changed
        for (uint32_t i = begin + tid; i < end; i += kSmThreads) { a.completion[i] = 0; a.stall[i] = 0; }
        if (a.die_stats) for (uint32_t e = (uint32_t)tid; e < d_n * 6u; e += kSmThreads) reinterpret_cast<int64_t *>(a.die_stats + d_lo)[e] = 0;
    }
    // ---- close: the others have sent their totals and are done (with the bus on the first one has to see what they staged).  The batch is
    // committed by now, so this is no wait to give up: should its polls run out, the cluster's barrier holds this warp until every other
    // thread of the cluster has ended, and all has been sent by then.  (The barrier in place of the polls: 48 windows 881 -> 907 us, and
    // 926 where the blocks also wait for one another at their ends.)
    if (a.bus_on) cluster.sync();
    if (rank != 0u || (!a.bus_on && warp != 0)) return;
    long long modeled = 0, service = 0, latest = 0;
    if (code == HBF_OK) {
        uint32_t polls = 0;
        bool late = false;
        if (!a.bus_on)
            while (!smem_poll(smem_addr(&s_bar), 0u)) if (++polls > a.state->spin_limit) { late = true; break; }
        if (__any_sync(0xffffffffu, late)) {
            asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
            for (polls = 0; polls <= kClusterPolls && !smem_poll(smem_addr(&s_bar), 0u); ) ++polls;
            if (polls > kClusterPolls) { a.state->poisoned = 1; code = HBF_E_TIMEOUT; }
        }
        const bool from = (uint32_t)lane < blocks;
        modeled = warp_sum(from ? s_tot[lane][0] : 0); service = warp_sum(from ? s_tot[lane][1] : 0); latest = warp_max(from ? s_tot[lane][2] : 0);
    }
    if (a.bus_on) {                                          // commit what the blocks staged, or refuse (array-done times are sort keys of 47 bits)
        if (code == HBF_OK && n_ready && latest >= HBF_ISSUE_LIMIT) {
            code = HBF_E_INVAL;
            for (uint32_t i = (uint32_t)tid; i < n; i += kSmThreads) { a.completion[i] = 0; a.stall[i] = 0; }
            if (a.die_stats) for (uint32_t e = (uint32_t)tid; e < mp.n_dies * 6u; e += kSmThreads) reinterpret_cast<int64_t *>(a.die_stats)[e] = 0;
        } else if (code == HBF_OK) {
            for (uint32_t q = (uint32_t)tid; q < mp.n_queues; q += kSmThreads) a.busy[q] = __ldcg(a.busy_stage + q);
            for (uint32_t d = (uint32_t)tid; d < mp.n_dies; d += kSmThreads) {
                hbf_die_stats_t ds;
                int64_t *w = reinterpret_cast<int64_t *>(&ds);
#pragma unroll
                for (int k = 0; k < 6; ++k) w[k] = __ldcg(reinterpret_cast<const int64_t *>(a.stats_stage + d) + k);
                if (!a.ledger) a.pending[d] += ds.energy_pj;
                if (a.die_stats) a.die_stats[d] = ds;
            }
        }
    }
    if (tid == 0) {
        hbf_batch_result_t r;
        const bool ok = code == HBF_OK, seen = ok || code == HBF_E_ACCESS_FAULT;
        r.code = code; r.mode = mode; r.q_ppm = q_ppm;
        r.n_native = seen ? n_native : 0u; r.n_modeled = ok ? n_ready : 0u; r.n_fault = n_fault;
        r.modeled_ns = ok ? modeled : 0; r.service_ns = ok ? service : 0; r.max_completion_ns = ok && n_ready ? latest : 0;
        *a.result = r;                                       // (not to the host as well: the kernel would end a microsecond later)
        BatchCtrl *c = a.ctrl;                               // what later stages and hbf_queue_order read of a batch
        c->code = code; c->skip = ok ? 0 : 1; c->mode = mode; c->q_ppm = q_ppm; c->div_q = div_q;
        c->n_ready = n_ready; c->inorder_used = ok && !unsorted ? 1u : 0u; c->run_sort = 0u; c->regrouped = 0u; c->plan.n_passes = 1u;
        if (EXTRA && a.ret_on && !a.bus_on && ok && claims) atomicAdd(&a.ret.st->claimed, claims);      // (nothing waits for it)
    }
}

using SmallKernel = void (*)(const SmallArgs);
static SmallKernel small_kernel(int blocks, uint32_t n, bool extra) {
    const bool two = (n + blocks - 1) / blocks > (uint32_t)kSmThreads;
    return two ? (extra ? k_small_serve<2, true> : k_small_serve<2, false>) : (extra ? k_small_serve<1, true> : k_small_serve<1, false>);
}

// how many blocks the cluster gets on the current device: 16 where it can place such a cluster (allowed per kernel), else 8;
// asked once per device and remembered.  0: not even that.
static int small_blocks() {
    struct Entry { int device, blocks; };
    static std::mutex mu;
    static std::vector<Entry> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lock(mu);
    for (const Entry &e : known) if (e.device == dev) return e.blocks;
    auto places = [&](SmallKernel k, int blocks) {
        const void *fn = (const void *)k;
        if (ensure_dyn_smem(fn, small_smem(kInSmallMax)) != cudaSuccess) return false;
        if (blocks > kSmPortable && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(blocks); cfg.blockDim = dim3(kSmThreads); cfg.dynamicSmemBytes = small_smem(kInSmallMax);
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension; at[0].val.clusterDim.x = blocks; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
        int count = 0;
        return cudaOccupancyMaxActiveClusters(&count, fn, &cfg) == cudaSuccess && count >= 1;
    };
    int blocks = 0;
    if (places(k_small_serve<1, false>, kSmCluster) && places(k_small_serve<1, true>, kSmCluster)) blocks = kSmCluster;
    else if (places(k_small_serve<1, false>, kSmPortable) && places(k_small_serve<1, true>, kSmPortable) &&
             places(k_small_serve<2, false>, kSmPortable) && places(k_small_serve<2, true>, kSmPortable)) blocks = kSmPortable;
    (void)cudaGetLastError();                                // a refusal here only means the tiled route is used
    known.push_back(Entry{dev, blocks});
    return blocks;
}

// whether a batch takes this route (launch_small serves it whole)
bool small_route(const SubmitArgs &a) {
    if (a.n == 0 || a.n > kInSmallMax || !a.inorder_ok || a.paged || (a.path != HBF_PATH_AUTO && a.path != HBF_PATH_INORDER)) return false;
    const int blocks = small_blocks();
    return blocks != 0 && small_slice(a.mp, blocks) != 0u;
}

cudaError_t launch_small(const SubmitArgs &a, const SmallExtras &x, cudaStream_t st) {
    const int blocks = small_blocks();
    SmallArgs s{};
    s.acc = a.acc; s.n = (uint32_t)a.n; s.chunk = ((s.n + blocks - 1) / blocks + 31u) / 32u * 32u;
    s.slice = small_slice(a.mp, blocks); s.forced = a.path == HBF_PATH_INORDER ? 1u : 0u; s.bus_on = a.bus_on ? 1u : 0u;
    s.ranges = a.ranges; s.fast = a.fast; s.mp = a.mp; s.state = a.state; s.ctrl = a.ctrl; s.result = a.result;
    s.busy = a.busy; s.busy_stage = a.busy_stage; s.pending = a.pending; s.stats_stage = a.stats_stage; s.die_stats = a.die_stats;
    s.completion = a.completion; s.stall = a.stall; s.status = a.status; s.order = a.ws.idx[1];
    s.ledger = x.ledger; s.bin_ns = x.bin_ns; s.cur_bin = x.cur_bin; s.n_bins = x.n_bins; s.ret_on = a.ret ? 1u : 0u;
    if (a.ret) s.ret = *a.ret;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks); cfg.blockDim = dim3(kSmThreads); cfg.dynamicSmemBytes = small_smem(s.n); cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension; at[0].val.clusterDim.x = blocks; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization; at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = a.plain_next && *a.plain_next ? 1 : 2;      // (see launch_first)
    g_kernel_launches += 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, small_kernel(blocks, s.n, s.ledger || s.ret_on), s);
    if (e == cudaSuccess && a.plain_next) *a.plain_next = false;
    return e;
}

}  // namespace hbf

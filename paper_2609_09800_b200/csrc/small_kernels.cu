// Small batches (at most kInSmallMax records) in one launch, instead of tiles, a scan, a fix-up and a straggle pass whose fixed
// costs a few thousand records cannot pay for.  Queues do not interact, so they are dealt to the blocks in slices of whole
// dies (64 queues, or the dies that fit), and a block serves and commits its slice on its own; no block waits for another.
// Every block looks at ALL the records (a few hundred KB, from the L2 after the first block), so every block knows the whole
// batch's statuses, order and claims and takes the same decision about it:
//   look    status and queue of records i, i + 1024, ...; counts per row of 32; the slice's records are listed in batch order
//           (a block's tenth part of a batch of a few thousand accesses: what follows works on that list only)
//   terms   one listed record per thread: service, transfer, arrival, per-die bytes and counts, read disturb
//   sort    by queue, stable, in shared memory (a row of 32 ranks itself with match_any); a batch that is not in issue order
//           is sorted by issue time first, 6 bits a pass over the bits that differ
//   serve   a segmented max-plus scan over the sorted list (a queue's run is a segment): a thread composes the maps of its
//           entries, the block scans the threads' maps, the thread walks its entries again from the busy-until that reaches
//           it; results, ledger events, busy-until and per-die totals go out
// The block that finishes last adds up the batch's totals and writes the summary.  With the channel-bus stage on the batch may
// still be refused once its largest completion is known: the blocks then stage what they commit, and the last one commits it.
// Bound by latency: 16 blocks of a 1,024-queue device, about 25 dependent steps.
#include <algorithm>

#include "ledger.cuh"
#include "serve_terms.cuh"

namespace hbf {

constexpr int kSmThreads = 1024, kSmWarps = kSmThreads / 32;
constexpr uint32_t kSmSlice = 64;                        // queues per block, at most: the bins of the sort
constexpr uint32_t kSmRounds = kInSmallMax / kSmThreads;
constexpr uint32_t kSmIdxBits = 13;
static_assert((1u << kSmIdxBits) == kInSmallMax && kSmWarps == 32 && kSmRounds == 8, "index bits of an entry; a lane per warp, eight counts per lane in the scans");

struct SmallArgs {
    const hbf_access_t *acc; uint32_t n, slice, forced, bus_on;
    const RangeSnap *ranges; FastRange fast; ModelParams mp;
    DevState *state; BatchCtrl *ctrl; SmallTotals *tot; hbf_batch_result_t *result;
    int64_t *busy, *busy_stage, *pending; hbf_die_stats_t *stats_stage, *die_stats;
    int64_t *completion, *stall; uint8_t *status; uint32_t *order;
    unsigned long long *ledger; int64_t bin_ns, cur_bin; uint32_t n_bins, ret_on;     // ledger == null: energy to the pending totals
    RetDev ret;
};

size_t small_smem(uint32_t n) {
    const size_t padded = (n + kSmThreads - 1) / kSmThreads * kSmThreads;
    return padded * (8 + 8 + 4 + 2 + 2 + 1);
}
uint32_t small_slice(const ModelParams &mp) {            // whole dies; 0: a die has more queues than a block takes
    const uint32_t per_die = mp.queue_level == 0u ? mp.planes : 1u;
    return per_die > kSmSlice ? 0u : kSmSlice / per_die * per_die;
}

// one stable pass over m places: src -> dst by digit(place) < 64
template <class Digit>
__device__ __forceinline__ void small_sort_pass(const uint16_t *src, uint16_t *dst, uint32_t m, uint32_t (*hist)[kSmSlice + 1], uint32_t *dtot, Digit digit) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rows = (m + 31u) / 32u, per_warp = (rows + kSmWarps - 1) / kSmWarps, first = warp * per_warp * 32u;
    hist[warp][lane] = 0u; hist[warp][lane + 32] = 0u;
    __syncwarp();
    for (uint32_t r = 0; r < per_warp; ++r) {                // counts per (warp, digit)
        const uint32_t at = first + r * 32u + lane;
        if (first + r * 32u >= m) break;
        const uint32_t d = at < m ? digit(src[at]) : kSmSlice;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        if (lane == __ffs(peers) - 1 && d < kSmSlice) hist[warp][d] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 2; ++k) {                            // a lane per warp: where every warp's keys of a digit begin
        const uint32_t d = warp * 2 + k, v = hist[lane][d];
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
        hist[lane][d] = inc - v;
        if (lane == 31) dtot[d] = inc;
    }
    __syncthreads();
    const uint32_t t0 = dtot[2 * lane], t1 = dtot[2 * lane + 1];       // every warp scans the 64 totals for itself
    uint32_t inc = t0 + t1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
    const uint32_t b0 = inc - (t0 + t1), b1 = b0 + t0;
    for (uint32_t r = 0; r < per_warp; ++r) {
        const uint32_t at = first + r * 32u + lane;
        if (first + r * 32u >= m) break;
        const uint32_t p = at < m ? src[at] : 0u, d = at < m ? digit(p) : kSmSlice;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t rank = __popc(peers & lanemask_lt());
        const uint32_t e0 = __shfl_sync(0xffffffffu, b0, (int)(d >> 1) & 31), e1 = __shfl_sync(0xffffffffu, b1, (int)(d >> 1) & 31);
        uint32_t before = 0;
        if (d < kSmSlice) { before = hist[warp][d]; dst[((d & 1u) ? e1 : e0) + before + rank] = (uint16_t)p; }
        __syncwarp();
        if (lane == __ffs(peers) - 1 && d < kSmSlice) hist[warp][d] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
}

struct SmMap { int64_t S, M; int f; };                     // B -> max(B + S, M); f: holds the head of a run, so B no longer matters
__device__ __forceinline__ SmMap sm_then(const SmMap &x, const SmMap &y) {        // x first, then y
    if (y.f) return y;
    SmMap r; r.S = x.S + y.S; r.M = max((int64_t)(x.M + y.S), y.M); r.f = x.f; return r;
}
__device__ __forceinline__ SmMap sm_shfl_up(const SmMap &v, int o) {
    SmMap u; u.S = __shfl_up_sync(0xffffffffu, v.S, o); u.M = __shfl_up_sync(0xffffffffu, v.M, o); u.f = __shfl_up_sync(0xffffffffu, v.f, o); return u;
}

__device__ __noinline__ Served small_terms_general(const RangeSnap &rs, const ModelParams &mp, uint64_t addr, int64_t issue, uint64_t bf, int64_t q_ppm, Div64 div_q) {
    unsigned ignored = 0;                                    // (services are 64 bits here)
    return serve_terms(rs, mp, addr, issue, bf, q_ppm, div_q, ignored, 63);
}

// EXTRA: with the ledger or retention
template <bool EXTRA>
__global__ void __launch_bounds__(kSmThreads, 1)
k_small_serve(const __grid_constant__ SmallArgs a) {
    extern __shared__ __align__(16) unsigned char sm_small[];
    __shared__ uint32_t s_cnt[kSmRounds * kSmWarps];         // rows: listed | ready << 16, then the same before the row
    __shared__ uint32_t s_native, s_fault, s_unsorted, s_m, s_ready, s_below, s_last;
    __shared__ unsigned long long s_lo, s_hi;                // smallest and largest issue time of the list (unsorted batches)
    __shared__ int64_t s_busy[kSmSlice];
    __shared__ uint32_t s_nr[kSmSlice], s_np[kSmSlice], s_br[2][kSmSlice], s_bp[2][kSmSlice], s_claims[kSmSlice];
    __shared__ unsigned long long s_work[kSmSlice];
    __shared__ long long s_tot[3];                           // stalls, services, largest completion
    __shared__ Div64 s_div;
    __shared__ uint32_t s_hist[kSmWarps][kSmSlice + 1], s_dtot[kSmSlice];
    __shared__ int64_t w_S[kSmWarps], w_M[kSmWarps];
    __shared__ int w_f[kSmWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const ModelParams &mp = a.mp;
    const RangeSnap &rs = *a.ranges;
    const uint32_t n = a.n, padded = (n + kSmThreads - 1u) / kSmThreads * kSmThreads, rounds = padded / kSmThreads;
    const uint32_t q_lo = blockIdx.x * a.slice, q_n = min(a.slice, mp.n_queues - q_lo);
    const uint32_t per_die = mp.queue_level == 0u ? mp.planes : 1u, d_lo = q_lo / per_die, d_n = q_n / per_die;
    int64_t *s_s = reinterpret_cast<int64_t *>(sm_small);                     // by place in the list: service time
    uint64_t *s_key = reinterpret_cast<uint64_t *>(s_s + padded);             //   issue time << 16 | program << 13 | batch index
    uint32_t *s_px = reinterpret_cast<uint32_t *>(s_key + padded);            //   transfer | claim << 31
    uint16_t *perm0 = reinterpret_cast<uint16_t *>(s_px + padded), *perm1 = perm0 + padded;
    uint8_t *s_lq = reinterpret_cast<uint8_t *>(perm1 + padded);              //   queue in the slice
    const uint64_t *rec0 = reinterpret_cast<const uint64_t *>(a.acc);
    if (tid < (int)kSmSlice) { s_nr[tid] = s_np[tid] = s_br[0][tid] = s_br[1][tid] = s_bp[0][tid] = s_bp[1][tid] = s_claims[tid] = 0u; s_work[tid] = 0ull; }
    if (tid < 3) s_tot[tid] = tid == 2 ? INT64_MIN : 0;
    if (tid == 0) { s_native = s_fault = s_unsorted = s_below = 0u; s_lo = ~0ull; s_hi = 0ull; }
    __syncthreads();
    pdl_wait();                                              // everything above reads kernel arguments only
    pdl_trigger();

    int code = HBF_OK;
    const int32_t mode = a.state->mode;
    const int64_t q_ppm = a.state->q_ppm;
    if (a.state->poisoned) code = HBF_E_TIMEOUT;
    else if (mode == HBF_MODE_SHUTDOWN) code = HBF_E_LINK_SHUTDOWN;
    else if (mode == HBF_MODE_SEVERE) code = HBF_E_THROTTLED;
    if (q_ppm != 1000000) {                                  // (a 128-bit division: one thread makes it)
        if (tid == 0) s_div = make_div64((uint64_t)q_ppm);
        __syncthreads();
    }
    const Div64 div_q = s_div;                               // (not looked at without thermal scaling)
    const bool fast = a.fast.on != 0u && mp.pow2_geom != 0u && mp.xfer_tab_max_cb != 0u && q_ppm == 1000000;
    const bool one_range = a.fast.on != 0u && mp.pow2_geom != 0u;
    unsigned long long debt = 0ull;
    if (EXTRA && a.ret_on) debt = a.ret.st->planned - a.ret.st->claimed - a.ret.st->decayed;
    if ((uint32_t)tid < q_n) { s_busy[tid] = a.busy[q_lo + tid]; if (a.bus_on) a.busy_stage[q_lo + tid] = s_busy[tid]; }   // (the stage of queues without an access)
    uint32_t m = 0, n_ready = 0;
    bool unsorted = false;
    unsigned long long claims = 0ull;

    if (code == HBF_OK) {
        // ---- look: a bit per round (record tid + 1024 k) for ready, listed and native
        uint32_t ready_b = 0, mine_b = 0, native_b = 0, c_fault = 0, c_below = 0;
        unsigned uns = 0;
        for (uint32_t k0 = 0; k0 < rounds; k0 += 4u) {
            uint64_t r_addr[4], r_issue[4], r_bf[4];
#pragma unroll
            for (uint32_t k = 0; k < 4u; ++k) {
                const uint32_t i = (k0 + k) * kSmThreads + tid;
                r_addr[k] = r_issue[k] = r_bf[k] = 0ull;
                if (i < n) { const uint64_t *rec = rec0 + (size_t)i * 3; r_addr[k] = __ldg(rec); r_issue[k] = __ldg(rec + 1); r_bf[k] = __ldg(rec + 2); }
            }
#pragma unroll
            for (uint32_t k = 0; k < 4u; ++k) {
                const uint32_t i = (k0 + k) * kSmThreads + tid;
                if (k0 + k >= rounds) break;                 // (the same for the whole block)
                int64_t prev = (int64_t)__shfl_up_sync(0xffffffffu, r_issue[k], 1);
                if (lane == 0) prev = i > 0u && i < n ? (int64_t)__ldg(rec0 + (size_t)i * 3 - 2) : INT64_MIN;
                bool ready = false, mine = false;
                if (i < n) {
                    if ((int64_t)r_issue[k] < prev) uns = 1u;
                    const uint32_t bytes = (uint32_t)r_bf[k], flags = (uint32_t)(r_bf[k] >> 32);
                    uint32_t q;
                    int st;
                    if (one_range) {
                        const uint64_t rel = r_addr[k] - a.fast.base;
                        st = ((a.fast.perms >> (flags & 1u)) & 1u) ? HBF_ST_READY : HBF_ST_FAULT_PERM;
                        if ((uint64_t)bytes > a.fast.length - rel) st = HBF_ST_FAULT_PARTIAL;
                        if (rel >= a.fast.length) st = HBF_ST_NATIVE;
                        if (bytes == 0u || flags > 1u || (r_issue[k] >> kIssueBits) != 0ull) st = HBF_ST_UNSUPPORTED;
                        const uint32_t u = (uint32_t)((a.fast.media_offset + rel) >> mp.stripe_shift);
                        const uint32_t ch = u & (mp.channels - 1u), di = (u >> mp.ch_shift) & (mp.dies - 1u), pl = (u >> (mp.ch_shift + mp.die_shift)) & (mp.planes - 1u);
                        q = (ch << mp.die_shift) + di;
                        if (mp.queue_level == 0u) q = (q << mp.plane_shift) + pl;
                    } else {
                        int g = 0;
                        st = classify(rs, r_addr[k], (int64_t)r_issue[k], bytes, flags, &g);
                        q = st == HBF_ST_READY ? decode(mp, rs.media_offset[g] + (r_addr[k] - rs.base[g]), bytes).queue : 0u;
                    }
                    ready = st == HBF_ST_READY;
                    mine = ready && q - q_lo < q_n;
                    if (ready && q < q_lo) ++c_below;
                    if (st == HBF_ST_NATIVE) native_b |= 1u << (k0 + k);
                    else if (!ready) ++c_fault;
                    if (a.status && (k0 + k) % gridDim.x == blockIdx.x) a.status[i] = (uint8_t)st;
                }
                ready_b |= ready ? 1u << (k0 + k) : 0u; mine_b |= mine ? 1u << (k0 + k) : 0u;
                const uint32_t c = (uint32_t)__popc(__ballot_sync(0xffffffffu, mine)) | (uint32_t)__popc(__ballot_sync(0xffffffffu, ready)) << 16;
                if (lane == 0) s_cnt[(k0 + k) * kSmWarps + warp] = c;
            }
        }
        {
            const uint32_t w_native = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(native_b)), w_fault = __reduce_add_sync(0xffffffffu, c_fault);
            const uint32_t w_below = __reduce_add_sync(0xffffffffu, c_below);
            uns = __any_sync(0xffffffffu, uns);
            if (lane == 0) {
                if (w_native) atomicAdd(&s_native, w_native);
                if (w_fault) atomicAdd(&s_fault, w_fault);
                if (w_below) atomicAdd(&s_below, w_below);
                if (uns) s_unsorted = 1u;
            }
        }
        __syncthreads();
        if (warp == 0) {                                     // what is listed and ready before every row: eight rows per lane
            uint32_t v[8], sum = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) { v[k] = (uint32_t)(lane * 8 + k) < rounds * kSmWarps ? s_cnt[lane * 8 + k] : 0u; sum += v[k]; }
            uint32_t inc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
            uint32_t run = inc - sum;
#pragma unroll
            for (int k = 0; k < 8; ++k) { if ((uint32_t)(lane * 8 + k) < rounds * kSmWarps) s_cnt[lane * 8 + k] = run; run += v[k]; }
            if (lane == 31) { s_m = inc & 0xffffu; s_ready = inc >> 16; }
        }
        __syncthreads();
        m = s_m; n_ready = s_ready; unsorted = s_unsorted != 0u;
        if (s_fault) code = HBF_E_ACCESS_FAULT;              // fail closed: refuse the batch
        else if (unsorted && a.forced) code = HBF_E_INVAL;
        if (code == HBF_OK) {
            claims = min(debt, (unsigned long long)n_ready);
            for (uint32_t k = 0; k < rounds; ++k) {
                const unsigned bm = __ballot_sync(0xffffffffu, (mine_b >> k) & 1u), br = __ballot_sync(0xffffffffu, (ready_b >> k) & 1u);
                const uint32_t i = k * kSmThreads + tid, before = s_cnt[k * kSmWarps + warp];
                const uint32_t rank = (before >> 16) + __popc(br & lanemask_lt());                 // among the batch's modeled accesses
                const bool claim = EXTRA && ((ready_b >> k) & 1u) && rank < claims;
                if ((mine_b >> k) & 1u) perm1[(before & 0xffffu) + __popc(bm & lanemask_lt())] = (uint16_t)(i | (claim ? 0x8000u : 0u));
                if (EXTRA && a.bus_on && claim && rank + 1u == claims && blockIdx.x == 0) { a.ret.st->claim_limit = claims == debt ? i + 1u : n; a.ret.st->claims_now = claims; }
                if ((native_b >> k) & 1u) if (k % gridDim.x == blockIdx.x) { a.completion[i] = (int64_t)__ldg(rec0 + (size_t)i * 3 + 1); a.stall[i] = 0; }
            }
        }
    }
    const int64_t quantum_ns = !EXTRA ? 0 : q_ppm == 1000000 ? mp.t_read_ns + mp.t_prog_ns
        : (int64_t)div64((uint64_t)(mp.t_read_ns + mp.t_prog_ns) * 1000000ull + (uint64_t)q_ppm - 1ull, div_q);
    if (code == HBF_OK) {
        __syncthreads();                                     // (the code is the same for the whole block, and for every block)
        // ---- terms of the listed records
        unsigned long long lo = ~0ull, hi = 0ull;
        for (uint32_t p = (uint32_t)tid; p < m; p += kSmThreads) {
            const uint32_t i = perm1[p] & (kInSmallMax - 1u), claim = perm1[p] >> 15;
            const uint64_t *rec = rec0 + (size_t)i * 3;
            const uint64_t addr = __ldg(rec), bf = __ldg(rec + 2);
            const int64_t issue = (int64_t)__ldg(rec + 1);
            const Served v = fast ? serve_terms_fast(a.fast, mp, addr, issue, bf) : small_terms_general(rs, mp, addr, issue, bf, q_ppm, div_q);
            s_s[p] = v.s + (claim ? quantum_ns : 0);
            s_key[p] = ((uint64_t)issue << 16) | (v.op << kSmIdxBits) | i;
            s_px[p] = v.xfer | (claim << 31);
            s_lq[p] = (uint8_t)(v.queue - q_lo);
            perm0[p] = (uint16_t)p;
            lo = min(lo, (unsigned long long)issue); hi = max(hi, (unsigned long long)issue);
            const uint32_t ld = v.die - d_lo, lw = (uint32_t)v.cb, hw = (uint32_t)((uint64_t)v.cb >> 32);
            atomicAdd(v.op ? &s_np[ld] : &s_nr[ld], 1u);
            uint32_t *plo = v.op ? &s_bp[0][ld] : &s_br[0][ld], *phi = v.op ? &s_bp[1][ld] : &s_br[1][ld];
            const uint32_t old = atomicAdd(plo, lw), carry = hw + (old + lw < old ? 1u : 0u);
            if (carry) atomicAdd(phi, carry);
            if (EXTRA && claim) atomicAdd(&s_claims[ld], 1u);
            if (EXTRA && a.ret_on && !a.bus_on && !v.op) {   // read disturb: the read's pages, on the block of its first page
                int g = 0;
                uint64_t off;
                if (a.fast.on) off = a.fast.media_offset + (addr - a.fast.base);
                else { classify(rs, addr, issue, (uint32_t)bf, 0u, &g); off = rs.media_offset[g] + (addr - rs.base[g]); }
                const uint64_t page = 1ull << mp.page_shift;
                atomicAdd(&a.ret.disturb[ret_block_of(mp, a.ret, off)], (uint32_t)(((off & (page - 1ull)) + (uint32_t)bf + page - 1ull) >> mp.page_shift));
            }
        }
        if (unsorted) {
            for (int o = 16; o > 0; o >>= 1) { lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
            if (lane == 0 && lo <= hi) { atomicMin(&s_lo, lo); atomicMax(&s_hi, hi); }
        }
        __syncthreads();
        // ---- sort
        uint16_t *src = perm0, *dst = perm1;
        if (unsorted && m > 1u) {
            const unsigned long long first = s_lo, span = s_hi - first;
            for (uint32_t sh = 0; sh < 48u && (span >> sh) != 0ull; sh += 6u) {
                small_sort_pass(src, dst, m, s_hist, s_dtot, [&](uint32_t p) { return (uint32_t)(((s_key[p] >> 16) - first) >> sh) & 63u; });
                uint16_t *t = src; src = dst; dst = t;
            }
        }
        small_sort_pass(src, dst, m, s_hist, s_dtot, [&](uint32_t p) { return (uint32_t)s_lq[p]; });
        const uint16_t *sorted = dst;
        // ---- serve
        long long sum_stall = 0, sum_s = 0, max_c = INT64_MIN;
        const uint32_t per = (m + kSmThreads - 1u) / kSmThreads, p0 = (uint32_t)tid * per, p1 = min(m, p0 + per);   // this thread's entries
        const uint32_t prev_q = p0 > 0u && p0 < m ? s_lq[sorted[p0 - 1u]] : 0xffffffffu;
        SmMap agg; agg.S = 0; agg.M = kNegInf; agg.f = 0;
        {
            uint32_t pq = prev_q, run_die = 0xffffffffu;
            unsigned long long run = 0;
            for (uint32_t p = p0; p < p1; ++p) {
                const uint32_t e = sorted[p], lq = s_lq[e], px = s_px[e], die = lq / per_die;
                const uint64_t key = s_key[e];
                const int64_t s = s_s[e], at = (int64_t)(key >> 16) + ((key >> kSmIdxBits) & 1u ? (int64_t)(px & 0x7fffffffu) : 0);
                SmMap x; x.S = s; x.f = lq != pq; x.M = (x.f ? max(at, s_busy[lq]) : at) + s;
                agg = sm_then(agg, x);
                if (die != run_die) { if (run) atomicAdd(&s_work[run_die], run); run = 0; run_die = die; }
                run += (unsigned long long)s; sum_s += s;
                pq = lq;
            }
            if (run) atomicAdd(&s_work[run_die], run);
        }
        SmMap inc = agg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const SmMap u = sm_shfl_up(inc, o); if (lane >= o) inc = sm_then(u, inc); }
        if (lane == 31) { w_S[warp] = inc.S; w_M[warp] = inc.M; w_f[warp] = inc.f; }
        __syncthreads();
        SmMap wm; wm.S = w_S[lane]; wm.M = w_M[lane]; wm.f = w_f[lane];               // every warp scans the warps' maps for itself
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const SmMap u = sm_shfl_up(wm, o); if (lane >= o) wm = sm_then(u, wm); }
        SmMap ex; ex.S = 0; ex.M = kNegInf; ex.f = 0;         // everything before this thread's entries
        {
            const int w = warp > 0 ? warp - 1 : 0;
            SmMap u; u.S = __shfl_sync(0xffffffffu, wm.S, w); u.M = __shfl_sync(0xffffffffu, wm.M, w); u.f = __shfl_sync(0xffffffffu, wm.f, w);
            if (warp > 0) ex = u;
            u = sm_shfl_up(inc, 1);
            if (lane > 0) ex = sm_then(ex, u);
        }
        // (the first entry of the list is a head, so a map without a head never reaches an entry that needs its input)
        int64_t B = ex.M;
        uint32_t pq = prev_q;
        for (uint32_t p = p0; p < p1; ++p) {
            const uint32_t e = sorted[p], lq = s_lq[e], px = s_px[e], i = (uint32_t)s_key[e] & (kInSmallMax - 1u), op = (uint32_t)(s_key[e] >> kSmIdxBits) & 1u;
            const int64_t issue = (int64_t)(s_key[e] >> 16), s = s_s[e], x = (int64_t)(px & 0x7fffffffu);
            if (lq != pq) B = s_busy[lq];
            B = max(issue + (op ? x : 0), B) + s;
            const int64_t c = B + (op ? 0 : x), waited = c - issue;
            a.completion[i] = c; a.stall[i] = waited;
            sum_stall += waited; max_c = max(max_c, (long long)c);
            if (p + 1u == m || s_lq[sorted[p + 1u]] != lq)   // last access of its queue in this batch
                (a.bus_on ? a.busy_stage : a.busy)[q_lo + lq] = B;
            if (unsorted) a.order[s_below + p] = i;
            if (EXTRA && a.ledger && !a.bus_on) {
                const bool claim = (px >> 31) != 0u;
                const int64_t own = s - (claim ? quantum_ns : 0), page = (int64_t)1 << mp.page_shift;
                const uint64_t gm = (1ull << (op ? mp.prog_gran_shift : mp.read_gran_shift)) - 1ull, cb = ((uint64_t)(uint32_t)__ldg(rec0 + (size_t)i * 3 + 2) + gm) & ~gm;
                const uint32_t die = d_lo + lq / per_die;
                const int64_t pj = op ? mp.e_cmd_prog_pj + mp.e_byte_prog_pj * (int64_t)cb : mp.e_cmd_read_pj + mp.e_byte_read_pj * (int64_t)cb;
                if (claim) ledger_event(a.ledger, mp.n_dies, a.n_bins, a.cur_bin, a.bin_ns, die, B - s, quantum_ns,
                                        mp.e_cmd_read_pj + mp.e_byte_read_pj * page + mp.e_cmd_prog_pj + mp.e_byte_prog_pj * page);
                ledger_event(a.ledger, mp.n_dies, a.n_bins, a.cur_bin, a.bin_ns, die, B - own, own, pj);
            }
            pq = lq;
        }
        sum_stall = warp_sum(sum_stall); sum_s = warp_sum(sum_s); max_c = warp_max(max_c);
        if (lane == 0) {
            if (sum_stall) atomicAdd((unsigned long long *)&s_tot[0], (unsigned long long)sum_stall);
            if (sum_s) atomicAdd((unsigned long long *)&s_tot[1], (unsigned long long)sum_s);
            if (max_c != INT64_MIN) atomicMax(&s_tot[2], max_c);
        }
        __syncthreads();
        // ---- per-die totals of the slice
        const int64_t page = (int64_t)1 << mp.page_shift;
        const int64_t quantum_pj = mp.e_cmd_read_pj + mp.e_byte_read_pj * page + mp.e_cmd_prog_pj + mp.e_byte_prog_pj * page;
        if ((uint32_t)tid < d_n) {
            hbf_die_stats_t ds;
            ds.busy_ns = (int64_t)s_work[tid];
            ds.bytes_read = (int64_t)(((uint64_t)s_br[1][tid] << 32) | s_br[0][tid]); ds.bytes_prog = (int64_t)(((uint64_t)s_bp[1][tid] << 32) | s_bp[0][tid]);
            ds.n_read = s_nr[tid]; ds.n_prog = s_np[tid];
            ds.energy_pj = mp.e_cmd_read_pj * ds.n_read + mp.e_byte_read_pj * ds.bytes_read + mp.e_cmd_prog_pj * ds.n_prog + mp.e_byte_prog_pj * ds.bytes_prog;
            const uint32_t d = d_lo + tid;
            if (a.bus_on) {
                a.stats_stage[d] = ds;
                if (EXTRA && a.ret_on) a.ret.die_claims[d] = s_claims[tid];
            } else {
                if (a.die_stats) a.die_stats[d] = ds;
                if (!a.ledger) a.pending[d] += ds.energy_pj + (EXTRA ? (int64_t)s_claims[tid] * quantum_pj : 0);
            }
        }
        if (EXTRA && a.ret_on && !a.bus_on && claims) {      // blocks whose last quantum is now claimed commit one cycle
            const unsigned long long mark = a.ret.st->planned - debt + claims;
            for (uint64_t b = (uint64_t)blockIdx.x * kSmThreads + tid; b < a.ret.n_blocks; b += (uint64_t)gridDim.x * kSmThreads)
                if (a.ret.epoch_of[b] != 0u && a.ret.last_pos[b] < mark) ret_commit_block(a.ret, b);
        }
    } else if (code != HBF_E_LINK_SHUTDOWN && code != HBF_E_THROTTLED) {              // refused: zeroed outputs, nothing changed
        for (uint32_t i = blockIdx.x * kSmThreads + tid; i < n; i += gridDim.x * kSmThreads) { a.completion[i] = 0; a.stall[i] = 0; }
        if (a.die_stats) for (uint32_t e = (uint32_t)tid; e < d_n * 6u; e += kSmThreads) reinterpret_cast<int64_t *>(a.die_stats + d_lo)[e] = 0;
    }
    // ---- totals; the block that comes last writes the summary
    __syncthreads();
    if (tid == 0) {
        if (code == HBF_OK) {
            if (s_tot[0]) atomicAdd(&a.tot->modeled_ns, (unsigned long long)s_tot[0]);
            if (s_tot[1]) atomicAdd(&a.tot->service_ns, (unsigned long long)s_tot[1]);
            if (s_tot[2] != INT64_MIN) atomicMax(&a.tot->max_completion_ns, s_tot[2]);
        }
        __threadfence();
        s_last = atomicAdd(&a.tot->done, 1u) == gridDim.x - 1u ? 1u : 0u;
        __threadfence();
        if (s_last) { s_tot[0] = (long long)__ldcg(&a.tot->modeled_ns); s_tot[1] = (long long)__ldcg(&a.tot->service_ns); s_tot[2] = __ldcg(&a.tot->max_completion_ns); }
    }
    __syncthreads();
    if (!s_last) return;
    const long long modeled = s_tot[0], service = s_tot[1], latest = s_tot[2];
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
        a.tot->modeled_ns = 0ull; a.tot->service_ns = 0ull; a.tot->max_completion_ns = 0; a.tot->done = 0u;
        hbf_batch_result_t r;
        const bool ok = code == HBF_OK, seen = ok || code == HBF_E_ACCESS_FAULT;
        r.code = code; r.mode = mode; r.q_ppm = q_ppm;
        r.n_native = seen ? s_native : 0u; r.n_modeled = ok ? n_ready : 0u; r.n_fault = code == HBF_E_INVAL ? 0u : s_fault;
        r.modeled_ns = ok ? modeled : 0; r.service_ns = ok ? service : 0; r.max_completion_ns = ok && n_ready ? latest : 0;
        *a.result = r;
        BatchCtrl *c = a.ctrl;                               // what later stages and hbf_queue_order read of a batch
        c->code = code; c->skip = ok ? 0 : 1; c->mode = mode; c->q_ppm = q_ppm; c->div_q = div_q;
        c->n_ready = n_ready; c->inorder_used = ok && !unsorted ? 1u : 0u; c->run_sort = 0u; c->plan.n_passes = 1u;
        if (EXTRA && a.ret_on && !a.bus_on && ok) a.ret.st->claimed += claims;
    }
}

// whether a batch takes this route (launch_small serves it whole)
bool small_route(const SubmitArgs &a) {
    return a.n > 0 && a.n <= kInSmallMax && a.inorder_ok && !a.paged && (a.path == HBF_PATH_AUTO || a.path == HBF_PATH_INORDER) && small_slice(a.mp) != 0u;
}

cudaError_t launch_small(const SubmitArgs &a, const SmallExtras &x, cudaStream_t st) {
    SmallArgs s{};
    s.acc = a.acc; s.n = (uint32_t)a.n; s.slice = small_slice(a.mp); s.forced = a.path == HBF_PATH_INORDER ? 1u : 0u; s.bus_on = a.bus_on ? 1u : 0u;
    s.ranges = a.ranges; s.fast = a.fast; s.mp = a.mp; s.state = a.state; s.ctrl = a.ctrl; s.tot = x.tot; s.result = a.result;
    s.busy = a.busy; s.busy_stage = a.busy_stage; s.pending = a.pending; s.stats_stage = a.stats_stage; s.die_stats = a.die_stats;
    s.completion = a.completion; s.stall = a.stall; s.status = a.status; s.order = a.ws.idx[1];
    s.ledger = x.ledger; s.bin_ns = x.bin_ns; s.cur_bin = x.cur_bin; s.n_bins = x.n_bins; s.ret_on = a.ret ? 1u : 0u;
    if (a.ret) s.ret = *a.ret;
    auto k = s.ledger || s.ret_on ? k_small_serve<true> : k_small_serve<false>;
    const size_t smem = small_smem(s.n);
    cudaError_t e = ensure_dyn_smem((const void *)k, small_smem(kInSmallMax));
    if (e != cudaSuccess) return e;
    g_kernel_launches += 1;
    return launch_pdl(k, (a.mp.n_queues + s.slice - 1) / s.slice, kSmThreads, smem, st, s);
}

}  // namespace hbf

// In-order path of hbf_submit_batch: serves a batch whose records arrive in non-decreasing issue order
// without a global sort.  In such a batch the (issue, index) order of every queue is plain index order,
// so the batch is cut into contiguous tiles, one per resident thread block, that are served independently:
//   serve     every tile classifies and decodes its records, writes status[], counts, sums per-die bytes, and
//             serves its accesses AS IF every queue were idle when the tile begins; completions and stalls
//             are written as they are computed, in batch order.  Per queue it also keeps the composition
//             (S, M) of the maps B -> max(B + s, a + s) of its accesses (M is exactly the busy-until of the
//             as-if run) and the first few accesses of the queue in the tile (the head table);
//   scan      one thread per queue walks the tiles' aggregates in order: the true busy-until entering each
//             tile, and the final busy-until;
//   fix-up    one thread per (tile, queue) starts from the true entering busy-until and re-serves the head
//             table's accesses in order, until it meets an access that arrives when the queue is idle: from
//             there on the as-if run and the true run coincide (busy-until is monotone in its start value, so
//             the as-if run was idle there too);
//   straggle  a queue still backlogged past its head entries is re-served from the records: the tile's
//             block streams the tile again, keeps only that tile's straggling queues, and stops as soon as
//             each of them has fallen idle;
//   re-serve  a tile with many stragglers (the batch arrived on queues that were far behind) is served
//             again from the true entering busy-until, exactly.
// Smaller batches (twice_max) skip fix-up and straggle: serve without results, scan, re-serve of every tile.
// The serve pass is the only one that streams the whole batch: 24 B read and 16 B + 1 B written per access.
// Every global access of it is coalesced; nothing waits on another thread block, and no thread spins.
//
// Inside a tile the busy-until of every queue lives in shared memory.  The records are taken 32 at a time
// (a row per warp, rows dealt round-robin to the block's warps); all the per-record arithmetic runs in
// parallel, and only the read-serve-write of the queue state is done row after row, handed from warp to
// warp through the hardware's named barriers.  Records of one queue that fall into the same row are chained
// in registers with shuffles.
#include <algorithm>
#include <cstddef>
#include <type_traits>

#include "serve_terms.cuh"

namespace hbf {

// Block shape of the serve kernel: two blocks per SM, each with its own tile and its own row-after-row chain of queue updates.
// (12 warps a block: with the 32-bit form a 200 M batch takes 1,587 us, with 10 warps 1,667, 11: 1,700, 13: 1,720, 14: 1,669;
// three or four blocks of 8 to 10 warps 1,890 to 2,500: more tiles in flight are more streams to DRAM, which the pass keeps
// at 5.7 TB/s.)
#ifndef HBF_IN_THREADS
#define HBF_IN_THREADS 384
#endif
#ifndef HBF_IN_BLOCKS
#define HBF_IN_BLOCKS 2
#endif
constexpr int kInThreads = HBF_IN_THREADS;               // threads of a serve block
constexpr uint32_t kInTwiceRun = 15;                      // batches served twice at once before one takes the fix-up again (see twice_max)
constexpr int kInBlocksPerSM = HBF_IN_BLOCKS;            // resident serve blocks per SM
constexpr int kInWarps = kInThreads / 32;
constexpr uint32_t kInTagStride = kInMaxQueues + 32;      // bytes of a warp's table of lane numbers: one per queue, one per lane
#ifndef HBF_IN_ROWS
#define HBF_IN_ROWS 2
#endif
#ifndef HBF_IN_PFDIST
#define HBF_IN_PFDIST 2
#endif
constexpr int kInPrefetchTurns = HBF_IN_PFDIST;          // how many of the warp's turns ahead its records are called into the L2
constexpr int kInRows = HBF_IN_ROWS;                     // rows of 32 records a warp serves per turn
static_assert(kInWarps >= 2 && kInWarps <= 15, "every warp owns one of the hardware barriers 1..15");

// No branches: every access computes every term, and the classification (the same tests in the same order as classify())
// only selects the status; the terms of an access that is not READY are never used.  (Early returns cost this pass
// about 47 instructions per row of 32 accesses, measured.)
__device__ __forceinline__ Served serve_terms_geom(const FastGeom &g, const ModelParams &mp, uint64_t addr, int64_t issue, uint64_t bf,
                                                  int64_t q_ppm, const Div64 &div_q, unsigned &long_service, int long_bits) {
    Served r; r.parts = 1;
    const uint32_t bytes = (uint32_t)bf, flags = (uint32_t)(bf >> 32);
    const uint64_t rel = addr - g.base;                       // wraps to a huge value below the base
    const uint32_t op = flags & 1u;
    const bool unsupported = bytes == 0u || flags > 1u || (uint32_t)((uint64_t)issue >> 32) >= (1u << (kIssueBits - 32));
    const bool outside = rel >= g.length;
    const bool partial = (uint64_t)bytes > g.length - rel;
    const bool denied = ((g.perms >> op) & 1u) == 0u;
    int st = denied ? HBF_ST_FAULT_PERM : HBF_ST_READY;
    st = partial ? HBF_ST_FAULT_PARTIAL : st;
    st = outside ? HBF_ST_NATIVE : st;
    r.st = unsupported ? HBF_ST_UNSUPPORTED : st;
    r.op = op;
    const uint64_t off = g.media_offset + rel;
    const uint32_t u = (uint32_t)(off >> g.stripe_shift);     // only the low interleave bits are used
    const uint32_t ch = u & g.ch_mask, di = (u >> g.ch_shift) & g.die_mask, pl = (u >> g.chdie_shift) & g.plane_mask_q;
    r.die = ch * g.dies + di;
    r.queue = r.die * g.planes_q + pl;
    const uint32_t npages = (uint32_t)(((uint64_t)((uint32_t)off & g.page_mask) + bytes + g.page_mask) >> g.page_shift);
    const uint32_t gs = op ? g.gran_shift_prog : g.gran_shift_read;
    const uint64_t gm = (1ull << gs) - 1ull;
    const uint64_t cb = ((uint64_t)bytes + gm) & ~gm;
    r.cb = (int64_t)cb;
    const uint64_t s0 = (uint64_t)npages * (op ? g.t_prog : g.t_read);
    if (cb <= (uint64_t)g.tab_max_cb) {
        r.xfer = __ldg(g.xfer_tab + ((uint32_t)cb >> g.tab_shift));
    } else {                                                  // a large access: rare
        r.xfer = (uint32_t)div64(cb * 1000ull + mp.chan_bytes_per_us - 1ull, mp.div_chan);
        if (s0 >> long_bits) long_service = 1u;
    }
    if (q_ppm == 1000000) {
        r.s = (int64_t)s0;
    } else {                                                  // thermal scaling in force: Eq. 3 (s0 < 2^50)
        r.s = (int64_t)div64(s0 * 1000000ull + (uint64_t)q_ppm - 1ull, div_q);
        if ((uint64_t)r.s >> long_bits) long_service = 1u;
    }
    return r;
}
// ---- page-granular submit, without the list of parts ----------------------------------------------------------------
// The pages of an access that stays inside one stripe unit lie on one plane, so its parts are consecutive requests of one
// queue: together they are one map B -> max(B + S, M) again, and the access ends with the latest of them.  With k parts of
// service s each and transfers x_1, x, ..., x, x_k (the first and the last part may be shorter than a page):
//   reads     all parts arrive when the access is issued: M = issue + k s; part j is done k - j services before the last, so the
//             access ends max(x_k, x - s, x_1 - (k - 1) s) after the last service
//   programs  part j arrives x_j after the issue: M = issue + max(x_1 + k s, x + (k - 1) s, x_k + s), S = k s; it ends with the
//             last service
// so an access is served as one entry with these terms in the place of its own (xfer: what follows the service of a read, or
// M - S - issue of a program).  Bytes are charged and operations counted per part.
__device__ __forceinline__ void paged_terms(const ModelParams &mp, uint64_t off, uint32_t bytes, int64_t q_ppm, const Div64 &div_q,
                                            unsigned &long_service, int long_bits, Served &r) {
    const uint64_t page = 1ull << mp.page_shift, in_page = off & (page - 1ull);
    const uint64_t k = (in_page + bytes + page - 1ull) >> mp.page_shift;
    const uint64_t head = min((uint64_t)bytes, page - in_page), tail = in_page + bytes - (k - 1ull) * page;      // (k == 1: the head is the access)
    const uint64_t gm = (1ull << (r.op ? mp.prog_gran_shift : mp.read_gran_shift)) - 1ull;
    auto charged = [&](uint64_t b) { return (b + gm) & ~gm; };
    auto transfer = [&](uint64_t cb) { return (int64_t)div64(cb * 1000ull + mp.chan_bytes_per_us - 1ull, mp.div_chan); };
    const int64_t t = r.op ? mp.t_prog_ns : mp.t_read_ns;
    const int64_t s1 = q_ppm == 1000000 ? t : (int64_t)div64((uint64_t)t * 1000000ull + (uint64_t)q_ppm - 1ull, div_q);
    r.parts = (uint32_t)k;
    r.s = (int64_t)k * s1;
    if ((uint64_t)r.s >> long_bits) long_service = 1u;
    const int64_t xh = transfer(charged(head));
    r.cb = (int64_t)charged(head);
    if (k == 1ull) { r.xfer = (uint32_t)xh; return; }
    const int64_t xp = transfer(charged(page)), xt = transfer(charged(tail));
    r.cb += (int64_t)(charged(tail) + (k - 2ull) * charged(page));
    const int64_t n1 = (int64_t)k - 1;
    int64_t x = r.op ? max(xh, xt - n1 * s1) : max(xt, xh - n1 * s1);
    if (k > 2ull) x = max(x, xp - s1);
    r.xfer = (uint32_t)x;
}
// media offset of a modeled access
__device__ __forceinline__ uint64_t media_offset_of(const RangeSnap &rs, const FastRange &f, bool one, uint64_t addr, int64_t issue, uint64_t bf) {
    if (one) return f.media_offset + (addr - f.base);
    int g = 0;
    classify(rs, addr, issue, (uint32_t)bf, (uint32_t)(bf >> 32), &g);
    return rs.media_offset[g] + (addr - rs.base[g]);
}
// The first kInHead accesses of every (tile, queue), as the serve pass saw them: all the fix-up needs in the common case.
// (Six, measured on the capacity stream at loads 0.3 to 0.9: eight cost 2.5 % more at every load for the table's traffic
// and bookkeeping and fell back to a second pass at the same load, between 0.6 and 0.7; five or fewer are faster still
// at low load but need the second pass from 0.6 on.)
constexpr int kInHead = 6;
struct InHead { int64_t m, s; uint32_t xo, idx; };       // arrival + service, service, transfer | op << 31, batch index
// Where entry ci of (tile, queue) sits: a tile's first entries side by side (the fix-up reads the first entry of every
// queue: one coalesced stretch instead of a record every 192 bytes), then every queue's later entries side by side (read
// only for the queues still behind, all of them at once).
__device__ __forceinline__ uint64_t head_slot(uint32_t tile, uint32_t R, uint32_t q, uint32_t ci) {
    const uint64_t base = (uint64_t)tile * R * kInHead;
    return ci == 0u ? base + q : base + R + (uint64_t)q * (kInHead - 1) + (ci - 1u);
}

// ======================================================================================================
// serve.  RESERVE = false: the streaming pass over every tile, every queue taken as idle at the tile's start.
// RESERVE = true: only for tiles the fix-up flagged (many queues stayed backlogged far into the tile): the
// same pass from the true entering busy-until, writing the exact results and nothing else.
//
// A tile is cut into rows of 32 consecutive records; warp w takes rows w, w + W, w + 2W, ...  Everything that
// does not depend on the queues' state (load, classification, decode, service terms, the ranking of lanes that
// hold the same queue) happens in parallel.  The queue update itself (read the busy-until, serve, write it
// back: a handful of instructions) is done row after row: the warp of row r waits on a hardware barrier that
// the warp of row r - 1 arrives at when its update is in shared memory.  Warp w owns barrier 1 + w: it is the
// only one that waits on it, and warp w - 1 the only one that arrives, so uses of a barrier cannot overlap.
// ======================================================================================================
// The extra operands are not used by the instruction: naming them makes the compiler finish computing them
// before the wait instead of after it.  The aligned forms of the barrier instructions are used (measured a
// little faster): like __syncthreads(), they sit where the warp's control flow is uniform.
__device__ __forceinline__ void row_pass(int id) { asm volatile("barrier.cta.arrive.aligned %0, 64;" ::"r"(id) : "memory"); }

__device__ __forceinline__ void row_wait2(int id, int64_t m, long long s8, const void *pq, uint32_t pc, bool last,
                                          int64_t m2, long long s82, const void *pq2, uint32_t pc2, bool last2) {
    asm volatile("barrier.cta.sync.aligned %0, 64;" ::"r"(id), "l"(m), "l"(s8), "l"(pq), "r"(pc), "r"((int)last),
                 "l"(m2), "l"(s82), "l"(pq2), "r"(pc2), "r"((int)last2) : "memory");
}


// ======================================================================================================
// The streaming pass in 32-bit arithmetic, for the common configuration (one range, powers of two, no thermal scaling).  A
// tile spans milliseconds, so inside it a time is 32 bits from the tile's first issue time: the maps, their composition
// and the ordered update are single instructions where 64-bit ones take two to four, and the state of a queue has room for
// the bytes and the number of its reads, which the update that owns the queue adds up (they were three shared-memory
// atomics per access).  The transfer time is a multiply-high instead of a table look-up.  Programs, accesses near the end
// of the range or larger than nw_bytes, and whatever is not modeled take a branch of their own.
// Bound by DRAM (42.2 B per access at 5.7 TB/s, 0.87 of a copy) with the L1's data pipe close behind (70 % busy).  Measured on
// the 200 M capacity batch, pass with everything around it: 2,086 -> 1,687 us (7.4 -> 5.3 warp instructions per access).
// Tried and not kept: the records through shared memory by a bulk copy per turn (L1 pipe 70 -> 55 % busy, but 1,650 us with an L2
// prefetch ahead of it and 1,710 without, against 1,587 for the submit alone); both rows of a turn updated side by side, with
// queues shared across the rows composed in registers (shorter chain, 8 % more instructions: 1,626); four rows per turn (the same).
// Queue states lie by slot (queue_slot), and tiles that have to be served again take this form too: 24 M records of the prefix
// stream, whose rows walk along the channels, 359 -> 234 us and 306 -> 175 (the L1's data pipe was 84 % busy, 66 bank conflicts per
// row); with everything around it 790 -> 503.  (In the 64-bit form the slots cost mixed batches 4 %: it keeps the queue's number.)
// What the form cannot hold (a time 2^31 ns or more past the tile's first, by a gap in the stream or by a backlog) is
// only noticed, in bits that are OR-ed along; such a tile is then served again in the 64-bit form.
// Queue state (16 bytes; the first 8 or 4 in the other two modes below): busy-until, service time in this tile, read granules,
// reads << 4 | head entries written.
// ======================================================================================================
// What a launch of the pass does: all of it; the results only, from known busy-until; what those follow from only, a map per queue.
// Where the second follows the third (the tile's `reserve` is 2) it also counts what the third leaves out: bytes and accesses per die
// and claims.  The chain of updates then carries 8 bytes a queue and 4, where all 16 take four times the shared memory's turns (4 M decode
// reads 117.6 -> 111.9 us, 24 M prefix records 397 -> 385, first half of 48 M with retention: light 216 -> 199, again 184 -> 174).  Read
// disturb stays with the third: its atomics, all over the L2, take 50 us of a 24 M batch there and 105 beside the stores of the results.
// The last is the third on a page-granular batch whose accesses are not known to stay inside their stripe units: it finds out, and counts pages.
enum { kInFull = 0, kInAgain = 1, kInLight = 2, kInLook = 3 };
struct NarrowSums { uint32_t native, fault, max_done; unsigned unsorted, over; long long stall; };

__device__ __forceinline__ uint32_t nw_transfer(const FastGeom &g, uint32_t granules, uint32_t mul) {
    return __umulhi(granules * mul + g.nw_add, g.nw_magic) >> g.nw_shift;
}

__device__ __forceinline__ void row_wait_n(int id, uint32_t m, uint32_t s, const void *pq, uint32_t gn, bool last,
                                           uint32_t m2, uint32_t s2, const void *pq2, uint32_t gn2, bool last2) {
    asm volatile("barrier.cta.sync.aligned %0, 64;" ::"r"(id), "r"(m), "r"(s), "l"(pq), "r"(gn), "r"((int)last),
                 "r"(m2), "r"(s2), "l"(pq2), "r"(gn2), "r"((int)last2) : "memory");
}

// MODE: see k_inorder_serve.  Everything per queue goes by the queue's slot.
// count: see kInLight (a pass that knows its busy-until).  prog_pages: pages of programs (kInLook).
template <int MODE, bool DEBT, bool PAGED>
__device__ __forceinline__ NarrowSums serve_narrow(const FastGeom &geom, const ModelParams &mp, const ModelParams &mp_arg, const hbf_access_t *acc_t, const uint32_t tile_begin,
                                                   const uint32_t tile_len, const int64_t T0, uint4 *qst, uint8_t *warp_tag, uint8_t *status_t,
                                                   uint16_t *qid_t, const uint32_t qid_stride, int64_t *completion_t, int64_t *stall_t,
                                                   InHead *__restrict__ in_head, const uint32_t tile, const uint32_t R, const uint32_t head_depth,
                                                   uint32_t *s_heads_full, uint32_t *st_br_lo, const uint32_t n_dies,
                                                   const uint64_t claim_limit, const uint32_t quantum_ns, const RetDev &ret, const uint32_t ret_row_shift, const bool count, uint32_t *prog_pages) {
    constexpr bool RESERVE = MODE == kInAgain, LOOK = MODE == kInLook, LIGHT = MODE == kInLight || LOOK;
    const bool counts = MODE == kInFull || (RESERVE && count);
    constexpr int K = kInRows;
    using State = typename std::conditional<RESERVE, uint32_t, typename std::conditional<LIGHT, uint2, uint4>::type>::type;
    const uint32_t die_mask = (1u << geom.chdie_shift) - 1u, unit_mask = (1u << geom.stripe_shift) - 1u;
    uint32_t *st_gran = reinterpret_cast<uint32_t *>(qst) + kInMaxQueues;      // (counting with known busy-until: read granules by the low bits of the slot)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t *st_br_hi = st_br_lo + n_dies, *st_bp_lo = st_br_hi + n_dies, *st_bp_hi = st_bp_lo + n_dies, *st_nr = st_bp_hi + n_dies, *st_np = st_nr + n_dies, *st_claims = st_np + n_dies;
    NarrowSums r; r.native = 0; r.fault = 0; r.max_done = 0; r.unsorted = 0; r.over = 0; r.stall = 0;
    uint32_t b_time = 0, b_hi = 0, b_sort = 0;               // OR-ed along: bit 31 of times, high words of times, sign of issue - previous issue
    const uint32_t rows = (tile_len + 31u) / 32u, turns = (rows + K - 1) / K;
    const unsigned le_mask = lanemask_lt() | (1u << lane);
    const int my_bar = 1 + warp, next_bar = 1 + (warp + 1 == kInWarps ? 0 : warp + 1);
    uint64_t nx_addr[K], nx_issue[K], nx_bf[K];
    uint32_t nx_prev[K];                                     // low word of the issue time before the lane's own
#pragma unroll
    for (int u = 0; u < K; ++u) { nx_addr[u] = 0; nx_issue[u] = 0; nx_bf[u] = 0; nx_prev[u] = 0; }
    const bool pf_lane = lane < 24;
    const char *pf_base = reinterpret_cast<const char *>(acc_t) + lane * 32;
    auto fetch = [&](uint32_t turn) {
#pragma unroll
        for (int u = 0; u < K; ++u) {
            const uint32_t j = (turn * K + u) * 32u + (uint32_t)lane;
            if (j < tile_len) {
                const uint64_t *rec = reinterpret_cast<const uint64_t *>(acc_t + j);
                nx_addr[u] = __ldcs(rec); nx_issue[u] = __ldcs(rec + 1); nx_bf[u] = __ldcs(rec + 2);   // read once: streaming loads
                if (!RESERVE) nx_prev[u] = j > 0u ? ld_after(reinterpret_cast<const uint32_t *>(rec - 2)) : (uint32_t)T0;   // (the tile's first record was compared before)
            }
        }
    };
    fetch((uint32_t)warp);
    for (uint32_t turn = (uint32_t)warp; turn < turns; turn += kInWarps) {
      auto whole_turn = [&](auto full_tag) {
        constexpr bool FULL = decltype(full_tag)::value;
        uint32_t i[K], ri[K], q[K], S[K], M[K], xo[K], gn[K];
        bool valid[K], ready[K];
        uint64_t addr[K], bf[K]; int64_t issue[K]; uint32_t prev[K];
#pragma unroll
        for (int u = 0; u < K; ++u) {
            i[u] = (turn * K + u) * 32u + (uint32_t)lane;
            valid[u] = FULL || i[u] < tile_len;
            addr[u] = nx_addr[u]; bf[u] = nx_bf[u]; issue[u] = (int64_t)nx_issue[u]; prev[u] = nx_prev[u];
        }
        fetch(turn + kInWarps);
        {                                                    // and the turn after that is called into the L2
            const uint32_t first = (turn + kInPrefetchTurns * kInWarps) * (uint32_t)(K * 32);
            if (pf_lane && first + K * 32 <= tile_len) {
                const char *p = pf_base + (size_t)first * sizeof(hbf_access_t);
#pragma unroll
                for (int u = 0; u < K; ++u) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + u * 768));
            }
        }
        // ---- terms
#pragma unroll
        for (int u = 0; u < K; ++u) {
            const uint32_t bytes = (uint32_t)bf[u], flags = (uint32_t)(bf[u] >> 32);
            const uint64_t dt = (uint64_t)(issue[u] - T0), rel = addr[u] - geom.base, off = addr[u] + geom.nw_delta;
            ri[u] = (uint32_t)dt;
            ready[u] = valid[u] && rel <= geom.nw_lim && bytes - 1u < geom.nw_bytes && flags - geom.nw_flag_lo < geom.nw_flag_n;
            if (valid[u]) { b_hi |= (uint32_t)(dt >> 32); b_time |= ri[u]; if (!RESERVE) b_sort |= (uint32_t)issue[u] - prev[u]; }
            q[u] = 0; S[u] = 0; M[u] = 0; xo[u] = 0; gn[u] = 0;
            uint32_t st = HBF_ST_READY;
            const bool common = ready[u];
            if (common) {
                const uint32_t w = (uint32_t)(off >> geom.stripe_shift), in_page = (uint32_t)off & geom.page_mask;
                q[u] = w & geom.nw_slot_mask;
                const uint32_t npages = (in_page + bytes + geom.page_mask) >> geom.page_shift;
                if (LOOK) b_hi |= (((uint32_t)off & unit_mask) + bytes - 1u) >> geom.stripe_shift;   // (crosses its unit: for the 64-bit form to see)
                if (flags == 0u) {
                    const uint32_t g = (bytes + ((1u << geom.gran_shift_read) - 1u)) >> geom.gran_shift_read;
                    S[u] = npages * geom.t_read; xo[u] = nw_transfer(geom, g, geom.nw_mul_read);
                    uint32_t parts = 1u, sum = g;
                    if (PAGED && npages > 1u) {              // (see paged_terms)
                        const uint32_t head = geom.page_mask + 1u - in_page, tail = in_page + bytes - (npages - 1u) * (geom.page_mask + 1u), gm = (1u << geom.gran_shift_read) - 1u;
                        const uint32_t gh = (head + gm) >> geom.gran_shift_read, gt = (tail + gm) >> geom.gran_shift_read;
                        const int32_t s1 = (int32_t)geom.t_read;
                        int32_t x = max((int32_t)nw_transfer(geom, gt, geom.nw_mul_read), (int32_t)nw_transfer(geom, gh, geom.nw_mul_read) - (int32_t)(npages - 1u) * s1);
                        if (npages > 2u) x = max(x, (int32_t)geom.nw_page_read - s1);
                        xo[u] = (uint32_t)x;
                        parts = npages; sum = gh + gt + (npages - 2u) * geom.nw_page_gran;
                    }
                    M[u] = ri[u] + S[u];
                    if (MODE == kInFull) gn[u] = sum | (parts << kNwCountShift);
                    else if (counts) { atomicAdd(&st_gran[q[u] & die_mask], sum); atomicAdd(&st_nr[slot_die(geom, q[u])], parts); }
                } else {                                     // a program: its data is transferred first; bytes and count by atomics
                    uint32_t g = (bytes + ((1u << geom.gran_shift_prog) - 1u)) >> geom.gran_shift_prog, xf = nw_transfer(geom, g, geom.nw_mul_prog);
                    S[u] = npages * geom.t_prog;
                    if (LOOK) atomicAdd(prog_pages, npages);
                    if (PAGED && npages > 1u) {
                        const uint32_t head = geom.page_mask + 1u - in_page, tail = in_page + bytes - (npages - 1u) * (geom.page_mask + 1u), gm = (1u << geom.gran_shift_prog) - 1u;
                        const uint32_t gh = (head + gm) >> geom.gran_shift_prog, gt = (tail + gm) >> geom.gran_shift_prog;
                        const int32_t s1 = (int32_t)geom.t_prog;
                        int32_t x = max((int32_t)nw_transfer(geom, gh, geom.nw_mul_prog), (int32_t)nw_transfer(geom, gt, geom.nw_mul_prog) - (int32_t)(npages - 1u) * s1);
                        if (npages > 2u) x = max(x, (int32_t)geom.nw_page_prog - s1);
                        xf = (uint32_t)x; g = gh + gt + (npages - 2u) * ((geom.page_mask + 1u + gm) >> geom.gran_shift_prog);
                    }
                    xo[u] = xf | 0x80000000u;
                    M[u] = ri[u] + xf + S[u];
                    if (counts) {
                        const uint32_t die = slot_die(geom, q[u]), lo = g << geom.gran_shift_prog;
                        atomicAdd(&st_np[die], PAGED ? npages : 1u);
                        const uint32_t old = atomicAdd(&st_bp_lo[die], lo);
                        if (old + lo < old) atomicAdd(&st_bp_hi[die], 1u);
                    }
                }
                if (DEBT && tile_begin + i[u] < claim_limit) {
                    S[u] += quantum_ns; M[u] += quantum_ns;
                    if (counts) atomicAdd(&st_claims[slot_die(geom, q[u])], 1u);
                }
            } else if (valid[u]) {                           // near the range's end, large, or not modeled
                unsigned lng = 0;
                Served v = serve_terms_geom(geom, mp, addr[u], issue[u], bf[u], 1000000, Div64{}, lng, (int)kNwServeBits - 1);
                if (PAGED && v.st == HBF_ST_READY) paged_terms(mp, off, bytes, 1000000, Div64{}, lng, (int)kNwServeBits - 1, v);
                st = (uint32_t)v.st;
                if (LOOK && v.st == HBF_ST_READY) {
                    if ((uint64_t)((uint32_t)off & unit_mask) + bytes > (uint64_t)unit_mask + 1u) b_hi |= 1u;
                    if (v.op) atomicAdd(prog_pages, v.parts);
                }
                if (v.st == HBF_ST_READY) {
                    ready[u] = true; q[u] = queue_slot(geom, v.queue);
                    if (lng || ((uint64_t)v.s >> (kNwServeBits - 1)) || (v.xfer >> 30)) b_time |= 0x80000000u;
                    S[u] = (uint32_t)v.s; xo[u] = v.xfer | (v.op << 31);
                    if (counts) {
                        const uint32_t lo = (uint32_t)v.cb, hi = (uint32_t)((uint64_t)v.cb >> 32);
                        uint32_t *plo = v.op ? st_bp_lo : st_br_lo, *phi = v.op ? st_bp_hi : st_br_hi;
                        atomicAdd(v.op ? &st_np[v.die] : &st_nr[v.die], v.parts);
                        const uint32_t old = atomicAdd(&plo[v.die], lo), carry = hi + ((old + lo) < old ? 1u : 0u);
                        if (carry) atomicAdd(&phi[v.die], carry);
                    }
                    if (DEBT && tile_begin + i[u] < claim_limit) { S[u] += quantum_ns; if (counts) atomicAdd(&st_claims[v.die], 1u); }
                    M[u] = ri[u] + (v.op ? v.xfer : 0u) + S[u];
                } else if (v.st == HBF_ST_NATIVE) {
                    r.native += 1u;
                } else {
                    r.fault += 1u;
                }
            }
            // read disturb: the read's pages, on the block of its first page.  (`ready` does not ask for the issue time's limits; a
            // time beyond them sends the tile to the 64-bit form, which refuses the record but counts no disturb a second time)
            if (DEBT && !RESERVE && ready[u] && flags == 0u && ((uint64_t)issue[u] >> kIssueBits) == 0ull) {
                const uint32_t npages = (uint32_t)(((uint64_t)((uint32_t)off & geom.page_mask) + bytes + geom.page_mask) >> geom.page_shift);
                if (ret.pow2 != 0u) {
                    const uint32_t row = (uint32_t)((off >> geom.stripe_shift) >> ret_row_shift);
                    const uint32_t in_stripe = ((uint32_t)off & ((1u << geom.stripe_shift) - 1u)) >> geom.page_shift;
                    const uint32_t blk = ((row << mp_arg.pages_per_stripe_shift) + in_stripe) >> ret.ppb_shift;
                    const uint32_t pl = (uint32_t)(off >> (geom.stripe_shift + geom.chdie_shift)) & geom.plane_mask;
                    const uint32_t die = slot_die(geom, q[u]);
                    atomicAdd(&ret.disturb[((die << mp_arg.plane_shift) + pl) * ret.bpp + (blk & (ret.bpp - 1u))], npages);
                } else {
                    atomicAdd(&ret.disturb[ret_block_of(mp, ret, off)], npages);
                }
            }
            if ((PAGED || !RESERVE) && status_t && valid[u]) status_t[i[u]] = (uint8_t)st;
        }
        // ---- which lanes of a row hold the same queue (see the 64-bit form)
        uint8_t *tag_at[K];
        uint32_t tagged[K];
#pragma unroll
        for (int u = 0; u < K; ++u) { tag_at[u] = warp_tag + u * kInTagStride + (ready[u] ? q[u] : kInMaxQueues + (uint32_t)lane); *tag_at[u] = (uint8_t)lane; }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < K; ++u) tagged[u] = *reinterpret_cast<volatile uint8_t *>(tag_at[u]);
        if (MODE == kInFull && turn * (uint32_t)(K * 32) < qid_stride) {
#pragma unroll
            for (int u = 0; u < K; ++u)
                if (valid[u]) qid_t[i[u]] = ready[u] ? (uint16_t)slot_queue(geom, q[u]) : (uint16_t)kInMaxQueues;
        }
        const bool heads_on = MODE != kInFull ? false : *reinterpret_cast<volatile uint32_t *>(s_heads_full) < R;
        auto rest_of_turn = [&](auto heads_tag) {
        constexpr bool HEADS = decltype(heads_tag)::value;
        uint32_t rank1[K], pc[K], c0[K], c1[K], m_own[K], s_own[K], B[K];
        bool last[K];
        State *pq[K];
#pragma unroll
        for (int u = 0; u < K; ++u) {
            rank1[u] = 1u; last[u] = ready[u]; pc[u] = HEADS ? 1u : 0u;
            m_own[u] = M[u]; s_own[u] = S[u];
            const bool loser = tagged[u] != (uint32_t)lane;
            if (__any_sync(0xffffffffu, loser)) {
                if (loser) *tag_at[u] = (uint8_t)lane;
                __syncwarp();
                const uint32_t t2 = *reinterpret_cast<volatile uint8_t *>(tag_at[u]);
                if (!__any_sync(0xffffffffu, loser && t2 != (uint32_t)lane)) {
                    const uint32_t peer = loser ? tagged[u] : t2;                  // the lane itself when it has none
                    const bool second = peer < (uint32_t)lane;
                    const uint32_t mp_ = __shfl_sync(0xffffffffu, M[u], (int)peer), sp_ = __shfl_sync(0xffffffffu, S[u], (int)peer), gp_ = MODE == kInFull ? __shfl_sync(0xffffffffu, gn[u], (int)peer) : 0u;
                    if (second) { M[u] = max(mp_ + S[u], M[u]); S[u] += sp_; gn[u] += gp_; rank1[u] = 2u; }
                    if (peer > (uint32_t)lane) last[u] = false;
                    if (HEADS && peer != (uint32_t)lane) pc[u] = 2u;
                } else {
                    const unsigned peers = __match_any_sync(0xffffffffu, ready[u] ? q[u] : (0x10000u | (uint32_t)lane));
                    const unsigned le = peers & le_mask;
                    rank1[u] = (uint32_t)__popc(le);
                    last[u] = ready[u] && (peers >> lane) == 1u;
                    pc[u] = HEADS ? (uint32_t)__popc(peers) : 0u;
                    const unsigned before = le & ~(1u << lane);
                    int prev_l = before ? 31 - __clz((int)before) : -1;
                    const uint32_t n_max = __reduce_max_sync(0xffffffffu, rank1[u]);
                    for (uint32_t span = 1; span < n_max; span <<= 1) {
                        const int src = prev_l >= 0 ? prev_l : lane;
                        const uint32_t Se = __shfl_sync(0xffffffffu, S[u], src), Me = __shfl_sync(0xffffffffu, M[u], src), ge = MODE == kInFull ? __shfl_sync(0xffffffffu, gn[u], src) : 0u;
                        const int pe = __shfl_sync(0xffffffffu, prev_l, src);
                        if (prev_l >= 0) { M[u] = max(Me + S[u], M[u]); S[u] += Se; gn[u] += ge; prev_l = pe; }
                    }
                }
            }
            pq[u] = reinterpret_cast<State *>(qst) + q[u];
        }
        // ---- the queue updates, in row order
        if (turn > 0) row_wait_n(my_bar, M[0], S[0], pq[0], gn[0], last[0], M[K - 1], S[K - 1], pq[K - 1], gn[K - 1], last[K - 1]);
#pragma unroll
        for (int u = 0; u < K; ++u) {
            if (u > 0) __syncwarp();                         // (the row before may hold the same queues)
            const State state = *pq[u];
            if constexpr (RESERVE) {
                B[u] = max(state + S[u], M[u]);
                if (last[u]) *pq[u] = B[u];
            } else if constexpr (LIGHT) {
                B[u] = max(state.x + S[u], M[u]);
                if (last[u]) *pq[u] = make_uint2(B[u], state.y + S[u]);
            } else {
            B[u] = max(state.x + S[u], M[u]);
            uint32_t inc = 0u;
            if (HEADS) {
                c0[u] = min(state.w & 15u, head_depth);
                inc = min(pc[u], head_depth - c0[u]);
                c1[u] = c0[u] + inc;
            }
            if (last[u]) *pq[u] = make_uint4(B[u], state.y + S[u], state.z + (gn[u] & ((1u << kNwCountShift) - 1u)), state.w + ((gn[u] >> kNwCountShift) << 4) + inc);
            }
        }
        if (turn + 1 < turns) row_pass(next_bar);
        // ---- results
#pragma unroll
        for (int u = 0; u < K; ++u) {
            if (LIGHT) { if (ready[u]) b_time |= B[u]; }
            else if (valid[u]) {
                const uint32_t done = ready[u] ? B[u] + (uint32_t)max((int)xo[u], 0) : ri[u], waited = done - ri[u];
                if (ready[u]) { b_time |= B[u]; r.max_done = max(r.max_done, done); }
                r.stall += (long long)(unsigned long long)waited;
                if (HEADS && ready[u]) {
                    const uint32_t ci = c0[u] + rank1[u] - 1u;
                    if (ci < head_depth) {
                        InHead h; h.m = T0 + (int64_t)m_own[u]; h.s = (int64_t)s_own[u]; h.xo = xo[u]; h.idx = tile_begin + i[u];
                        in_head[head_slot(tile, R, slot_queue(geom, q[u]), ci)] = h;
                    }
                    if (last[u] && c1[u] != c0[u] && c1[u] == head_depth) atomicAdd(s_heads_full, 1u);
                }
                __stcs(reinterpret_cast<long long *>(completion_t + i[u]), (long long)(T0 + (int64_t)(uint64_t)done));
                __stcs(reinterpret_cast<long long *>(stall_t + i[u]), (long long)(unsigned long long)waited);
            }
        }
        };
        if constexpr (MODE == kInFull) { if (heads_on) rest_of_turn(std::true_type{}); else rest_of_turn(std::false_type{}); }
        else { (void)heads_on; rest_of_turn(std::false_type{}); }
      };
      if ((turn * K + K) * 32u <= tile_len) whole_turn(std::true_type{}); else whole_turn(std::false_type{});
    }
    r.unsorted = b_sort >> 31; r.over = (b_time >> 31) | b_hi;
    return r;
}

// DEBT = true (retention on): a modeled access with a batch index below the claim limit pays one refresh quantum (a page
// read and a page program, scaled like any service, Eq. 3) before its own service; the streaming pass counts the
// claims per die.
// PAGED = true: the page-granular submit of accesses that stay inside one stripe unit each (paged_terms).
// MODE: kInFull, kInAgain or kInLight (above).
template <int MODE, bool DEBT, bool PAGED>
__global__ void __launch_bounds__(kInThreads, kInBlocksPerSM)
k_inorder_serve(const hbf_access_t *__restrict__ acc, uint64_t n, const __grid_constant__ InTileMap tmap, const RangeSnap *__restrict__ ranges_g,
                const __grid_constant__ ModelParams mp_arg, const __grid_constant__ FastRange fast_arg, BatchCtrl *ctrl, uint8_t *__restrict__ status, int64_t *__restrict__ in_agg,
                hbf_die_stats_t *stats_stage, int64_t *__restrict__ completion, int64_t *__restrict__ stall,
                const int64_t *__restrict__ in_bin, InTile *in_tile, InHead *__restrict__ in_head, uint8_t *__restrict__ in_headcnt,
                const int64_t *__restrict__ busy, const unsigned long long *claim_limit_p, uint32_t *die_claims,
                const __grid_constant__ RetDev ret, uint16_t *__restrict__ in_qid, uint32_t qid_stride,
                TileBalance *bal, uint32_t bal_seq, const __grid_constant__ FastGeom geom, const uint32_t head_depth, const OrderedCopy copy, const int decided) {
    constexpr bool RESERVE = MODE == kInAgain, LOOK = MODE == kInLook, LIGHT = MODE == kInLight || LOOK;
    extern __shared__ __align__(16) unsigned char in_smem[];
    __shared__ long long s_red[2];
    __shared__ unsigned long long s_t0;                   // when this block took its tile (0: its time is not recorded)
    __shared__ uint32_t s_heads_full;                     // queues whose head entries are complete
    __shared__ ModelParams mp;                            // measured: reads from shared memory beat reads of the argument
    __shared__ FastRange fast_range;

    pdl_wait();
    pdl_trigger();
    if (ctrl->skip || ctrl->run_sort) return;             // (run_sort set this early: the batch went to the sort path at its start)
    if (LOOK && ctrl->sample_crossed) return;             // (the samples showed it: the records are cut first)
    if (!RESERVE && decided && (ctrl->twice != 0u) != LIGHT) return;      // (the batch's load has chosen the other of the two)
    if (RESERVE && decided && blockIdx.x == 0 && threadIdx.x == 0 && ctrl->inorder_used && !ctrl->twice && 2u * bal->strag_flagged >= tmap.n_tiles) {
        bal->twice_load = ctrl->load; bal->twice_left = kInTwiceRun;
    }
    if (RESERVE && (!ctrl->inorder_used || !in_tile[blockIdx.x].reserve)) return;
    const bool count = RESERVE && in_tile[blockIdx.x].reserve == 2u, counts = MODE == kInFull || count;
    if (ctrl->regrouped) { acc = copy.recs; completion = copy.comp; stall = copy.stall; status = nullptr; }   // (brought into order: regroup_kernels.cu)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const RangeSnap &rs = *ranges_g;                      // read through the cache; the common configuration does not touch it
    // (by one thread it is some ninety stores one after the other: 65,536 reads, two such passes, 45.5 -> 44.0 us, 1.5 M mixed accesses 99.2 -> 97.9,
    // 4 M decode reads 108.5 -> 107.4)
    static_assert(sizeof(ModelParams) % 4 == 0 && sizeof(ModelParams) / 4 <= kInThreads && sizeof(FastRange) % 4 == 0, "a word per thread");
    if (tid < (int)(sizeof(ModelParams) / 4)) reinterpret_cast<uint32_t *>(&mp)[tid] = reinterpret_cast<const uint32_t *>(&mp_arg)[tid];
    if (tid < (int)(sizeof(FastRange) / 4)) reinterpret_cast<uint32_t *>(&fast_range)[tid] = reinterpret_cast<const uint32_t *>(&fast_arg)[tid];
    if (DEBT && !RESERVE && tid == 0 && blockIdx.x == 0) ret.st->observed_inline = 1u;
    if (!RESERVE && bal && tid == 0 && blockIdx.x == 0) { bal->strag_seq = bal_seq; bal->strag_max = 0u; bal->strag_flagged = 0u; bal->strag_depth = LIGHT ? 0u : head_depth; }
    const uint32_t R = mp_arg.n_queues, n_dies = mp_arg.n_dies;
    const int64_t q_ppm = ctrl->q_ppm;
    const Div64 div_q = ctrl->div_q;
    // one range, power-of-two geometry, transfer table, no thermal scaling in force: the short form of the terms
    const bool fast_on = fast_geom_ok(fast_arg, mp_arg);
    const uint32_t ret_row_shift = mp_arg.ch_shift + mp_arg.die_shift + mp_arg.plane_shift;   // stripe unit -> row of stripe units on its plane
    const uint64_t claim_limit = DEBT ? *claim_limit_p : 0ull;
    const int64_t quantum_ns = !DEBT ? 0 : q_ppm == 1000000 ? mp_arg.t_read_ns + mp_arg.t_prog_ns
        : (int64_t)div64((uint64_t)(mp_arg.t_read_ns + mp_arg.t_prog_ns) * 1000000ull + (uint64_t)q_ppm - 1ull, div_q);

    // [queues] x: busy-until of the run in progress; y: service time served in this tile << 8 | head-table entries written
    longlong2 *qst = reinterpret_cast<longlong2 *>(in_smem);
    uint32_t *st_br_lo = reinterpret_cast<uint32_t *>(qst + kInMaxQueues), *st_br_hi = st_br_lo + n_dies;   // per die
    uint32_t *st_bp_lo = st_br_hi + n_dies, *st_bp_hi = st_bp_lo + n_dies;
    uint32_t *st_nr = st_bp_hi + n_dies, *st_np = st_nr + n_dies;
    uint32_t *st_claims = st_np + n_dies;                 // refresh quanta claimed on each die (claims variant)
    // per warp and row of a turn: a byte per queue (which lane of the row holds it) and one per lane
    uint8_t *warp_tag = reinterpret_cast<uint8_t *>(st_claims + n_dies) + (uint32_t)(threadIdx.x >> 5) * (kInRows * kInTagStride);

    // Which tile this block serves.  Two blocks share an SM, and the hardware favours the one in the lower warp slots: with
    // equal tiles it finishes about 12 % earlier (measured) and the pass lasts as long as the other one.  So the tiles come in
    // two sizes; a block reads off its warp slot which kind of block it is and takes the next tile of the matching size (or,
    // should one size run out, of the other: every tile is handed out exactly once whatever the slots say).
    __shared__ uint32_t s_tile_id;
    if (!RESERVE) {
        if (tid == 0) {
            uint32_t t = blockIdx.x;
            unsigned long long t0 = 0ull;
            if (tmap.n_big != 0u) {
                unsigned slot;
                asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
                const uint32_t late = slot >= 4u ? 1u : 0u;   // warp 0 of the block that came second sits past the first four slots
                if (bal) {
                    // the tile of this SM and this kind; should it be gone (the slots did not say what they usually say),
                    // any tile that is left: every tile is taken exactly once, marked with the batch's number
                    unsigned sm;
                    asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
                    const uint32_t want = late * tmap.n_big + sm;
                    bool mine = sm < tmap.n_big && atomicExch(&bal->claim[want], bal_seq) != bal_seq;
                    t = want;
                    for (uint32_t k = 0; !mine && k < tmap.n_tiles; ++k) { t = k; mine = atomicExch(&bal->claim[k], bal_seq) != bal_seq; }
                    if (t == want) asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
                } else {
                    const uint32_t have[2] = {tmap.n_big, tmap.n_tiles - tmap.n_big};
                    uint32_t k = atomicAdd(&ctrl->role_count[late], 1u);
                    if (k < have[late]) t = late ? tmap.n_big + k : k;
                    else { k = atomicAdd(&ctrl->role_count[1u - late], 1u); t = late ? k : tmap.n_big + k; }
                }
            }
            s_tile_id = t; s_t0 = t0;
        }
        __syncthreads();
    }
    const uint32_t tile = RESERVE ? blockIdx.x : s_tile_id;
    const uint64_t tile_begin = tile_first(tmap, tile);
    const uint64_t tile_end = tile_last(tmap, tile);

    const uint32_t tile_len = tile_end > tile_begin ? (uint32_t)(tile_end - tile_begin) : 0u;   // inside a tile everything is indexed by 32-bit offsets from its first record (a batch is below 2^30 records)
    const hbf_access_t *acc_t = acc + tile_begin;
    int64_t *completion_t = completion + tile_begin, *stall_t = stall + tile_begin;
    uint8_t *status_t = status ? status + tile_begin : nullptr;
    uint16_t *qid_t = in_qid + (uint64_t)tile * qid_stride;   // the straggle pass filters the head of the tile by these
    if (tid < 2) s_red[tid] = tid == 1 ? INT64_MIN : 0;
    if (tid == 0) s_heads_full = 0u;
    unsigned c_unsorted = (DEBT && ((uint64_t)quantum_ns >> 32)) ? 1u : 0u;   // (or a service, or a refresh quantum, of 2^32 ns or more)
    long long sum_stall = 0, max_c = INT64_MIN;
    long long t_native = 0, t_ready = 0, t_fault = 0;        // this thread's share of the tile's counts
    unsigned long long t_pages = 0; unsigned c_crossed = 0;  // kInLook: see BatchCtrl
    __shared__ uint32_t s_prog_pages; __shared__ unsigned long long s_work;
    if (LOOK && tid == 0) { s_prog_pages = 0u; s_work = 0ull; }
    bool narrow_done = false, again = false;
    {
        // The 32-bit form serves the tile when the configuration allows it, the tile's times lie within 2^31 ns and its read
        // granules sum below 2^32; should it turn out not to fit after all (a backlog), the 64-bit form below serves the tile again.
        int64_t T0 = 0, T1 = -1;
        if (tile_len) { T0 = ld_after(&acc_t[0].issue_ns); T1 = ld_after(&acc_t[tile_len - 1u].issue_ns); }
        if (geom.narrow != 0u && q_ppm == 1000000 && T0 >= 0 && T0 < HBF_ISSUE_LIMIT - (1ll << 32) && T1 >= T0 && T1 - T0 < (1ll << 31) &&
            (uint64_t)tile_len * geom.nw_gmax < (1ull << 32) && (uint64_t)quantum_ns < (1ull << (kNwServeBits - 1))) {
            uint4 *q4 = reinterpret_cast<uint4 *>(qst);
            unsigned over = 0;
            if (counts) for (uint32_t d = tid; d < n_dies * 7u; d += kInThreads) st_br_lo[d] = 0u;
            if (count) for (uint32_t d = tid; d < n_dies; d += kInThreads) reinterpret_cast<uint32_t *>(qst)[kInMaxQueues + d] = 0u;
            for (uint32_t q = tid; q < kInMaxQueues; q += kInThreads) {
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if ((RESERVE || (MODE == kInFull && tile == 0u)) && q < R) {   // the first tile knows its entering state: it is served exactly
                    const int64_t b = (RESERVE ? ld_after(in_bin + (uint64_t)tile * R + q) : busy[q]) - T0;
                    v.x = b > 0 ? (uint32_t)b : 0u;
                    if (b >= (RESERVE ? 1ll << 30 : 1ll << 31)) over = 1u;
                }
                const uint32_t at = q < R ? queue_slot(geom, q) : q;
                if (RESERVE) reinterpret_cast<uint32_t *>(qst)[at] = v.x; else if (LIGHT) reinterpret_cast<uint2 *>(qst)[at] = make_uint2(0u, 0u); else q4[at] = v;
            }
            // (a backlog that reaches far into the tile grows while the tile is served: not even tried then)
            const bool try_narrow = __syncthreads_or((int)over) == 0;
            NarrowSums nw{};
            if (try_narrow) nw = serve_narrow<MODE, DEBT, PAGED>(geom, mp, mp_arg, acc_t, (uint32_t)tile_begin, tile_len, T0, q4, warp_tag, status_t, qid_t, qid_stride,
                                                     completion_t, stall_t, in_head, tile, R, head_depth, &s_heads_full, st_br_lo, n_dies, claim_limit,
                                                     (uint32_t)quantum_ns, ret, ret_row_shift, count, &s_prog_pages);
            if (__syncthreads_or((int)(over | nw.over)) == 0) {
                narrow_done = true;
                sum_stall = nw.stall;
                if (nw.max_done) max_c = T0 + (int64_t)(uint64_t)nw.max_done;      // (a modeled access ends after its tile's first issue time)
                if constexpr (!RESERVE) {
                    c_unsorted |= nw.unsorted;
                    unsigned long long work = 0;
                    if (tid == 0 && tile_begin > 0 && ld_after(&acc_t[-1].issue_ns) > T0) c_unsorted = 1u;
                    t_native = nw.native; t_fault = nw.fault; t_ready = (tid == 0 ? (long long)tile_len : 0ll) - t_native - t_fault;
                    longlong2 *out = reinterpret_cast<longlong2 *>(in_agg) + (uint64_t)tile * R;
                    for (uint32_t q = tid; q < R; q += kInThreads) {
                        uint2 v;                             // busy-until, service time
                        if (LIGHT) v = reinterpret_cast<const uint2 *>(qst)[queue_slot(geom, q)];
                        else { const uint4 f = q4[queue_slot(geom, q)]; v = make_uint2(f.x, f.y); in_headcnt[(uint64_t)tile * R + q] = (uint8_t)(f.w & 15u); }
                        work += v.y;
                        out[q] = make_longlong2((long long)(uint64_t)v.y, v.y ? T0 + (int64_t)(uint64_t)v.x : kNegInf);   // (no service time: no access)
                    }
                    if (LOOK) {                              // the tile's pages follow from its service time
                        work = (unsigned long long)warp_sum((long long)work);
                        if (lane == 0) atomicAdd(&s_work, work);
                        __syncthreads();
                        if (tid == 0) t_pages = (s_work - (unsigned long long)s_prog_pages * geom.t_prog) / geom.t_read + s_prog_pages;
                        t_pages += (unsigned long long)t_native;
                    }
                    if (MODE == kInFull) for (uint32_t d = tid; d < n_dies; d += kInThreads) {              // a die's reads: the sums its queues carry
                        unsigned long long g = 0, cnt = 0;
                        for (uint32_t p = 0; p < geom.planes_q; ++p) { const uint4 v = q4[queue_slot(geom, d * geom.planes_q + p)]; g += v.z; cnt += v.w >> 4; }
                        unsigned long long *gd = reinterpret_cast<unsigned long long *>(stats_stage + d);
                        if (g) atomicAdd(&gd[1], g << geom.gran_shift_read);
                        if (cnt) atomicAdd(&gd[4], cnt);
                    }
                }
                if (count)
                    for (uint32_t d = tid; d < n_dies; d += kInThreads) {              // (d: channel, then die)
                        const uint32_t g = reinterpret_cast<const uint32_t *>(qst)[kInMaxQueues + d];
                        if (g) atomicAdd(reinterpret_cast<unsigned long long *>(stats_stage + slot_die(geom, d)) + 1, (unsigned long long)g << geom.gran_shift_read);
                    }
            } else {
                again = try_narrow;                          // (its read disturb is counted)
                if (tid == 0) s_heads_full = 0u;
            }
        }
    }
    if (!narrow_done) {
    using State = typename std::conditional<RESERVE, int64_t, longlong2>::type;   // (with known busy-until: that alone)
    if (counts) for (uint32_t d = tid; d < n_dies * 7u; d += kInThreads) st_br_lo[d] = 0u;
    if (RESERVE) {
        for (uint32_t q = tid; q < kInMaxQueues; q += kInThreads) reinterpret_cast<int64_t *>(qst)[q] = q < R ? ld_after(in_bin + (uint64_t)blockIdx.x * R + q) : kNegInf;
    } else {
        for (uint32_t i = tid; i < kInMaxQueues; i += kInThreads) qst[i] = make_longlong2(kNegInf, 0);
        if (MODE == kInFull && tile == 0u) {                 // the first tile knows its entering state: it is served exactly
            __syncthreads();
            for (uint32_t q = tid; q < R; q += kInThreads) qst[q].x = busy[q];
        }
    }
    uint32_t c_native = 0, c_ready = 0, c_valid = 0;         // per thread: far below 2^32 (a batch is below 2^30 records)
    __syncthreads();

    // A warp's turn covers kInRows consecutive rows: their arithmetic interleaves, and their queue updates
    // follow one another inside one wait/pass pair.
    constexpr int K = kInRows;
    const uint32_t rows = (tile_len + 31u) / 32u;
    const uint32_t turns = (rows + K - 1) / K;
    const unsigned le_mask = lanemask_lt() | (1u << lane);
    const int my_bar = 1 + warp, next_bar = 1 + (warp + 1 == kInWarps ? 0 : warp + 1);

    // the records of the warp's next turn are already on their way while this one is served
    uint64_t nx_addr[K], nx_issue[K], nx_bf[K];
    int64_t nx_prev[K];                                      // issue time of the record before the lane's own (same cache line, mostly)
#pragma unroll
    for (int u = 0; u < K; ++u) { nx_addr[u] = 0; nx_issue[u] = 0; nx_bf[u] = 0; nx_prev[u] = INT64_MIN; }
    const bool first_tile = tile_begin == 0;
    const bool pf_lane = lane < 24;
    const char *pf_base = reinterpret_cast<const char *>(acc_t) + lane * 32;
    auto fetch = [&](uint32_t turn) {
#pragma unroll
        for (int u = 0; u < K; ++u) {
            const uint32_t j = (turn * K + u) * 32u + (uint32_t)lane;
            if (j < tile_len) {
                const uint64_t *rec = reinterpret_cast<const uint64_t *>(acc_t + j);
                nx_addr[u] = __ldcs(rec); nx_issue[u] = __ldcs(rec + 1); nx_bf[u] = __ldcs(rec + 2);   // read once: streaming loads
                if (!RESERVE) nx_prev[u] = (j > 0u || !first_tile) ? (int64_t)ld_after(rec - 2) : INT64_MIN;
            }
        }
    };
    fetch((uint32_t)warp);

    // A turn whose rows are all complete (every turn but the last of a batch whose size is not a multiple of 32) runs
    // a copy of the code that has no bounds tests.
    for (uint32_t turn = (uint32_t)warp; turn < turns; turn += kInWarps) {
      auto whole_turn = [&](auto full_tag) {
        constexpr bool FULL = decltype(full_tag)::value;
        uint32_t i[K];                                       // offsets from the tile's first record
        bool valid[K], ready[K], last[K];
        int64_t issue[K], a[K], S[K], M[K], B[K];
        Served v[K];
        uint32_t rank1[K], pc[K], c0[K], c1[K], qi[K];
        State *pq[K];
        int64_t prev[K];
        uint64_t addr[K], bf[K];
#pragma unroll
        for (int u = 0; u < K; ++u) {
            i[u] = (turn * K + u) * 32u + (uint32_t)lane;
            valid[u] = FULL || i[u] < tile_len;
            addr[u] = nx_addr[u]; bf[u] = nx_bf[u]; issue[u] = (int64_t)nx_issue[u]; prev[u] = nx_prev[u];
        }
        fetch(turn + kInWarps);
        {                                                    // and the turn after that is called into the L2
            const uint32_t first = (turn + kInPrefetchTurns * kInWarps) * (uint32_t)(K * 32);
            if (pf_lane && first + K * 32 <= tile_len) {     // 24 lanes cover a row's 768 bytes in 32-byte sectors
                const char *p = pf_base + (size_t)first * sizeof(hbf_access_t);
#pragma unroll
                for (int u = 0; u < K; ++u) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + u * 768));
            }
        }
        // ---- terms ---------------------------------------------------------------------------------------
#pragma unroll
        for (int u = 0; u < K; ++u) {
            v[u].st = HBF_ST_NATIVE; v[u].queue = 0; v[u].die = 0; v[u].op = 0; v[u].s = 0; v[u].xfer = 0; v[u].cb = 0; v[u].parts = 1;
            if (valid[u])
                v[u] = fast_on ? serve_terms_geom(geom, mp, addr[u], issue[u], bf[u], q_ppm, div_q, c_unsorted, DEBT ? 32 : 33)
                                 : serve_terms(rs, mp, addr[u], issue[u], bf[u], q_ppm, div_q, c_unsorted, DEBT ? 32 : 33);
            ready[u] = valid[u] && v[u].st == HBF_ST_READY;
            if (PAGED && ready[u]) {
                const uint64_t off = media_offset_of(rs, fast_range, fast_on, addr[u], issue[u], bf[u]), unit = 1ull << mp.stripe_shift;
                paged_terms(mp, off, (uint32_t)bf[u], q_ppm, div_q, c_unsorted, 33, v[u]);
                if (LOOK && (off & (unit - 1ull)) + (uint32_t)bf[u] > unit) c_crossed = 1u;
            }
            if (LOOK && valid[u]) t_pages += v[u].parts;
            if (DEBT && ready[u] && tile_begin + i[u] < claim_limit) {
                v[u].s += quantum_ns;
                if (counts) atomicAdd(&st_claims[v[u].die], 1u);
            }
            if (DEBT && !RESERVE && ready[u] && !v[u].op && !again) {  // read disturb (counted already when the tile is served again): the read's pages, on the block of its first page
                if (fast_on && ret.pow2 != 0u) {
                    // one range, powers of two all the way down: the block from shifts and masks (the general form below
                    // divides twice; it took the pass from 2.0 to 2.9 ms)
                    const uint64_t off = geom.media_offset + (addr[u] - geom.base);
                    const uint32_t npages = (uint32_t)(((uint64_t)((uint32_t)off & geom.page_mask) + (uint32_t)bf[u] + geom.page_mask) >> geom.page_shift);
                    const uint32_t row = (uint32_t)((off >> geom.stripe_shift) >> ret_row_shift);     // (the wrap of the general form too: the block inside the plane)
                    const uint32_t in_stripe = ((uint32_t)off & ((1u << geom.stripe_shift) - 1u)) >> geom.page_shift;
                    const uint32_t blk = ((row << mp_arg.pages_per_stripe_shift) + in_stripe) >> ret.ppb_shift;
                    const uint32_t pl = (uint32_t)(off >> (geom.stripe_shift + geom.chdie_shift)) & geom.plane_mask;
                    atomicAdd(&ret.disturb[((v[u].die << mp_arg.plane_shift) + pl) * ret.bpp + (blk & (ret.bpp - 1u))], npages);
                } else {
                    const uint64_t off = media_offset_of(rs, fast_range, fast_on, addr[u], issue[u], bf[u]);
                    const uint32_t page_mask = (1u << mp.page_shift) - 1u;
                    const uint32_t npages = (uint32_t)(((uint64_t)((uint32_t)off & page_mask) + (uint32_t)bf[u] + page_mask) >> mp.page_shift);
                    atomicAdd(&ret.disturb[ret_block_of(mp, ret, off)], npages);
                }
            }
        }
        // ---- which lanes of a row hold the same queue: every lane writes its number where its queue's entry is in the
        // warp's own table and reads the entry back (the answer is needed only further down: the latency is covered).
        // Nothing is ever cleared: a lane reads what a lane of this row wrote.  Accesses that are not modeled have an
        // entry per lane.  (`match_any` for every row kept the unit that executes it busy three quarters of the time.)
        uint8_t *tag_at[K];
        uint32_t tagged[K];
#pragma unroll
        for (int u = 0; u < K; ++u) { tag_at[u] = warp_tag + u * kInTagStride + (ready[u] ? v[u].queue : kInMaxQueues + (uint32_t)lane); *tag_at[u] = (uint8_t)lane; }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < K; ++u) tagged[u] = *reinterpret_cast<volatile uint8_t *>(tag_at[u]);
        if (MODE == kInFull && turn * (uint32_t)(K * 32) < qid_stride) {   // (the stride is a multiple of a turn's records)
#pragma unroll
            for (int u = 0; u < K; ++u)
                if (valid[u]) qid_t[i[u]] = ready[u] ? (uint16_t)v[u].queue : (uint16_t)kInMaxQueues;   // (one past the last queue: not modeled)
        }
        if (!RESERVE || counts || (PAGED && status_t)) {
#pragma unroll
            for (int u = 0; u < K; ++u) {
                if (valid[u]) {
                    if ((PAGED || !RESERVE) && status_t) status_t[i[u]] = (uint8_t)v[u].st;
                    if (!RESERVE) {
                        c_unsorted |= issue[u] < prev[u] ? 1u : 0u;
                        c_valid += 1u;
                        c_ready += ready[u] ? 1u : 0u;
                        c_native += v[u].st == HBF_ST_NATIVE ? 1u : 0u;
                    }
                    if (counts && ready[u]) {
                        // charged bytes < 2^33: add the low word, carry into the high word when it wraps (a form that counts
                        // granules in one word and sends oversized accesses to the 64-bit totals measured slower)
                        const uint32_t lo = (uint32_t)v[u].cb, hi = (uint32_t)((uint64_t)v[u].cb >> 32);
                        uint32_t *plo = v[u].op ? st_bp_lo : st_br_lo, *phi = v[u].op ? st_bp_hi : st_br_hi;
                        atomicAdd(v[u].op ? &st_np[v[u].die] : &st_nr[v[u].die], PAGED ? v[u].parts : 1u);
                        const uint32_t old = atomicAdd(&plo[v[u].die], lo);
                        const uint32_t carry = hi + ((old + lo) < old ? 1u : 0u);
                        if (carry) atomicAdd(&phi[v[u].die], carry);
                    }
                }
            }
        }
        // The rest of the turn exists twice: with the head-table bookkeeping, and without it once every queue of the
        // tile has its head entries (after a few percent of a large tile).  The flag is the same for the whole warp.
        const bool heads_on = MODE == kInFull && *reinterpret_cast<volatile uint32_t *>(&s_heads_full) < R;
        auto rest_of_turn = [&](auto heads_tag) {
        constexpr bool HEADS = decltype(heads_tag)::value;
        // ---- per row: the accesses of a lane's queue, up to the lane's own, as one map B -> max(B + S, M), composed
        // in lane order, so that the ordered part below is one application of it whatever the row holds
#pragma unroll
        for (int u = 0; u < K; ++u) {
            a[u] = issue[u] + (int64_t)(v[u].op ? v[u].xfer : 0u);   // arrival at the queue: a program's data is transferred first
            rank1[u] = 1u;                                  // this access is the rank1-th of its queue in the row
            last[u] = ready[u];                             // no later access of this queue in the row
            pc[u] = HEADS ? 1u : 0u;                        // accesses of this queue in the row
            S[u] = v[u].s; M[u] = a[u] + v[u].s;
            // A lane that did not read its own number back shares its queue with another lane of the row: one row in five.
            const bool loser = tagged[u] != (uint32_t)lane;
            if (__any_sync(0xffffffffu, loser)) {
                // Second round: the lanes that lost write again.  In a pair the winner now reads its peer's number and the
                // loser its own; a loser that loses again has two peers or more, and only then is the row matched in full.
                if (loser) *tag_at[u] = (uint8_t)lane;
                __syncwarp();
                const uint32_t t2 = *reinterpret_cast<volatile uint8_t *>(tag_at[u]);
                if (!__any_sync(0xffffffffu, loser && t2 != (uint32_t)lane)) {
                    // pairs only (nearly always): the second lane of a pair composes its peer's map with its own
                    const uint32_t peer = loser ? tagged[u] : t2;                  // the lane itself when it has none
                    const bool second = peer < (uint32_t)lane;
                    const int64_t mp_ = __shfl_sync(0xffffffffu, M[u], (int)peer), sp_ = __shfl_sync(0xffffffffu, (int64_t)v[u].s, (int)peer);
                    if (second) { M[u] = max(mp_, a[u]) + v[u].s; S[u] = sp_ + v[u].s; rank1[u] = 2u; }
                    if (peer > (uint32_t)lane) last[u] = false;
                    if (HEADS && peer != (uint32_t)lane) pc[u] = 2u;
                } else {
                    const unsigned peers = __match_any_sync(0xffffffffu, ready[u] ? v[u].queue : (0x10000u | (uint32_t)lane));
                    const unsigned le = peers & le_mask;
                    rank1[u] = (uint32_t)__popc(le);
                    last[u] = ready[u] && (peers >> lane) == 1u;
                    pc[u] = HEADS ? (uint32_t)__popc(peers) : 0u;
                    // Every lane composes the maps of the lanes of its queue up to its own by doubling: it holds the map of a
                    // stretch of them that ends with itself and the lane before that stretch, takes that lane's stretch in front
                    // of its own, and goes on from the lane before that one; ceil(log2(most lanes on one queue)) rounds.
                    // (One lane after the other took as many rounds as lanes: 12.7 warp instructions per part where the parts
                    // of a split access, neighbours on one queue, fill the rows, against 9 per access unsplit.)
                    const unsigned before = le & ~(1u << lane);
                    int prev = before ? 31 - __clz((int)before) : -1;
                    const uint32_t n_max = __reduce_max_sync(0xffffffffu, rank1[u]);
                    for (uint32_t span = 1; span < n_max; span <<= 1) {
                        const int src = prev >= 0 ? prev : lane;
                        const int64_t Se = __shfl_sync(0xffffffffu, S[u], src), Me = __shfl_sync(0xffffffffu, M[u], src);
                        const int pe = __shfl_sync(0xffffffffu, prev, src);
                        if (prev >= 0) { M[u] = max((int64_t)(Me + S[u]), M[u]); S[u] = Se + S[u]; prev = pe; }
                    }
                }
            }
            qi[u] = ready[u] ? v[u].queue : 0u;
            pq[u] = reinterpret_cast<State *>(qst) + qi[u];
        }
        // ---- the queue updates, in row order: everything they need is in registers before the wait ---------------
        if (turn > 0) row_wait2(my_bar, M[0], S[0], pq[0], pc[0], last[0], M[K - 1], S[K - 1], pq[K - 1], pc[K - 1], last[K - 1]);
#pragma unroll
        for (int u = 0; u < K; ++u) {
            if (u > 0) __syncwarp();                         // (the row before may hold the same queues)
            const State state = *pq[u];
            if constexpr (RESERVE) {
                B[u] = max((int64_t)(state + S[u]), M[u]);
                if (last[u]) *pq[u] = B[u];
            } else {
            B[u] = max((int64_t)(state.x + S[u]), M[u]);
            uint32_t inc = 0u;
            if (HEADS) {
                c0[u] = min((uint32_t)state.y & 0xffu, head_depth);
                inc = min(pc[u], head_depth - c0[u]);
                c1[u] = c0[u] + inc;
            }
            if (last[u]) *pq[u] = make_longlong2(B[u], state.y + (S[u] << 8) + (long long)inc);
            }
        }
        if (turn + 1 < turns) row_pass(next_bar);
        // ---- results ---------------------------------------------------------------------------------------
#pragma unroll
        for (int u = 0; u < K; ++u) {
            if (!LIGHT && valid[u]) {
                const int64_t done = ready[u] ? B[u] + (int64_t)(v[u].op ? 0u : v[u].xfer) : issue[u];   // a read's data is transferred after its service;
                const int64_t st = done - issue[u];                                                    // not modeled: completion = issue, no stall
                sum_stall += st; max_c = max(max_c, ready[u] ? (long long)done : (long long)INT64_MIN);
                if (HEADS && ready[u]) {
                    const uint32_t ci = c0[u] + rank1[u] - 1u;
                    if (ci < head_depth) {
                        InHead h; h.m = a[u] + v[u].s; h.s = v[u].s; h.xo = v[u].xfer | (v[u].op << 31); h.idx = (uint32_t)tile_begin + i[u];
                        in_head[head_slot(tile, R, qi[u], ci)] = h;
                    }
                    if (last[u] && c1[u] != c0[u] && c1[u] == head_depth) atomicAdd(&s_heads_full, 1u);
                }
                // results are written once and not read again by this pass: streaming stores
                __stcs(reinterpret_cast<long long *>(completion_t + i[u]), (long long)done);
                __stcs(reinterpret_cast<long long *>(stall_t + i[u]), (long long)st);
            }
        }
        };
        if (heads_on) rest_of_turn(std::true_type{}); else rest_of_turn(std::false_type{});
      };
      if ((turn * K + K) * 32u <= tile_len) whole_turn(std::true_type{}); else whole_turn(std::false_type{});
    }

    t_native = c_native; t_ready = c_ready; t_fault = (long long)c_valid - c_ready - c_native;     // every other status is a fault
    __syncthreads();
    if (!RESERVE) {
        longlong2 *out = reinterpret_cast<longlong2 *>(in_agg) + (uint64_t)tile * R;
        for (uint32_t q = tid; q < R; q += kInThreads) {
            const longlong2 v = qst[q];
            out[q] = make_longlong2(v.y >> 8, v.x);
            if (!LIGHT) in_headcnt[(uint64_t)tile * R + q] = (uint8_t)(v.y & 0xff);
        }
    }
    }                                                        // (the 64-bit form)
    if (counts) {
        for (uint32_t d = tid; d < n_dies; d += kInThreads) {
            unsigned long long *g = reinterpret_cast<unsigned long long *>(stats_stage + d);
            const unsigned long long br = ((unsigned long long)st_br_hi[d] << 32) | st_br_lo[d];
            const unsigned long long bp = ((unsigned long long)st_bp_hi[d] << 32) | st_bp_lo[d];
            if (br) atomicAdd(&g[1], br);
            if (bp) atomicAdd(&g[2], bp);
            if (st_nr[d]) atomicAdd(&g[4], (unsigned long long)st_nr[d]);
            if (st_np[d]) atomicAdd(&g[5], (unsigned long long)st_np[d]);
            if (DEBT && st_claims[d]) atomicAdd(&die_claims[d], st_claims[d]);
        }
    }
    if (!RESERVE) {
        const unsigned long long w_native = (unsigned long long)warp_sum(t_native);
        const unsigned long long w_ready = (unsigned long long)warp_sum(t_ready);        // (a warp's share may be negative: the sum over the tile counts)
        const unsigned long long w_fault = (unsigned long long)warp_sum(t_fault);
        c_unsorted = __any_sync(0xffffffffu, c_unsorted);
        if (LOOK) {
            const unsigned long long w_pages = (unsigned long long)warp_sum((long long)t_pages);
            const bool crossed = __any_sync(0xffffffffu, c_crossed != 0u);
            if (lane == 0) { if (w_pages) atomicAdd(&ctrl->pages, w_pages); if (crossed) ctrl->crossed = 1u; }
        }
        if (lane == 0) {
            if (w_native) atomicAdd(&ctrl->n_native, w_native);
            if (w_ready) atomicAdd(&ctrl->n_ready, w_ready);
            if (w_fault) atomicAdd(&ctrl->n_fault, w_fault);
            if (c_unsorted) atomicOr(&ctrl->unsorted, 1u);
        }
    }
    sum_stall = warp_sum(sum_stall); max_c = warp_max(max_c);
    if (lane == 0) { atomicAdd((unsigned long long *)&s_red[0], (unsigned long long)sum_stall); atomicMax(&s_red[1], max_c); }
    __syncthreads();
    if (tid == 0) {
        if (RESERVE) in_tile[tile].true_sum = s_red[0];
        else { InTile t; t.spec_sum = s_red[0]; t.fix_delta = 0; t.true_sum = 0; t.reserve = LIGHT ? 2u : 0u; t.stragglers = 0u; in_tile[tile] = t; }
        if (s_red[1] != INT64_MIN) atomicMax(&ctrl->max_completion_ns, s_red[1]);
        if (!RESERVE && bal) {                               // how many records, how long: what the next batches' tile sizes follow from
            unsigned long long now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            bal->len[tile] = tile_len;
            bal->ns[tile] = s_t0 ? (uint32_t)min(now - s_t0, 0xffffffffull) : 0u;
        }
    }
}

// ======================================================================================================
// scan over tiles; also decides what happens to the batch.
// A block takes kInScanQueues consecutive queues (threadIdx.x) and cuts the tiles into kInScanChunks runs of
// consecutive tiles (threadIdx.y).  Every thread composes the aggregates (S, M) of its run, the runs' maps are
// composed in order through shared memory, and the thread walks its run again from the true busy-until entering
// it, which it stores for every tile.  The kInScanQueues lanes of a run read consecutive 16-byte aggregates:
// whole 128-byte lines.  A few tiles per thread and all blocks resident at once: no long chain of loads.
// ======================================================================================================
constexpr int kInScanChunks = 64;
constexpr int kInScanQueues = 8;

__global__ void __launch_bounds__(kInScanQueues * kInScanChunks)
k_inorder_scan(BatchCtrl *ctrl, const ModelParams *__restrict__ mp, uint32_t n_tiles, const int64_t *__restrict__ in_agg,
               int64_t *__restrict__ in_bin, const int64_t *__restrict__ busy, int64_t *__restrict__ busy_stage,
               hbf_die_stats_t *stats_stage, int forced) {
    __shared__ longlong2 s_map[kInScanChunks][kInScanQueues];
    pdl_wait();
    pdl_trigger();
    if (ctrl->skip || ctrl->run_sort) return;
    const bool fault = ctrl->n_fault != 0, unsorted = ctrl->unsorted != 0u;   // settled by the serve pass: every thread sees the same
    if (blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0) {
        if (fault) { ctrl->code = HBF_E_ACCESS_FAULT; ctrl->skip = 1; }                 // fail closed: refuse the batch
        else if (unsorted && forced) { ctrl->code = HBF_E_INVAL; ctrl->skip = 1; }
        else if (unsorted) ctrl->run_sort = 1u;                                         // hand the batch to the sort path
        else ctrl->inorder_used = 1u;
    }
    if (fault || unsorted) return;
    const uint32_t R = mp->n_queues;
    const uint32_t r = blockIdx.x * (uint32_t)kInScanQueues + threadIdx.x, chunk = threadIdx.y;
    const uint32_t per = (n_tiles + kInScanChunks - 1) / kInScanChunks;
    const uint32_t t_lo = min(n_tiles, chunk * per), t_hi = min(n_tiles, t_lo + per);
    const bool live = r < R;
    const longlong2 *agg = reinterpret_cast<const longlong2 *>(in_agg) + r;
    long long S = 0, M = kNegInf;                            // the run's own map
    if (live) {
        for (uint32_t t = t_lo; t < t_hi; ++t) {
            const longlong2 v = ld_after(agg + (uint64_t)t * R);
            M = max((int64_t)(M + v.x), (int64_t)v.y); S += v.x;
        }
    }
    s_map[chunk][threadIdx.x] = make_longlong2(S, M);
    __syncthreads();
    long long tot = 0;
    if (live) {
        // busy-until entering the run: the state earlier batches left, through the maps of the runs before it
        int64_t B = busy[r];
        for (uint32_t c = 0; c < chunk; ++c) { const longlong2 v = s_map[c][threadIdx.x]; B = max((int64_t)(B + v.x), (int64_t)v.y); }
        for (uint32_t t = t_lo; t < t_hi; ++t) {
            const longlong2 v = ld_after(agg + (uint64_t)t * R);
            in_bin[(uint64_t)t * R + r] = B;
            B = max((int64_t)(B + v.x), (int64_t)v.y);
        }
        if (chunk == kInScanChunks - 1) {                    // the last run ends at the batch's end (empty runs pass B through)
            busy_stage[r] = B;
            for (uint32_t c = 0; c < (uint32_t)kInScanChunks; ++c) tot += s_map[c][threadIdx.x].x;
            const uint32_t die = mp->queue_level == 0u ? r / mp->planes : r;
            if (tot) atomicAdd(reinterpret_cast<unsigned long long *>(&stats_stage[die].busy_ns), (unsigned long long)tot);
        }
    }
    tot = warp_sum(tot);                                     // (only the last run's threads carry a total)
    if (((threadIdx.y * kInScanQueues + threadIdx.x) & 31u) == 0u && tot)
        atomicAdd((unsigned long long *)&ctrl->service_ns, (unsigned long long)tot);
}

// Queue of an access of the common configuration (one range, power-of-two geometry), or ~0 when the address
// lies outside the range.  In a batch that was not refused every access inside the range is modeled.
__device__ __forceinline__ uint32_t fast_queue(const FastRange &f, const ModelParams &mp, uint64_t addr) {
    const uint64_t rel = addr - f.base;
    if (rel >= f.length) return 0xffffffffu;
    const uint32_t u = (uint32_t)((f.media_offset + rel) >> mp.stripe_shift);
    const uint32_t ch = u & (mp.channels - 1u), di = (u >> mp.ch_shift) & (mp.dies - 1u);
    const uint32_t pl = (u >> (mp.ch_shift + mp.die_shift)) & (mp.planes - 1u);
    const uint32_t die = ch * mp.dies + di;
    return mp.queue_level == 0u ? die * mp.planes + pl : die;
}

// ======================================================================================================
// fix-up and straggle: one block per tile.
// Fix-up.  The true run differs from the as-if-idle run only at the head of each (tile, queue): a thread starts
// from the true entering busy-until of its queues and re-serves the head table's accesses in order, until it meets
// one that arrives on an idle queue; from there on the as-if run was right.  The head entries of a (tile, queue) are
// contiguous, so they are fetched in two rounds (the first two, which settle nearly every queue, then the rest at
// once) instead of one dependent load per entry.  A queue still backlogged after kInHead accesses is a straggler;
// a tile with many of them (the batch arrived on queues that were far behind) is flagged to be served again whole.
// Straggle.  The block streams the head of the tile again, keeps the modeled records of the straggling queues in
// batch order and re-serves them a chunk at a time, carrying both the true run (from the true entering
// busy-until) and the as-if-idle run (to know what the serve pass wrote).  A queue is done when the two runs meet:
// from there on the serve pass was right.  The block stops at the chunk in which its last queue is done.
// What it streams: for the first kInQidPrefix records of every tile the serve pass left the queue of each record
// as a 16-bit number (kInMaxQueues: not modeled), so the filter reads 2 bytes per record, 32 records per thread and turn;
// past that prefix (queues that stay backlogged for very long) it decodes the queue from the records.
// ======================================================================================================
// The general form of the terms (several ranges, any geometry, thermal scaling), kept out of line here: this kernel runs
// nearly straight through once per block, so what it costs is fetching its instructions, and the common configuration
// never takes this path.
template <bool PAGED>
__device__ __noinline__ Served serve_terms_general(const RangeSnap &rs, const ModelParams &mp, uint64_t addr, int64_t issue, uint64_t bf,
                                                   int64_t q_ppm, Div64 div_q) {
    unsigned ignored = 0;                                    // (the serve pass has already vetted every service time)
    Served r = serve_terms(rs, mp, addr, issue, bf, q_ppm, div_q, ignored, 33);
    if (PAGED && r.st == HBF_ST_READY) paged_terms(mp, media_offset_of(rs, FastRange{}, false, addr, issue, bf), (uint32_t)bf, q_ppm, div_q, ignored, 33, r);
    return r;
}

struct FixRun { int64_t B, Bs; long long dstall, max_c; bool settled; };
__device__ __forceinline__ void fix_entry(FixRun &f, const InHead &h, int64_t *completion, int64_t *stall) {
    if (f.settled) return;
    if (f.B <= h.m - h.s) { f.settled = true; return; }      // idle on arrival: from here on the as-if run was right
    f.B += h.s;                                              // it waited for the queue: starts at B
    f.Bs = max(f.Bs + h.s, h.m);
    const bool op = (h.xo >> 31) != 0u;
    const int64_t xfer = (int64_t)(h.xo & 0x7fffffffu);
    const int64_t done = f.B + (op ? 0 : xfer);
    f.dstall += f.B - f.Bs;                                  // completion moved from Bs + post to B + post
    completion[h.idx] = done; stall[h.idx] = done - (h.m - h.s - (op ? xfer : 0));
    f.max_c = max(f.max_c, (long long)done);
}

constexpr int kInStrThreads = 512;
constexpr int kInStrWarps = kInStrThreads / 32;
constexpr int kInStrQItems = 32;                          // records per thread and turn inside the queue-number prefix
constexpr int kInStrQChunk = kInStrThreads * kInStrQItems;
constexpr int kInStrKeep = 1024;                          // kept records served at a time (a chunk with more is served in windows)
constexpr int kInStrMaxStragglers = 255;                   // a tile with as many is served again whole instead (a queue's place, plus one, is a byte)
constexpr int kInStrList = 32;                            // records of one queue in a window that its list holds (more: the window is scanned)
constexpr int kInStrQueuesPerThread = (kInMaxQueues + kInStrThreads - 1) / kInStrThreads;
static_assert(kInStrQChunk <= 65536, "a kept record's position in its chunk is stored in 16 bits");
static_assert(kInQidPrefix % kInStrQChunk == 0 && kInStrQItems == 32, "a thread's 32 queue numbers are four 16-byte loads");

template <bool DEBT, bool PAGED>
__global__ void __launch_bounds__(kInStrThreads, 2)
k_inorder_fixstraggle(const hbf_access_t *__restrict__ acc, uint64_t n, const __grid_constant__ InTileMap tmap,
                      const RangeSnap *__restrict__ ranges_g, const __grid_constant__ ModelParams mp_arg,
                      const __grid_constant__ FastRange fast_arg, BatchCtrl *ctrl,
                      const int64_t *__restrict__ in_bin, const InHead *__restrict__ in_head,
                      const uint8_t *__restrict__ in_headcnt, int64_t *completion, int64_t *stall, InTile *in_tile,
                      const unsigned long long *claim_limit_p, const uint16_t *__restrict__ in_qid, uint32_t qid_stride,
                      const uint32_t head_depth, TileBalance *bal, const OrderedCopy copy) {
    extern __shared__ __align__(16) unsigned char str_smem[];
    __shared__ ModelParams mp;
    __shared__ FastRange fast_range;
    __shared__ uint32_t s_cells[kInStrWarps];
    __shared__ uint32_t s_total;
    __shared__ uint32_t s_stragglers;                        // straggling queues of the tile
    __shared__ int s_open;                                   // those whose two runs have not met yet
    __shared__ long long s_red[2];

    pdl_wait();
    pdl_trigger();
    if (ctrl->skip || ctrl->run_sort || !ctrl->inorder_used || ctrl->twice) return;
    if (ctrl->regrouped) { acc = copy.recs; completion = copy.comp; stall = copy.stall; }
    const uint32_t tile = blockIdx.x;
    if (tile == 0u) return;                                  // the first tile was served from its true entering state
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const RangeSnap &rs = *ranges_g;
    const uint32_t R = mp_arg.n_queues;
    int64_t *Bt = reinterpret_cast<int64_t *>(str_smem);                       // [queues] true run
    int64_t *Ba = Bt + kInMaxQueues;                                           // [queues] as-if-idle run
    longlong2 *ent_as = reinterpret_cast<longlong2 *>(Ba + kInMaxQueues);      // [keep] kept records, batch order: issue time, service time
    uint2 *ent_pq = reinterpret_cast<uint2 *>(ent_as + kInStrKeep);            //        transfer | op << 31, queue | position << 16
    uint16_t *oq = reinterpret_cast<uint16_t *>(ent_pq + kInStrKeep);          // [stragglers] their queues
    uint8_t *open = reinterpret_cast<uint8_t *>(oq + kInMaxQueues);            // [2 x queues] 0, or 1 + the queue's place in oq while its runs have not met
    uint16_t *lst = reinterpret_cast<uint16_t *>(open + 2 * kInMaxQueues);     // [stragglers][kInStrList] the window's records of each queue
    uint32_t *lcount = reinterpret_cast<uint32_t *>(lst + kInStrMaxStragglers * kInStrList);   // [stragglers] how many
    __shared__ uint32_t s_overflow;
    if (tid < kInStrMaxStragglers) lcount[tid] = 0u;
    if (tid < (int)(sizeof(ModelParams) / 4)) reinterpret_cast<uint32_t *>(&mp)[tid] = reinterpret_cast<const uint32_t *>(&mp_arg)[tid];   // (as in the serve pass; 200 M capacity records 1,675 -> 1,665 us)
    if (tid < (int)(sizeof(FastRange) / 4)) reinterpret_cast<uint32_t *>(&fast_range)[tid] = reinterpret_cast<const uint32_t *>(&fast_arg)[tid];
    if (tid == 0) { s_stragglers = 0u; s_total = 0u; s_overflow = 0u; s_red[0] = 0; s_red[1] = INT64_MIN; }
    __syncthreads();

    // ---- fix-up, first entry: this thread's queues of the tile, their loads issued side by side.  Four queues in five
    // are idle when their first access of the tile arrives: they are done here.  The others go on a list.
    long long dstall = 0, max_c = INT64_MIN;
    uint16_t *deep = reinterpret_cast<uint16_t *>(ent_pq);   // [queues] the list (the record windows are not in use yet)
    {
        uint32_t c[kInStrQueuesPerThread]; int64_t Bin[kInStrQueuesPerThread];
        InHead e0[kInStrQueuesPerThread];
#pragma unroll
        for (int k = 0; k < kInStrQueuesPerThread; ++k) {
            const uint32_t q = (uint32_t)(k * kInStrThreads + tid);
            c[k] = 0u; Bin[k] = kNegInf;
            if (q < R) { c[k] = in_headcnt[(uint64_t)tile * R + q]; Bin[k] = ld_after(in_bin + (uint64_t)tile * R + q); }
        }
#pragma unroll
        for (int k = 0; k < kInStrQueuesPerThread; ++k)
            if (c[k] > 0u) e0[k] = in_head[head_slot(tile, R, (uint32_t)(k * kInStrThreads + tid), 0u)];
#pragma unroll
        for (int k = 0; k < kInStrQueuesPerThread; ++k) {
            const uint32_t q = (uint32_t)(k * kInStrThreads + tid);
            if (q < kInMaxQueues) { open[q] = 0; open[kInMaxQueues + q] = 0; Ba[q] = kNegInf; Bt[q] = Bin[k]; }   // (upper half: not modeled, or not defined)
            if (c[k] == 0u) continue;
            if (Bin[k] <= e0[k].m - e0[k].s) continue;       // idle on arrival: the as-if run was right from the start
            deep[atomicAdd(&s_total, 1u)] = (uint16_t)q;
        }
    }
    __syncthreads();
    // ---- fix-up, the rest: one thread per listed queue walks its head entries (fetched in two rounds) from the true
    // entering busy-until until an access arrives on an idle queue
    {
        const uint32_t n_deep = s_total;
        for (uint32_t d = (uint32_t)tid; d < n_deep; d += kInStrThreads) {
            const uint32_t q = deep[d];
            const uint64_t idx = (uint64_t)tile * R + q;
            const uint32_t c = in_headcnt[idx];
            const InHead *h = in_head + head_slot(tile, R, q, 1u) - 1;       // h[j], j >= 1: the queue's later entries, side by side
            FixRun f; f.B = Bt[q]; f.Bs = kNegInf; f.dstall = 0; f.max_c = INT64_MIN; f.settled = false;
            InHead g[4];
            g[0] = in_head[head_slot(tile, R, q, 0u)];       // (listed queues have at least one entry)
#pragma unroll
            for (int j = 1; j < 4; ++j) if ((uint32_t)j < c) g[j] = h[j];
#pragma unroll
            for (int j = 0; j < 4; ++j) if ((uint32_t)j < c) fix_entry(f, g[j], completion, stall);
            if (!f.settled && c > 4u) {
#pragma unroll
                for (int j = 4; j < kInHead; ++j) if ((uint32_t)j < c) g[j - 4] = h[j];
#pragma unroll
                for (int j = 4; j < kInHead; ++j) if ((uint32_t)j < c) fix_entry(f, g[j - 4], completion, stall);
            }
            max_c = max(max_c, f.max_c);                     // (true completions: valid whoever writes them last)
            if (!f.settled && c == head_depth) {
                // still backlogged after its head entries: the loop below serves this queue again from the tile's
                // start (Bt[q] still holds the entering value) and accounts for all of its corrections
                const uint32_t place = atomicAdd(&s_stragglers, 1u);
                oq[place] = (uint16_t)q;
                open[q] = (uint8_t)min(place + 1u, 255u);   // (a tile with more than kInStrMaxStragglers - 1 of them leaves below)
            } else {
                dstall += f.dstall;
            }
        }
    }
    __syncthreads();
    const uint32_t stragglers = s_stragglers;
    if (bal && tid == 0) {                                   // what the number of head entries of later batches follows from
        atomicMax(&bal->strag_max, stragglers);
        if (stragglers >= min(max(8u, R / 4u), (uint32_t)kInStrMaxStragglers)) atomicAdd(&bal->strag_flagged, 1u);
    }
    // many queues far behind: the re-serve pass takes the whole tile (one block serves it again from end to end, which costs
    // as much as the serve pass itself, so the bar is as high as this loop's tables allow)
    if (stragglers >= min(max(8u, R / 4u), (uint32_t)kInStrMaxStragglers)) {
        if (tid == 0) in_tile[tile].reserve = 1u;
        return;
    }
    if (stragglers > 0u) {
    const int64_t q_ppm = ctrl->q_ppm;
    const Div64 div_q = ctrl->div_q;
    const bool one_range = fast_arg.on != 0u && mp_arg.pow2_geom != 0u;
    const bool fast_terms = !PAGED && one_range && mp_arg.xfer_tab_max_cb != 0u && q_ppm == 1000000;
    const uint64_t claim_limit = DEBT ? *claim_limit_p : 0ull;     // as in the serve pass
    const int64_t quantum_ns = !DEBT ? 0 : q_ppm == 1000000 ? mp_arg.t_read_ns + mp_arg.t_prog_ns
        : (int64_t)div64((uint64_t)(mp_arg.t_read_ns + mp_arg.t_prog_ns) * 1000000ull + (uint64_t)q_ppm - 1ull, div_q);
    const uint64_t tile_begin = tile_first(tmap, tile), tile_end = tile_last(tmap, tile);
    const uint32_t tile_len = (uint32_t)(tile_end - tile_begin);       // offsets inside a tile fit 32 bits
    const hbf_access_t *acc_t = acc + tile_begin;
    const uint4 *qid_t = reinterpret_cast<const uint4 *>(in_qid + (uint64_t)tile * qid_stride);
    if (tid == 0) s_open = (int)stragglers;

    // the queue numbers of the next chunk are on their way while this one is filtered
    // (only the queue numbers: past the prefix, a rare stretch, the addresses are loaded when they are needed)
    uint4 nx_q[kInStrQItems / 8];
    auto fetch = [&](uint32_t cb) {
        if (cb < tile_len && cb + kInStrQChunk <= qid_stride) {
#pragma unroll
            for (int k = 0; k < kInStrQItems / 8; ++k) nx_q[k] = __ldg(qid_t + (cb >> 3) + tid * (kInStrQItems / 8) + k);
        }
    };
    // the kept records of a window, one per thread (their positions in the chunk are in the window already): the records are
    // fetched side by side, their terms computed once, and they take their places in the window
    constexpr int kPerThread = kInStrKeep / kInStrThreads;
    auto fill_window = [&](uint32_t cb, uint32_t wn) {
        uint64_t r_addr[kPerThread], r_bf[kPerThread]; int64_t r_issue[kPerThread]; uint32_t r_e[kPerThread];
#pragma unroll
        for (int k = 0; k < kPerThread; ++k) {
            const uint32_t slot = (uint32_t)(k * kInStrThreads + tid);
            if (slot < wn) {
                r_e[k] = ent_pq[slot].y;
                const uint64_t *rec = reinterpret_cast<const uint64_t *>(acc_t + cb + r_e[k]);
                r_addr[k] = __ldg(rec); r_issue[k] = (int64_t)__ldg(rec + 1); r_bf[k] = __ldg(rec + 2);
            }
        }
#pragma unroll
        for (int k = 0; k < kPerThread; ++k) {
            const uint32_t slot = (uint32_t)(k * kInStrThreads + tid);
            if (slot < wn) {
                Served v = fast_terms ? serve_terms_fast(fast_range, mp, r_addr[k], r_issue[k], r_bf[k])
                                      : serve_terms_general<PAGED>(rs, mp, r_addr[k], r_issue[k], r_bf[k], q_ppm, div_q);
                if (DEBT && tile_begin + cb + r_e[k] < claim_limit) v.s += quantum_ns;
                ent_as[slot] = make_longlong2(r_issue[k], v.s);
                ent_pq[slot] = make_uint2(v.xfer | (v.op << 31), v.queue | (r_e[k] << 16));
                const uint32_t place = open[v.queue];         // (0: the queue's runs met in an earlier window of this chunk)
                if (place) {
                    const uint32_t at = atomicAdd(&lcount[place - 1u], 1u);
                    if (at < (uint32_t)kInStrList) lst[(place - 1u) * kInStrList + at] = (uint16_t)slot; else s_overflow = 1u;
                }
            }
        }
    };
    fetch(0u);

    uint32_t cb = 0;
    while (cb < tile_len) {
        const bool by_qid = cb + kInStrQChunk <= qid_stride;  // the same for the whole block
        // ---- keep the modeled records of the open queues, in batch order: bit j of `keep` is this thread's item j, the
        // thread's items being 32 consecutive records
        uint32_t keep = 0;
        if (by_qid) {
            // (numbers past the tile's end are not defined: the table is indexed by 12 bits, twice the queues, and whatever
            // such a number finds there is masked off by position)
#pragma unroll
            for (int j = 0; j < kInStrQItems; ++j) {
                const uint4 v = nx_q[j >> 3];
                const uint32_t w = ((j >> 1) & 3) == 0 ? v.x : ((j >> 1) & 3) == 1 ? v.y : ((j >> 1) & 3) == 2 ? v.z : v.w;
                keep |= open[(w >> (16 * (j & 1))) & (2u * kInMaxQueues - 1u)] != 0 ? 1u << j : 0u;
            }
            const uint32_t room = tile_len - cb, mine = (uint32_t)(tid * kInStrQItems);   // records of the tile from this chunk on
            const uint32_t have = room > mine ? min(room - mine, (uint32_t)kInStrQItems) : 0u;
            keep &= have >= 32u ? 0xffffffffu : (1u << have) - 1u;
            fetch(cb + kInStrQChunk);
        } else {
            // past the prefix (a rare stretch: its size matters more than its speed) the queue comes from the record
#pragma unroll 2
            for (int j = 0; j < kInStrQItems; ++j) {
                const uint32_t i = cb + (uint32_t)(tid * kInStrQItems + j);
                if (i < tile_len) {
                    const uint64_t *rec = reinterpret_cast<const uint64_t *>(acc_t + i);
                    const uint64_t addr = __ldg(rec);
                    bool k;
                    if (one_range) {
                        const uint32_t q = fast_queue(fast_range, mp, addr);
                        k = q != 0xffffffffu && open[q] != 0;
                    } else {
                        const Served v = serve_terms_general<PAGED>(rs, mp, addr, (int64_t)__ldg(rec + 1), __ldg(rec + 2), q_ppm, div_q);
                        k = v.st == HBF_ST_READY && open[v.queue] != 0;
                    }
                    keep |= k ? 1u << j : 0u;
                }
            }
            fetch(cb + kInStrQChunk);
        }
        uint32_t first;                                      // place of this thread's first kept record among the chunk's
        {
            const uint32_t cnt = (uint32_t)__popc(keep);
            uint32_t incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += t; }
            if (lane == 31) s_cells[warp] = incl;
            __syncthreads();
            if (warp == 0) {
                const uint32_t c = lane < kInStrWarps ? s_cells[lane] : 0u;
                uint32_t in2 = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, in2, o); if (lane >= o) in2 += t; }
                if (lane < kInStrWarps) s_cells[lane] = in2 - c;
                if (lane == 31) s_total = in2;
            }
            __syncthreads();
            first = s_cells[warp] + incl - cnt;
        }
        // ---- the kept records, a window of kInStrKeep at a time (one window, nearly always)
        const uint32_t total = s_total;
        for (uint32_t wb = 0; wb < total; wb += (uint32_t)kInStrKeep) {
            const uint32_t wn = min(total - wb, (uint32_t)kInStrKeep);
            {
                uint32_t m = keep;
                while (m) {
                    const uint32_t j = (uint32_t)__ffs((int)m) - 1u;
                    m &= m - 1u;
                    const uint32_t slot = first + (uint32_t)__popc(keep & ((1u << j) - 1u)) - wb;   // (wraps below the window)
                    if (slot < wn) ent_pq[slot].y = (uint32_t)(tid * kInStrQItems) + j;
                }
            }
            __syncthreads();
            fill_window(cb, wn);
            __syncthreads();
            // Every straggling queue has the window's records of its own in a short list (in the order the threads happened
            // to append them): one thread per queue sorts its list by position (the window is in batch order) and re-serves
            // them, carrying the two runs.
            auto reserve_one = [&](uint32_t kk, int64_t &BT, int64_t &BA, bool writer) {
                const uint2 pq = ent_pq[kk];
                const longlong2 as = ent_as[kk];
                const int64_t xfer = (int64_t)(pq.x & 0x7fffffffu);
                const bool op = (pq.x >> 31) != 0u;
                const int64_t a = as.x + (op ? xfer : 0);
                BT = max(a, BT) + as.y; BA = max(a, BA) + as.y;
                if (BT != BA && writer) {                     // the serve pass wrote BA + post
                    const uint64_t i = min(tile_begin + cb + (pq.y >> 16), tile_end - 1);
                    const int64_t done = BT + (op ? 0 : xfer);
                    completion[i] = done; stall[i] = done - as.x;
                    dstall += BT - BA; max_c = max(max_c, (long long)done);
                }
            };
            if (!s_overflow) {
                for (uint32_t t = (uint32_t)tid; t < stragglers; t += kInStrThreads) {
                    const uint32_t q = oq[t];
                    const uint32_t cnt = lcount[t];
                    lcount[t] = 0u;
                    if (!open[q] || cnt == 0u) continue;
                    uint16_t *mine = lst + t * kInStrList;
                    for (uint32_t i = 1; i < cnt; ++i) {      // a handful of entries: insertion sort
                        const uint16_t key = mine[i];
                        uint32_t j = i;
                        while (j > 0u && mine[j - 1u] > key) { mine[j] = mine[j - 1u]; --j; }
                        mine[j] = key;
                    }
                    int64_t BT = Bt[q], BA = Ba[q];
                    for (uint32_t i = 0; i < cnt; ++i) reserve_one(mine[i], BT, BA, true);
                    Bt[q] = BT; Ba[q] = BA;
                    if (BT == BA) { open[q] = 0; atomicSub(&s_open, 1); }   // the runs have met: the rest of the tile was served right
                }
            } else {
                // some queue has more records in this window than a list holds: one warp per straggling queue scans the
                // window 32 records at a time and re-serves its own in order; every lane carries the two runs, lane 0 writes
                for (uint32_t t = (uint32_t)warp; t < stragglers; t += kInStrWarps) {
                    const uint32_t q = oq[t];
                    if (lane == 0) lcount[t] = 0u;
                    if (!open[q]) continue;
                    int64_t BT = Bt[q], BA = Ba[q];
                    for (uint32_t k0 = 0; k0 < wn; k0 += 32u) {
                        const uint32_t k = k0 + (uint32_t)lane;
                        unsigned hits = __ballot_sync(0xffffffffu, k < wn && (ent_pq[min(k, wn - 1u)].y & 0xffffu) == q);
                        while (hits) {
                            const uint32_t kk = k0 + (uint32_t)__ffs((int)hits) - 1u;
                            hits &= hits - 1u;
                            reserve_one(kk, BT, BA, lane == 0);
                        }
                    }
                    if (lane == 0) {
                        Bt[q] = BT; Ba[q] = BA;
                        if (BT == BA) { open[q] = 0; atomicSub(&s_open, 1); }
                    }
                }
                __syncthreads();
                if (tid == 0) s_overflow = 0u;
            }
            __syncthreads();
        }
        if (*reinterpret_cast<volatile int *>(&s_open) <= 0) break;
        cb += kInStrQChunk;
    }
    }
    dstall = warp_sum(dstall); max_c = warp_max(max_c);
    if (lane == 0) {
        if (dstall) atomicAdd((unsigned long long *)&s_red[0], (unsigned long long)dstall);
        if (max_c != INT64_MIN) atomicMax(&s_red[1], max_c);
    }
    __syncthreads();
    if (tid == 0) {
        if (s_red[0]) in_tile[tile].fix_delta = s_red[0];    // (cleared by the serve pass; this block is the tile's only writer)
        if (s_red[1] != INT64_MIN) atomicMax(&ctrl->max_completion_ns, s_red[1]);
    }
}


#ifndef HBF_IN_SKEW_PERMILLE
#define HBF_IN_SKEW_PERMILLE 60
#endif
// One wave of resident blocks: as many tiles as the device holds serve blocks.  When the batch is large enough to fill
// that wave, the tiles of the blocks that the hardware favours (one per SM) are larger by the skew, the others smaller,
// so that both blocks of an SM finish together.
InTileMap inorder_tile_map(uint64_t n, int sm_count, bool by_table) {
    InTileMap m{};
    m.n = n;
    const uint64_t sms = (uint64_t)std::max(1, sm_count);
    const uint64_t want_tiles = std::min<uint64_t>(kInMaxTiles, sms * kInBlocksPerSM);
    auto round_up = [](uint64_t v) { return std::max<uint64_t>((v + kInTileQuantum - 1) / kInTileQuantum * kInTileQuantum, kInTileQuantum); };
    const uint64_t even = round_up((n + want_tiles - 1) / want_tiles);
    if (kInBlocksPerSM == 2 && want_tiles == 2 * sms && even >= 64 * kInTileQuantum && HBF_IN_SKEW_PERMILLE > 0) {
        const uint64_t big = round_up(even * (1000 + HBF_IN_SKEW_PERMILLE) / 1000);
        if (by_table && 2 * sms <= kInBalMax) {
            // exactly two tiles per SM, their places in a table (launch_inorder writes it: the two nominal sizes until
            // measurements are at hand); big and small are the nominal sizes only
            m.n_big = (uint32_t)sms; m.n_tiles = (uint32_t)(2 * sms); m.big = (uint32_t)big;
            m.small = (uint32_t)round_up(even * (1000 - HBF_IN_SKEW_PERMILLE) / 1000);
            m.max_tile = (uint32_t)round_up(even * 1200 / 1000); m.by_sm = 1u;
            return m;
        }
        if (big * sms < n) {
            const uint64_t rest = n - big * sms;
            const uint64_t small = round_up((rest + sms - 1) / sms);
            m.n_big = (uint32_t)sms; m.big = (uint32_t)big; m.small = (uint32_t)small;
            m.n_tiles = (uint32_t)(sms + (rest + small - 1) / small);
            m.max_tile = (uint32_t)std::max(big, small);
            return m;
        }
    }
    m.n_big = 0; m.big = m.small = (uint32_t)even;
    m.n_tiles = (uint32_t)((n + even - 1) / even);
    m.max_tile = (uint32_t)even;
    return m;
}

// Where n_tiles tiles begin when tile t gets the share share[t] of a batch of n records, in whole quanta (every tile at
// least one); first[n_tiles] >= n.  (Finer ones than tiles of one size have: 1,024 records are 1.2 % of a tile of 24 M.)
constexpr uint32_t kInSizeQuantum = 256;
static void tiles_from_shares(const double *share, uint32_t n_tiles, uint64_t n, uint32_t *first, uint32_t *max_tile) {
    double sum_share = 0.0;
    for (uint32_t t = 0; t < n_tiles; ++t) sum_share += share[t];
    const uint64_t quanta = (n + kInSizeQuantum - 1) / kInSizeQuantum;
    uint64_t q[kInBalMax], used = 0;
    for (uint32_t t = 0; t < n_tiles; ++t) { q[t] = std::max<uint64_t>(1, (uint64_t)(share[t] / sum_share * (double)quanta)); used += q[t]; }
    for (uint32_t t = 0; used < quanta; t = (t + 1) % n_tiles) { ++q[t]; ++used; }           // what rounding down left over
    for (uint32_t t = 0; used > quanta; t = (t + 1) % n_tiles) if (q[t] > 1) { --q[t]; --used; }
    uint64_t at = 0, largest = 0;
    for (uint32_t t = 0; t < n_tiles; ++t) { first[t] = (uint32_t)(at * kInSizeQuantum); at += q[t]; largest = std::max(largest, q[t]); }
    first[n_tiles] = (uint32_t)(at * kInSizeQuantum);
    *max_tile = (uint32_t)(largest * kInSizeQuantum);
}

// Shares from the record an earlier batch left (see TileBalance): every tile in proportion to the rate measured at its
// place, blended with the share it had (so that one odd measurement moves a tile by little), within 15 % of the mean.
// False when the record is not a complete measurement of one batch with this many tiles.
static bool measured_shares(const TileBalance &rec, uint32_t n_tiles, double *share) {
    double rate[kInBalMax], sum_rate = 0.0, sum_len = 0.0;
    for (uint32_t t = 0; t < n_tiles; ++t) {
        if (rec.claim[t] != rec.claim[0] || rec.claim[t] == 0u || rec.ns[t] == 0u || rec.len[t] == 0u) return false;
        rate[t] = (double)rec.len[t] / (double)rec.ns[t];
        sum_rate += rate[t]; sum_len += (double)rec.len[t];
    }
    const double mean = 1.0 / n_tiles;
    for (uint32_t t = 0; t < n_tiles; ++t) {
        const double s = 0.3 * ((double)rec.len[t] / sum_len) + 0.7 * (rate[t] / sum_rate);
        share[t] = std::min(std::max(s, 0.85 * mean), 1.15 * mean);
    }
    return true;
}

// dynamic shared memory of the serve kernel: the per-queue state, the per-die counters, every warp's tables of lane numbers
size_t inorder_serve_smem(uint32_t n_dies) { return (size_t)kInMaxQueues * 16 + (size_t)n_dies * 28 + (size_t)kInWarps * kInRows * kInTagStride; }
static size_t inorder_straggle_smem() {
    return (size_t)kInMaxQueues * 16 + (size_t)kInStrKeep * 24 + (size_t)kInMaxQueues * 4 + (size_t)kInStrMaxStragglers * (kInStrList * 2 + 4);
}

size_t inorder_head_bytes(uint64_t tiles, uint32_t n_queues) { return tiles * n_queues * (size_t)kInHead * sizeof(InHead); }

// Batches whose tiles are all served twice, the first time without results and head entries (kInLight), in place of the fix-up.
// The second time reads 24 and writes 16 bytes per record; the fix-up and its head entries cost some 30 us and what the tiles
// times the queues make of them.  The line is drawn at 6.7 M records with 64 queues, 17.3 M with 1,024 and 28.5 M with 2,048, about where the two
// meet at a load of 0.3 (1,024 queues: a little before); with retention, where the first pass counts the reads into the disturb counters, they
// meet at 20 M with 2,048.  us, with the fix-up and served twice, whole passes, at 0.3: one-page reads, 64 queues, 4 M 142 and 123, 6 M 180 and
// 177, 7 M 189 and 187, 8 M 195 and 213; decode, 1,024 queues, 10 M 203 and 182, 12 M 220 and 224, 14 M 235 and 227, 16 M 263 and 243, 18 M 274
// and 274, 20 M 323 and 305, 22 M 313 and 344, 24 M 317 and 367; capacity, 2,048 queues, 24 M 379 and 364, 28 M 403 and 408, 32 M 431 and 449;
// two halves with retention, 18 M each 836 and 717, 24 M 856 and 928.  At 0.5 they meet at 7 M, 20 M and past 36 M: see below.
static uint64_t twice_max(uint32_t n_queues, bool retention) { return retention ? 5000000ull + 7500ull * n_queues : 6000000ull + 11000ull * n_queues; }
// Larger ones from a load on that rises with their size, towards 0.7, where queues begin to be behind everywhere (twice_from); and below
// it where a batch with about their load, or less, had to serve half of its tiles twice after all; every 16th of those takes the fix-up,
// to see whether it still does.  The device decides (begin_load), so both forms of the first pass are launched and one leaves at once
// (2 us).  us, with the fix-up and served twice, by load: capacity, 2,048 queues, 36 M 528 and 494 (0.5), 621 and 494 (0.6); 48 M 534 and 628 (0.3),
// 618 and 613 (0.5), 760 and 614 (0.6); 72 M 775 and 864 (0.5), 935 and 863 (0.6); two halves of 24 M with retention 1,006 and 912 (0.5).  With fewer
// queues it is later, for a tile has fewer of them to be behind: decode, 1,024, 24 M 321 and 346 (0.5), 346 and 344 (0.65), 36 M 426 and 470 (0.65);
// 64 queues, 32 M 480 and 536 (0.65).  Prefix, 1,024, 24 M, crowded on some queues at a time, 303 and 381 (0.2), 548 and 380 (0.3), 577 and 379 (0.5).
float twice_from(uint64_t n, uint32_t n_queues, bool retention) {
    const double x = (double)twice_max(n_queues, retention) / (double)std::max<uint64_t>(n, 1);
    return (float)std::min(0.70, 0.74 - 0.40 * ((double)n_queues / kInMaxQueues) * x);
}
TileBalance *inorder_decides(const SubmitArgs &a) {
    const bool by_table = a.bal && a.bal->on && a.bal->dev;
    return by_table && a.bal->depth_fixed == 0u && a.n > twice_max(a.mp.n_queues, a.claim_limit != nullptr) && inorder_tile_map(a.n, a.sm_count, true).by_sm ? a.bal->dev : nullptr;
}

cudaError_t launch_inorder(const SubmitArgs &a, cudaStream_t st) {
    const uint64_t n = a.n;
    const bool by_table = a.bal && a.bal->on && a.bal->dev;
    InTileMap tmap = inorder_tile_map(n, a.sm_count, by_table);
    const unsigned n_tiles = tmap.n_tiles;
    // one full wave of two tiles per SM: the blocks take their tiles by SM and kind and leave their times; the tiles' places
    // come from a table in device memory: sized by the record of an earlier batch when there is a complete one, else in the
    // two nominal sizes
    TileBalanceHost *bal = tmap.by_sm ? a.bal : nullptr;
    uint32_t bal_seq = 0;
    if (bal && a.stage == 2) {                               // (the tiles stand as the first stage left them)
        bal_seq = bal->seq; tmap.first = bal->dev->first;
    } else if (bal) {
        bal_seq = ++bal->seq;
        if (bal_seq == 0u) bal_seq = ++bal->seq;             // (0 marks a tile never taken)
        double share[kInBalMax];
        if (!measured_shares(*bal->pinned, n_tiles, share))
            for (uint32_t t = 0; t < n_tiles; ++t) share[t] = t < tmap.n_big ? (double)tmap.big : (double)tmap.small;
        uint32_t first[kInBalMax + 1], max_tile = 0;
        tiles_from_shares(share, n_tiles, n, first, &max_tile);
        // (from pageable memory: the copy is staged before the call returns, so the array may go out of scope)
        cudaError_t e = cudaMemcpyAsync(bal->dev->first, first, (n_tiles + 1) * sizeof(uint32_t), cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return e;
        tmap.first = bal->dev->first; tmap.max_tile = max_tile;
    }
    // Head entries per (tile, queue).  Fewer cost the serve pass less (a shorter stretch of every tile with the head
    // bookkeeping, a smaller table) and leave more queues to the straggle pass; past 254 of those in a tile the tile is
    // served a second time.  So the number follows what the last batch needed: one fewer while no tile had 148 straggling
    // queues (an entry fewer leaves about 1.3 times as many: 100, 130, 164, 224 per tile with 6, 5, 4, 3 entries on the
    // capacity stream at half load, so 148 become about 200), one more above 200, all of them after a tile was served twice.  Results do not
    // depend on it.
    uint32_t depth = (uint32_t)kInHead;
    if (bal) {
        if (bal->depth == 0u || bal->depth > (uint32_t)kInHead) bal->depth = (uint32_t)kInHead;
        const TileBalance &rec = *bal->pinned;
        if (rec.strag_seq != 0u && rec.strag_seq != bal->depth_seen && rec.strag_depth == bal->depth) {
            bal->depth_seen = rec.strag_seq;
            if (rec.strag_flagged != 0u) bal->depth = (uint32_t)kInHead;
            else if (rec.strag_max > 200u && bal->depth < (uint32_t)kInHead) ++bal->depth;
            else if (rec.strag_max < 148u && bal->depth > 3u) --bal->depth;
        }
        depth = bal->depth_fixed != 0u ? std::min<uint32_t>(bal->depth_fixed, (uint32_t)kInHead) : bal->depth;
    } else if (a.bal && a.bal->depth_fixed != 0u) {
        depth = std::min<uint32_t>(a.bal->depth_fixed, (uint32_t)kInHead);
    }
    const bool twice = a.stage != 0 || (n <= twice_max(a.mp.n_queues, a.claim_limit != nullptr) && !(a.bal && a.bal->depth_fixed != 0u));   // (a fixed number of head entries is the caller's)
    const bool decided = a.stage == 0 && inorder_decides(a) != nullptr;
    if (twice) depth = 0u;
    const uint64_t tile_records = tmap.max_tile;
    if (n_tiles > inorder_tiles_bound(n)) return cudaErrorInvalidValue;       // the workspace is carved for that many
    const uint32_t R = a.mp.n_queues, nd = a.mp.n_dies;
    const size_t smem_serve = inorder_serve_smem(nd), smem_str = inorder_straggle_smem();
    {
        const void *serve_fns[] = {(const void *)k_inorder_serve<kInFull, false, false>, (const void *)k_inorder_serve<kInAgain, false, false>, (const void *)k_inorder_serve<kInLight, false, false>,
                                   (const void *)k_inorder_serve<kInFull, true, false>, (const void *)k_inorder_serve<kInAgain, true, false>, (const void *)k_inorder_serve<kInLight, true, false>,
                                   (const void *)k_inorder_serve<kInLook, false, true>, (const void *)k_inorder_serve<kInFull, false, true>, (const void *)k_inorder_serve<kInAgain, false, true>, (const void *)k_inorder_serve<kInLight, false, true>};
        for (const void *f : serve_fns) { cudaError_t e = ensure_dyn_smem(f, smem_serve); if (e != cudaSuccess) return e; }
        cudaError_t e = ensure_dyn_smem((const void *)k_inorder_scan, 0);
        if (e != cudaSuccess) return e;
        const void *fix_fns[3] = {(const void *)k_inorder_fixstraggle<false, false>, (const void *)k_inorder_fixstraggle<true, false>,
                                  (const void *)k_inorder_fixstraggle<false, true>};
        for (const void *f : fix_fns) { e = ensure_dyn_smem(f, smem_str); if (e != cudaSuccess) return e; }
    }
    InTile *tiles = reinterpret_cast<InTile *>(a.ws.in_tile);
    InHead *heads = reinterpret_cast<InHead *>(a.ws.in_head);
    const bool debt = a.claim_limit != nullptr;              // retention on: the kernels that apply the claims
    const uint32_t qid_stride = twice ? 0u : (uint32_t)std::min<uint64_t>(tile_records, kInQidPrefix);
    if ((uint64_t)n_tiles * qid_stride > inorder_qid_entries(n)) return cudaErrorInvalidValue;
    auto serve = [&](int mode) {
        auto pick = [&](auto full, auto second, auto light) { return mode == kInAgain ? second : mode == kInLight ? light : full; };
        auto k = a.stage == 1 ? k_inorder_serve<kInLook, false, true>
               : a.paged ? pick(k_inorder_serve<kInFull, false, true>, k_inorder_serve<kInAgain, false, true>, k_inorder_serve<kInLight, false, true>)
               : debt ? pick(k_inorder_serve<kInFull, true, false>, k_inorder_serve<kInAgain, true, false>, k_inorder_serve<kInLight, true, false>)
                      : pick(k_inorder_serve<kInFull, false, false>, k_inorder_serve<kInAgain, false, false>, k_inorder_serve<kInLight, false, false>);
        return launch_pdl(k, n_tiles, kInThreads, smem_serve, st, a.acc, n, tmap, a.ranges, a.mp, a.fast, a.ctrl,
                          mode == kInAgain && a.stage == 0 ? (uint8_t *)nullptr : a.status, a.ws.in_agg,
                          a.stats_stage, a.completion, a.stall, (const int64_t *)a.ws.in_bin, tiles, heads, a.ws.in_headcnt,
                          (const int64_t *)a.busy, a.claim_limit, a.die_claims, debt ? *a.ret : RetDev{}, a.ws.in_qid, qid_stride,
                          bal ? bal->dev : nullptr, bal_seq, make_fast_geom(a.fast, a.mp), depth, ordered_copy(n, a.ws), decided ? 1 : 0);
    };
    cudaError_t le = cudaSuccess;
    if (a.stage != 2) le = twice ? serve(kInLight) : serve(kInFull);
    if (le == cudaSuccess && decided) le = serve(kInLight);
    if (a.stage == 1) { g_kernel_launches += 1; return le; }
    if (le == cudaSuccess)
        le = launch_first(a.stage == 2 ? a.plain_next : nullptr, k_inorder_scan, (R + kInScanQueues - 1) / kInScanQueues, dim3(kInScanQueues, kInScanChunks), 0, st, a.ctrl, a.mp_dev, n_tiles,
                        (const int64_t *)a.ws.in_agg, a.ws.in_bin, (const int64_t *)a.busy, a.busy_stage, a.stats_stage, a.path == HBF_PATH_INORDER ? 1 : 0);
    if (le == cudaSuccess && !twice)
        le = launch_pdl(a.paged ? k_inorder_fixstraggle<false, true> : debt ? k_inorder_fixstraggle<true, false> : k_inorder_fixstraggle<false, false>, n_tiles, kInStrThreads,
                        smem_str, st, a.acc, n, tmap, a.ranges, a.mp, a.fast, a.ctrl, (const int64_t *)a.ws.in_bin, (const InHead *)heads, (const uint8_t *)a.ws.in_headcnt,
                        a.completion, a.stall, tiles, a.claim_limit, (const uint16_t *)a.ws.in_qid, qid_stride, depth, bal ? bal->dev : nullptr, ordered_copy(n, a.ws));
    if (le == cudaSuccess) le = serve(kInAgain);
    if (le != cudaSuccess) return le;
    if (bal) {                                               // the tiles' times and straggler counts, for later batches; nothing waits for this copy
        cudaError_t e = cudaMemcpyAsync(bal->pinned, bal->dev, offsetof(TileBalance, first), cudaMemcpyDeviceToHost, st);
        if (e != cudaSuccess) return e;
    }
    g_kernel_launches += a.stage == 2 ? 2 : twice ? 3 : decided ? 5 : 4;
    return cudaGetLastError();
}

}  // namespace hbf

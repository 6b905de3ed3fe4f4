// Host side of the in-order path (its kernels: inorder_impl.cuh): how a batch is cut into tiles, and the launches.
#include <algorithm>
#include <cstddef>

#include "inorder_impl.cuh"

namespace hbf {

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
// least one); first[n_tiles] >= n.
static void tiles_from_shares(const double *share, uint32_t n_tiles, uint64_t n, uint32_t *first, uint32_t *max_tile) {
    double sum_share = 0.0;
    for (uint32_t t = 0; t < n_tiles; ++t) sum_share += share[t];
    const uint64_t quanta = (n + kInTileQuantum - 1) / kInTileQuantum;
    uint64_t q[kInBalMax], used = 0;
    for (uint32_t t = 0; t < n_tiles; ++t) { q[t] = std::max<uint64_t>(1, (uint64_t)(share[t] / sum_share * (double)quanta)); used += q[t]; }
    for (uint32_t t = 0; used < quanta; t = (t + 1) % n_tiles) { ++q[t]; ++used; }           // what rounding down left over
    for (uint32_t t = 0; used > quanta; t = (t + 1) % n_tiles) if (q[t] > 1) { --q[t]; --used; }
    uint64_t at = 0, largest = 0;
    for (uint32_t t = 0; t < n_tiles; ++t) { first[t] = (uint32_t)(at * kInTileQuantum); at += q[t]; largest = std::max(largest, q[t]); }
    first[n_tiles] = (uint32_t)(at * kInTileQuantum);
    *max_tile = (uint32_t)(largest * kInTileQuantum);
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
size_t inorder_straggle_smem() {
    return (size_t)kInMaxQueues * 16 + (size_t)kInStrKeep * 24 + (size_t)kInMaxQueues * 4 + (size_t)kInStrMaxStragglers * (kInStrList * 2 + 4);
}

size_t inorder_head_bytes(uint64_t tiles, uint32_t n_queues) { return tiles * n_queues * (size_t)kInHead * sizeof(InHead); }

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
    if (bal) {
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
    const uint64_t tile_records = tmap.max_tile;
    if (n_tiles > inorder_tiles_bound(n)) return cudaErrorInvalidValue;       // the workspace is carved for that many
    const uint32_t R = a.mp.n_queues, nd = a.mp.n_dies;
    const size_t smem_serve = inorder_serve_smem(nd), smem_str = inorder_straggle_smem();
    {
        const void *serve_fns[6] = {(const void *)k_inorder_serve<false, false, false>, (const void *)k_inorder_serve<true, false, false>,
                                    (const void *)k_inorder_serve<false, true, false>, (const void *)k_inorder_serve<true, true, false>,
                                    (const void *)k_inorder_serve<false, false, true>, (const void *)k_inorder_serve<true, false, true>};
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
    const uint32_t qid_stride = (uint32_t)std::min<uint64_t>(tile_records, kInQidPrefix);
    if ((uint64_t)n_tiles * qid_stride > inorder_qid_entries(n)) return cudaErrorInvalidValue;
    auto serve = [&](bool reserve) {
        auto k = a.paged ? (reserve ? k_inorder_serve<true, false, true> : k_inorder_serve<false, false, true>)
               : reserve ? (debt ? k_inorder_serve<true, true, false> : k_inorder_serve<true, false, false>)
                         : (debt ? k_inorder_serve<false, true, false> : k_inorder_serve<false, false, false>);
        return launch_pdl(k, n_tiles, kInThreads, smem_serve, st, a.acc, n, tmap, a.ranges, a.mp, a.fast, a.ctrl, a.status, a.ws.in_agg,
                          a.stats_stage, a.completion, a.stall, (const int64_t *)a.ws.in_bin, tiles, heads, a.ws.in_headcnt,
                          (const int64_t *)a.busy, a.claim_limit, a.die_claims, debt ? *a.ret : RetDev{}, a.ws.in_qid, qid_stride,
                          bal ? bal->dev : nullptr, bal_seq, make_fast_geom(a.fast, a.mp), depth);
    };
    cudaError_t le = serve(false);
    if (le == cudaSuccess)
        le = launch_pdl(k_inorder_scan, (R + kInScanQueues - 1) / kInScanQueues, dim3(kInScanQueues, kInScanChunks), 0, st, a.ctrl, a.mp_dev, n_tiles,
                        (const int64_t *)a.ws.in_agg, a.ws.in_bin, (const int64_t *)a.busy, a.busy_stage, a.stats_stage, a.path == HBF_PATH_INORDER ? 1 : 0);
    if (le == cudaSuccess)
        le = launch_pdl(a.paged ? k_inorder_fixstraggle<false, true> : debt ? k_inorder_fixstraggle<true, false> : k_inorder_fixstraggle<false, false>, n_tiles, kInStrThreads,
                        smem_str, st, a.acc, n, tmap, a.ranges, a.mp, a.fast, a.ctrl, (const int64_t *)a.ws.in_bin, (const InHead *)heads, (const uint8_t *)a.ws.in_headcnt,
                        a.completion, a.stall, tiles, a.claim_limit, (const uint16_t *)a.ws.in_qid, qid_stride, depth, bal ? bal->dev : nullptr);
    if (le == cudaSuccess) le = serve(true);
    if (le != cudaSuccess) return le;
    if (bal) {                                               // the tiles' times and straggler counts, for later batches; nothing waits for this copy
        cudaError_t e = cudaMemcpyAsync(bal->pinned, bal->dev, offsetof(TileBalance, first), cudaMemcpyDeviceToHost, st);
        if (e != cudaSuccess) return e;
    }
    g_kernel_launches += 4;
    return cudaGetLastError();
}

}  // namespace hbf

// What the in-order kernels need of one access, from its record.
#pragma once
#include "device_utils.cuh"

namespace hbf {

// One access, from its record: status, and for a modeled access its queue, die and service terms.
// (the in-order path is only chosen when every transfer time fits 31 bits)
struct Served { int st; uint32_t queue, die, op, xfer; int64_t s, cb; uint32_t parts; };
// long_service (here and below): set when one access's service time reaches 2^long_bits ns.  The serve pass keeps a tile's
// service-time sum per queue in 56 bits (55 and a sign); a tile has fewer than 2^22 records, so with every service below
// 2^33 ns (8.6 s) the sum cannot overflow; with retention on a claimed refresh quantum is added to a service, and both
// stay below 2^32.  A batch with a longer service is handed to the sort path like an unsorted one.
__device__ __forceinline__ Served serve_terms(const RangeSnap &rs, const ModelParams &mp, uint64_t addr, int64_t issue,
                                              uint64_t bf, int64_t q_ppm, const Div64 &div_q, unsigned &long_service, int long_bits) {
    Served r; r.queue = 0; r.die = 0; r.op = 0; r.s = 0; r.xfer = 0; r.cb = 0; r.parts = 1;
    const uint32_t bytes = (uint32_t)bf, flags = (uint32_t)(bf >> 32);
    int g = 0;
    r.st = classify(rs, addr, issue, bytes, flags, &g);
    if (r.st == HBF_ST_READY) {
        const uint64_t off = rs.media_offset[g] + (addr - rs.base[g]);
        const Decoded d = decode(mp, off, bytes);
        r.op = flags & 1u;
        const Terms t = service_terms(mp, bytes, d.npages, r.op, q_ppm, div_q);
        r.queue = d.queue; r.die = d.die; r.s = t.s; r.xfer = (uint32_t)t.xfer; r.cb = t.cb;
        if ((uint64_t)t.s >> long_bits) long_service = 1u;
    }
    return r;
}

// The same terms for the common configuration (one registered range, power-of-two geometry, no thermal
// scaling in force, transfer table present): 32-bit arithmetic wherever the values allow it.
// (TABLE = false: the transfer by multiply-high, for a kernel that waits for the table's entry and has nothing else to do meanwhile)
template <bool TABLE = true>
__device__ __forceinline__ Served serve_terms_fast(const FastRange &f, const ModelParams &mp, uint64_t addr, int64_t issue, uint64_t bf) {
    Served r; r.queue = 0; r.die = 0; r.op = 0; r.s = 0; r.xfer = 0; r.cb = 0; r.parts = 1;
    const uint32_t bytes = (uint32_t)bf, flags = (uint32_t)(bf >> 32);
    const uint64_t rel = addr - f.base;                       // wraps to a huge value below the base
    if (bytes == 0u || (flags & ~1u) != 0u || (uint32_t)((uint64_t)issue >> 32) >= (1u << (kIssueBits - 32))) { r.st = HBF_ST_UNSUPPORTED; return r; }
    if (rel >= f.length) { r.st = HBF_ST_NATIVE; return r; }
    if ((uint64_t)bytes > f.length - rel) { r.st = HBF_ST_FAULT_PARTIAL; return r; }
    r.op = flags & 1u;
    if (!(f.perms & (1u << r.op))) { r.st = HBF_ST_FAULT_PERM; return r; }
    r.st = HBF_ST_READY;
    const uint64_t off = f.media_offset + rel;
    const uint32_t u = (uint32_t)(off >> mp.stripe_shift);    // only the low interleave bits are used
    const uint32_t ch = u & (mp.channels - 1u), di = (u >> mp.ch_shift) & (mp.dies - 1u);
    const uint32_t pl = (u >> (mp.ch_shift + mp.die_shift)) & (mp.planes - 1u);
    r.die = ch * mp.dies + di;
    r.queue = mp.queue_level == 0u ? r.die * mp.planes + pl : r.die;
    const uint32_t page_mask = (1u << mp.page_shift) - 1u;
    const uint32_t npages = (uint32_t)(((uint64_t)((uint32_t)off & page_mask) + bytes + page_mask) >> mp.page_shift);
    const uint32_t gs = r.op ? mp.prog_gran_shift : mp.read_gran_shift;
    const uint64_t cb = (((uint64_t)bytes + ((1ull << gs) - 1ull)) >> gs) << gs;
    r.cb = (int64_t)cb;
    r.xfer = TABLE && cb <= (uint64_t)mp.xfer_tab_max_cb ? __ldg(mp.xfer_tab + (uint32_t)(cb >> mp.xfer_tab_shift))
                                                 : (uint32_t)div64(cb * 1000ull + mp.chan_bytes_per_us - 1ull, mp.div_chan);
    r.s = (int64_t)npages * (r.op ? mp.t_prog_ns : mp.t_read_ns);
    return r;
}

// The common configuration once more, laid out for the serve pass (a kernel argument: its fields are operands of the
// instructions that use them, which measured 1.8 % faster than seven 16-byte vectors in shared memory), every field a
// 32-bit operand where the values allow it (page times and the transfer table's reach below 2^32).
struct __align__(16) FastGeom {
    uint64_t base, length;                                  // the one registered range
    uint64_t media_offset; uint32_t perms, stripe_shift;
    uint32_t ch_mask, ch_shift, die_mask, chdie_shift;      // stripe unit -> channel, die, plane
    uint32_t plane_mask, dies, planes_q, plane_mask_q;      // planes_q = 1, plane_mask_q = 0 with one queue per die
    uint32_t page_mask, page_shift, gran_shift_read, gran_shift_prog;
    uint32_t tab_shift, tab_max_cb, t_read, t_prog;
    const uint32_t *xfer_tab; uint64_t pad;
    // the 32-bit form of the pass (serve_narrow below); narrow == 0: not for this configuration
    uint64_t nw_delta, nw_lim;                               // media offset = address + nw_delta; range offsets up to nw_lim hold any inline access
    uint32_t narrow, nw_bytes, nw_flag_lo, nw_flag_n;        // inline accesses: at most nw_bytes bytes, flags nw_flag_lo .. nw_flag_lo + nw_flag_n - 1
    uint32_t nw_gmax, nw_mul_read, nw_mul_prog, nw_add;      // most granules of an inline read; transfer = (granules * mul + add) / rate by
    uint32_t nw_magic, nw_shift, nw_chmul, nw_pad;           //   multiply-high; queues per channel
    uint32_t nw_page_read, nw_page_prog, nw_page_gran, nw_chmul_shift;   // page-granular submit: transfer of a whole page, read granules of one
    uint32_t nw_slot_mask, nw_plane_shift, nw_pad2, nw_pad3;  // a queue's slot (see queue_slot): these low bits of the stripe unit's number; planes_q as a shift
};
// Where a queue's state lies in shared memory (power-of-two geometry): channel first, then die, then plane, as in the number of
// the stripe unit.  Neighbouring stripe units, which the streams of weights and prefixes walk along, lie on neighbouring channels:
// by queue number (channel last) their 16-byte states were dies * planes apart, all in the same four banks.
__device__ __forceinline__ uint32_t queue_slot(const FastGeom &g, uint32_t q) {
    return (q >> g.nw_chmul_shift) | (((q >> g.nw_plane_shift) & g.die_mask) << g.ch_shift) | ((q & g.plane_mask_q) << g.chdie_shift);
}
__device__ __forceinline__ uint32_t slot_die(const FastGeom &g, uint32_t s) { return (s & g.ch_mask) * g.dies + ((s >> g.ch_shift) & g.die_mask); }
__device__ __forceinline__ uint32_t slot_queue(const FastGeom &g, uint32_t s) { return (slot_die(g, s) << g.nw_plane_shift) + ((s >> g.chdie_shift) & g.plane_mask_q); }
// Bounds of the 32-bit form.  A service is below 2^26 ns, so that the services of a row's 32 lanes compose below 2^31; the
// granules and the reads of an access fit 11 and 6 bits, so that a row's sums travel in one word (17 and 11 bits).
constexpr uint32_t kNwServeBits = 26, kNwGranules = 2048, kNwPages = 32, kNwCountShift = 17;
// (the last condition: an access within the transfer table's reach spans few pages, and their unscaled service stays
// below 2^32 ns, so the common path needs no test of its own)
__host__ __device__ __forceinline__ bool fast_geom_ok(const FastRange &f, const ModelParams &mp) {
    const uint64_t pages = ((uint64_t)mp.xfer_tab_max_cb >> mp.page_shift) + 2ull;
    return f.on != 0u && mp.pow2_geom != 0u && mp.xfer_tab_max_cb != 0u && mp.t_read_ns < (1ll << 32) && mp.t_prog_ns < (1ll << 32) &&
           pages * (uint64_t)(mp.t_read_ns > mp.t_prog_ns ? mp.t_read_ns : mp.t_prog_ns) < (1ull << 32);
}
__host__ __device__ __forceinline__ FastGeom make_fast_geom(const FastRange &f, const ModelParams &mp) {
    FastGeom g;
    g.base = f.base; g.length = f.length; g.media_offset = f.media_offset; g.perms = f.perms; g.stripe_shift = mp.stripe_shift;
    g.ch_mask = mp.channels - 1u; g.ch_shift = mp.ch_shift; g.die_mask = mp.dies - 1u; g.chdie_shift = mp.ch_shift + mp.die_shift;
    g.plane_mask = mp.planes - 1u; g.dies = mp.dies;
    g.planes_q = mp.queue_level == 0u ? mp.planes : 1u; g.plane_mask_q = mp.queue_level == 0u ? mp.planes - 1u : 0u;
    g.page_mask = (1u << mp.page_shift) - 1u; g.page_shift = mp.page_shift;
    g.gran_shift_read = mp.read_gran_shift; g.gran_shift_prog = mp.prog_gran_shift;
    g.tab_shift = mp.xfer_tab_shift; g.tab_max_cb = mp.xfer_tab_max_cb; g.t_read = (uint32_t)mp.t_read_ns; g.t_prog = (uint32_t)mp.t_prog_ns;
    g.xfer_tab = mp.xfer_tab; g.pad = 0;
    // 32-bit form: which accesses are inline, and the division by the channel rate d as a 32-bit multiply-high (exact for
    // numerators below 2^31: magic = floor(2^(31+l) / d) + 1 with l = ceil(log2 d), shift l - 1)
    g.nw_delta = f.media_offset - f.base; g.nw_chmul = mp.dies * g.planes_q; g.nw_pad = 0;
    g.nw_flag_lo = (f.perms & 1u) ? 0u : 1u; g.nw_flag_n = (f.perms & 3u) == 3u ? 2u : 1u;
    g.nw_mul_read = 1000u << (mp.read_gran_shift & 15u); g.nw_mul_prog = 1000u << (mp.prog_gran_shift & 15u);
    g.narrow = 0u; g.nw_bytes = g.nw_gmax = g.nw_add = g.nw_magic = g.nw_shift = 0u; g.nw_lim = 0; g.nw_page_read = g.nw_page_prog = g.nw_page_gran = g.nw_pad2 = g.nw_pad3 = 0u;
    g.nw_plane_shift = mp.queue_level == 0u ? mp.plane_shift : 0u; g.nw_chmul_shift = mp.die_shift + g.nw_plane_shift; g.nw_slot_mask = mp.channels * mp.dies * g.planes_q - 1u;
    const uint64_t d = mp.chan_bytes_per_us, t_max = (uint64_t)(mp.t_read_ns > mp.t_prog_ns ? mp.t_read_ns : mp.t_prog_ns);
    const uint64_t quantum = (uint64_t)mp.t_read_ns + (uint64_t)mp.t_prog_ns;   // (a claimed refresh quantum is added to a service)
    if (fast_geom_ok(f, mp) && d >= 2u && d < (1ull << 30) && mp.read_gran_shift <= 15u && mp.prog_gran_shift <= 15u && mp.page_shift <= 20u &&
        (f.perms & 3u) != 0u && quantum < (1ull << (kNwServeBits - 1))) {
        const uint64_t pages_s = ((1ull << kNwServeBits) - 1u - quantum) / t_max, pages = pages_s < kNwPages ? pages_s : kNwPages;
        uint64_t most = pages >= 2u ? (pages - 1u) << mp.page_shift : 0u;       // so many bytes never touch more than `pages` pages
        if (((uint64_t)kNwGranules << mp.read_gran_shift) < most) most = (uint64_t)kNwGranules << mp.read_gran_shift;
        if (f.length < most) most = f.length;
        const uint64_t worst = (most + ((1ull << mp.read_gran_shift) | (1ull << mp.prog_gran_shift)) * 2u) * 1000u + d;
        if (most >= 1u && worst < (1ull << 31)) {
            uint32_t l = 0;
            while ((1ull << l) < d) ++l;
            g.narrow = 1u; g.nw_bytes = (uint32_t)most; g.nw_lim = f.length - most;
            g.nw_gmax = (uint32_t)((most + (1ull << mp.read_gran_shift) - 1u) >> mp.read_gran_shift) + kNwPages;   // (every part of a paged access may round up)
            g.nw_add = (uint32_t)d - 1u; g.nw_magic = (uint32_t)((1ull << (31 + l)) / d + 1u); g.nw_shift = l - 1u;
            const uint64_t page = 1ull << mp.page_shift, gr = (1ull << mp.read_gran_shift) - 1u, gp = (1ull << mp.prog_gran_shift) - 1u;
            g.nw_page_read = (uint32_t)((((page + gr) & ~gr) * 1000u + d - 1u) / d); g.nw_page_prog = (uint32_t)((((page + gp) & ~gp) * 1000u + d - 1u) / d);
            g.nw_page_gran = (uint32_t)((page + gr) >> mp.read_gran_shift);
        }
    }
    return g;
}

}  // namespace hbf

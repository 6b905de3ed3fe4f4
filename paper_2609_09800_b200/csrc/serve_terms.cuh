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
    r.xfer = cb <= (uint64_t)mp.xfer_tab_max_cb ? __ldg(mp.xfer_tab + (uint32_t)(cb >> mp.xfer_tab_shift))
                                                 : (uint32_t)div64(cb * 1000ull + mp.chan_bytes_per_us - 1ull, mp.div_chan);
    r.s = (int64_t)npages * (r.op ? mp.t_prog_ns : mp.t_read_ns);
    return r;
}

}  // namespace hbf

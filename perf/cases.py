"""The work that a user of the library has it do, as cases that can be timed: inputs made on the GPU from a seed, one pass through
the public entry points, and what the pass cannot do without.

A case is a dict of plain values.  Its "kind" says which of the library's uses it is:

  batch      one batch of accesses on idle queues (`reset`, `submit_batch`, `thermal_step` where the geometry has a package
             floorplan, `last_result`): what the bench times; "bus" puts the channel-bus stage behind it
  paged      the same through the page-granular submit
  retention  two consecutive halves of a stream with retention on and an epoch between them, so that part of the second half
             claims refresh quanta
  windows    a coupled run: the stream in windows of 1 ms, a thermal step after each; "full" switches the energy bins and retention
             (one epoch per window, temperatures from the field) on
  online     the same loop for a caller that injects the stalls as it goes: records and results in pinned host memory, the thermal
             step on a reduced-order model, the hotspots read back after every window

and the rest says on which stream: "stream" (one of the generators below), "n" accesses (or "windows" of 1 ms), the offered load
"rho", and "order" ("issue": as issued; "shuffled": in no order; "rings": the concatenation of in-order logs, as when every SM of a
device keeps its own).  Every pass starts from `reset`, so that a pass can be repeated: the queues of the pass before are idle
again, the thermal field is at ambient.
"""
import functools
import math

import numpy as np
import torch

from paper_2609_09800_b200 import hbf, workloads as wl

WINDOW_NS = 1_000_000
# A batch spans seconds of simulated time and is charged to one thermal window of 1 ms, which is no physical power: the
# thresholds are raised so that the controller stays in Normal mode (as the bench does).
BATCH_THRESHOLDS = dict(rtt_c=1e6, ltt_c=2e6, stt_c=3e6, shutdown_c=4e6)
# a geometry that is no power of two
ODD_GEOMETRY = dict(channels=12, dies=6, planes=3, page_bytes=16384, stripe_bytes=65536)
RINGS = 148                       # in-order logs of the "rings" order
GRID_CELLS = 128 * 128
ROM_STATES, ROM_OUTPUTS = 224, 11


def listed():
    return [
        # Long-run coupled mode: the smallest calls, about 5,900 accesses (programs of the shared prefix, then decode reads) and a
        # thermal step per simulated millisecond; what counts is latency and launches.
        dict(name="windows_grid", kind="windows", stream="prefix", windows=48, rho=0.5, full=False),
        # The closed loop of temperature, retention, refresh debt and bandwidth: the same with bins and retention on.
        dict(name="windows_full", kind="windows", stream="prefix", windows=24, rho=0.5, full=True),
        # Online service of a running program: every millisecond's records come from the host and their stalls go back to it.
        dict(name="windows_online", kind="online", stream="prefix", windows=24, rho=0.5),
        # A small experiment: one-page reads on the tiny geometry.
        dict(name="uniform_65k", kind="batch", stream="uniform", n=65_536, rho=0.5, order="issue", bus=False),
        # Several ranges, one of them read-only, natives between them, programs, odd sizes, a ragged count.
        dict(name="mixed_1500k", kind="batch", stream="mixed", n=1_500_007, rho=0.6, order="issue", bus=False),
        # Decode weight streaming, 48 tokens: an ordinary batch.
        dict(name="decode_4m", kind="batch", stream="decode", n=3_981_312, rho=0.5, order="issue", bus=False),
        # Shared-prefix KV cache plus weights: programs and hot tiles, at a higher load.
        dict(name="prefix_24m", kind="batch", stream="prefix", n=24_000_011, rho=0.7, order="issue", bus=False),
        # Capacity mode: the largest batch, the bench's headline.
        dict(name="capacity_200m", kind="batch", stream="capacity", n=200_000_000, rho=0.5, order="issue", bus=False),
        # The same records in no order: merged logs of many producers.
        dict(name="shuffled_40m", kind="batch", stream="capacity", n=40_000_003, rho=0.5, order="shuffled", bus=False),
        # Page-granular back end: every page of an access queued on its own.
        dict(name="paged_64m", kind="paged", stream="capacity", n=64_000_000, rho=0.5),
        # Transfers queue per channel behind the array stage.
        dict(name="bus_32m", kind="batch", stream="capacity", n=32_000_000, rho=0.5, order="issue", bus=True),
        # A device that has to refresh part of its blocks: a batch without debt, an epoch, a batch that pays claims.
        dict(name="retention_48m", kind="retention", stream="capacity", n=48_000_000, rho=0.5, limit=1.06),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges.  (No size is above the listed one of its kind.)"""
    what = rng.choice(["windows", "windows", "online", "small", "mixed", "batch", "batch", "capacity", "unordered", "paged", "bus", "retention"])
    rho = round(rng.uniform(0.2, 0.9), 3)
    if what == "windows":
        full = rng.random() < 0.5
        return dict(kind="windows", stream=rng.choice(["prefix", "decode"]), windows=rng.randint(6, 24 if full else 48), rho=rho, full=full)
    if what == "online":
        return dict(kind="online", stream=rng.choice(["prefix", "decode"]), windows=rng.randint(6, 24), rho=rho)
    if what == "small":
        return dict(kind="batch", stream=rng.choice(["uniform", "decode", "capacity"]), n=_log_uniform(rng, 1_000, 400_000), rho=rho, order="issue", bus=False)
    if what == "mixed":
        return dict(kind="batch", stream="mixed", n=_log_uniform(rng, 5_000, 8_000_000), rho=rho, order=rng.choice(["issue", "issue", "shuffled"]), bus=False)
    if what == "batch":
        return dict(kind="batch", stream=rng.choice(["decode", "prefix"]), n=_log_uniform(rng, 400_000, 24_000_000), rho=rho, order="issue", bus=False)
    if what == "capacity":
        return dict(kind="batch", stream="capacity", n=_log_uniform(rng, 1_000_000, 120_000_000), rho=rho, order="issue", bus=False)
    if what == "unordered":
        return dict(kind="batch", stream=rng.choice(["capacity", "decode", "prefix"]), n=_log_uniform(rng, 20_000, 24_000_000), rho=rho,
                    order=rng.choice(["shuffled", "rings"]), bus=False)
    if what == "paged":
        stream = rng.choice(["capacity", "decode", "mixed"])
        return dict(kind="paged", stream=stream, n=_log_uniform(rng, 20_000, 4_000_000 if stream == "mixed" else 40_000_000), rho=rho)
    if what == "bus":
        return dict(kind="batch", stream=rng.choice(["capacity", "decode", "prefix"]), n=_log_uniform(rng, 20_000, 24_000_000), rho=rho, order="issue", bus=True)
    return dict(kind="retention", stream="capacity", n=_log_uniform(rng, 100_000, 40_000_000), rho=rho, limit=round(rng.uniform(0.9, 1.15), 3))


# ---- streams, made on the GPU -------------------------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & ((1 << 62) - 1))
    return g


def _records(off, nbytes, flags, mean_gap, g, out=None, t0=None, base=wl.RANGE_BASE):
    """Records [n][3] int64 (address, issue time, bytes | flags << 32) with Poisson issue times behind t0 (a device scalar)."""
    n = off.numel()
    rec = torch.empty((n, 3), dtype=torch.int64, device="cuda") if out is None else out
    gaps = torch.empty(n, dtype=torch.float64, device="cuda").exponential_(1.0 / mean_gap, generator=g).mul_(1024.0)
    t = gaps.long().cumsum_(0)                           # in 1/1024 ns, whole numbers: a float scan is not the same twice
    if t0 is not None:
        t += t0
    rec[:, 0] = off + base
    rec[:, 1] = t >> 10
    rec[:, 2] = nbytes + (flags << 32) if torch.is_tensor(flags) else nbytes
    return rec, t[-1].clone()


def _uniform(n, rho, g):
    prof = wl.load_profile("nominal", **wl.GEOMETRY["tiny"])
    off = torch.randint(0, wl.GIB // (4 * wl.KIB), (n,), device="cuda", generator=g) * (4 * wl.KIB)
    rec, _ = _records(off, 4 * wl.KIB, 0, prof["t_read_ns"] / (rho * 8 * 4 * 2), g)
    return prof, [(wl.RANGE_BASE, wl.GIB, 3, 0, 0, 0)], rec


def _top_experts(tokens, g):
    """Experts of every token and layer [tokens][layers][8]: Zipf(1.1) popularity without replacement (Gumbel top-k)."""
    logw = -1.1 * torch.log(torch.arange(1, wl.N_EXPERTS + 1, device="cuda", dtype=torch.float32))
    gumbel = -torch.log(torch.empty((tokens, wl.N_LAYERS, wl.N_EXPERTS), device="cuda").exponential_(generator=g))
    ranks = torch.topk(logw + gumbel, wl.TOP_K, dim=-1).indices
    perms = torch.argsort(torch.rand((wl.N_LAYERS, wl.N_EXPERTS), device="cuda", generator=g), dim=-1)
    return torch.gather(perms.expand(tokens, -1, -1), 2, ranks)


def _decode(n, rho, g):
    prof = wl.load_profile("nominal", **wl.GEOMETRY["serving"])
    per_token = wl.N_LAYERS * (wl.ATTN_TILES + wl.TOP_K * wl.EXPERT_TILES)
    tokens = -(-n // per_token)
    layer = (torch.arange(wl.N_LAYERS, device="cuda") * wl.LAYER_BYTES)[None, :, None]
    attn = (layer + (torch.arange(wl.ATTN_TILES, device="cuda") * wl.TILE)).expand(tokens, -1, -1)
    tiles = torch.arange(wl.EXPERT_TILES, device="cuda") * wl.TILE
    expert = ((layer + wl.ATTN_BYTES + _top_experts(tokens, g) * wl.EXPERT_BYTES)[..., None] + tiles).reshape(tokens, wl.N_LAYERS, -1)
    off = torch.cat([attn, expert], dim=2).reshape(-1)[:n]
    rec, _ = _records(off, wl.TILE, 0, 4 * prof["t_read_ns"] / (rho * 32 * 8 * 4), g)
    return prof, [(wl.RANGE_BASE, wl.SERVING_RANGE, 3, 0, 0, 0)], rec


def _prefix(n, rho, g, lead=None):
    """Programs of the prefix's KV (all of them, or the last `lead`), then decode steps of 64 requests, until n accesses are had."""
    prof = wl.load_profile("nominal", **wl.GEOMETRY["serving"])
    kib4 = 4 * wl.KIB
    n_prog = wl.KV_BYTES // kib4
    prog = wl.KV_OFFSET + torch.arange(n_prog, device="cuda") * kib4
    prog = prog[:n] if lead is None else prog[n_prog - min(lead, n_prog, n):]
    layer = (torch.arange(wl.N_LAYERS, device="cuda") * wl.LAYER_BYTES)[:, None]
    attn = layer + torch.arange(wl.ATTN_TILES, device="cuda") * wl.TILE
    expert = ((layer + wl.ATTN_BYTES + torch.arange(wl.N_EXPERTS, device="cuda") * wl.EXPERT_BYTES)[..., None]
              + torch.arange(wl.EXPERT_TILES, device="cuda") * wl.TILE).reshape(wl.N_LAYERS, -1)
    kv = (wl.KV_OFFSET + (torch.arange(wl.N_LAYERS, device="cuda") * wl.KV_LAYER_BYTES)[:, None]
          + torch.arange(wl.KV_LAYER_BYTES // wl.TILE, device="cuda") * wl.TILE).repeat(1, 64)
    every = torch.cat([attn, expert, kv], dim=1)
    parts, have = [prog], prog.numel()
    while have < n:
        routed = torch.zeros((wl.N_LAYERS, wl.N_EXPERTS), dtype=torch.bool, device="cuda")
        routed.scatter_(1, _top_experts(64, g).permute(1, 0, 2).reshape(wl.N_LAYERS, -1), True)
        keep = torch.ones(every.shape, dtype=torch.bool, device="cuda")
        keep[:, wl.ATTN_TILES:wl.ATTN_TILES + wl.N_EXPERTS * wl.EXPERT_TILES] = routed.repeat_interleave(wl.EXPERT_TILES, dim=1)
        parts.append(every[keep])
        have += parts[-1].numel()
    off = torch.cat(parts)[:n]
    flags = (torch.arange(n, device="cuda") < prog.numel()).long()
    nbytes = torch.where(flags == 1, kib4, wl.TILE)
    frac = prog.numel() / n if lead is None else 0.02      # (a window run keeps the rate of the whole stream)
    mean_service = frac * prof["t_prog_ns"] + (1.0 - frac) * 4 * prof["t_read_ns"]
    rec, _ = _records(off, nbytes, flags, mean_service / (rho * 32 * 8 * 4), g)
    return prof, [(wl.RANGE_BASE, wl.SERVING_RANGE, 3, 0, 0, 0)], rec


def _capacity(n, rho, g, chunk=16_000_000):
    prof = wl.load_profile("nominal", **wl.GEOMETRY["capacity"])
    rec = torch.empty((n, 3), dtype=torch.int64, device="cuda")
    t0 = None
    for lo in range(0, n, chunk):
        m = min(chunk, n - lo)
        lg = torch.randint(7, 17, (m,), device="cuda", generator=g)               # 128 B ... 64 KiB
        slots = torch.full_like(lg, wl.WEIGHT_BYTES) >> lg
        slot = torch.minimum((torch.rand(m, dtype=torch.float64, device="cuda", generator=g) * slots).long(), slots - 1)
        off = torch.randint(0, wl.CAPACITY_REPLICAS, (m,), device="cuda", generator=g) * wl.CAPACITY_SLOT + (slot << lg)
        _, t0 = _records(off, torch.ones_like(lg) << lg, 0, 1.4 * prof["t_read_ns"] / (rho * 64 * 8 * 4), g, rec[lo:lo + m], t0)
    return prof, [(wl.RANGE_BASE, wl.CAPACITY_RANGE, 3, 1, 0, 0)], rec


def _mixed(n, rho, g):
    """Three ranges with gaps (the last read-only), a tenth of the accesses outside them, a tenth programs, sizes of 64 B to
    64 KiB and odd ones, many of them across pages and stripe units, some issued at the same time."""
    prof = wl.load_profile("nominal", **ODD_GEOMETRY)
    span = 4 * wl.GIB
    ranges = [(wl.RANGE_BASE + 2 * k * span, span, 3 if k < 2 else 1, 0, k, k * span) for k in range(3)]
    where = torch.randint(0, 10, (n,), device="cuda", generator=g)                # 0-3, 4-6, 7-8: the ranges; 9: between them
    slot = torch.where(where < 4, 0, torch.where(where < 7, 2, torch.where(where < 9, 4, 1)))
    lg = torch.randint(6, 17, (n,), device="cuda", generator=g)
    nbytes = (torch.ones_like(lg) << lg) + torch.randint(0, 2, (n,), device="cuda", generator=g) * torch.randint(0, 4096, (n,), device="cuda", generator=g)
    off = slot * span + (torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * (span - 2 * wl.MIB)).long()
    flags = ((torch.rand(n, device="cuda", generator=g) < 0.15) & (where < 7)).long()
    mean_service = 0.1 * prof["t_prog_ns"] * 1.6 + 0.8 * prof["t_read_ns"] * 1.6
    rec, _ = _records(off, nbytes, flags, mean_service / (rho * 12 * 6 * 3), g)
    return prof, ranges, rec


_STREAMS = dict(uniform=_uniform, decode=_decode, prefix=_prefix, capacity=_capacity, mixed=_mixed)


def _ordered(rec, order, g):
    if order == "shuffled":
        return rec[torch.randperm(rec.shape[0], device="cuda", generator=g)]
    if order == "rings":                                   # each record in one of the logs; the logs one after the other
        ring = torch.randint(0, RINGS, (rec.shape[0],), dtype=torch.int16, device="cuda", generator=g)
        return rec[torch.sort(ring, stable=True).indices]
    return rec


# ---- what a user's program has in hand ----------------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _floorplan(channels):
    return wl.package_floorplan(channels=channels)


def _context(prof, ranges, case):
    channels = prof["channels"]
    fp = _floorplan(channels) if channels % 32 == 0 else None
    ctx = hbf.Context(prof, fp)
    for r in ranges:
        ctx.register_range(*r)
    return ctx, fp


def _rom(m, g):
    """A stable 224-state model of m inputs whose temperatures stay some kelvin above ambient."""
    def rand(*shape):
        return torch.rand(shape, dtype=torch.float64, device="cuda", generator=g).cpu().numpy()
    q, _ = np.linalg.qr(rand(ROM_STATES, ROM_STATES) - 0.5)
    decay = 0.5 + 0.48 * rand(ROM_STATES)
    kinds = np.array([hbf.KIND_HBF] * 6 + [hbf.KIND_HBM] * 2 + [hbf.KIND_GPU] * 3, np.int32)
    rom = hbf.Rom((q * decay) @ q.T, q @ (0.01 * rand(ROM_STATES, m)), (0.01 * rand(ROM_OUTPUTS, ROM_STATES)) @ q.T,
                  D=0.001 * rand(ROM_OUTPUTS, m), d=np.full(ROM_OUTPUTS, 35.0))
    return rom, kinds


def _window_edges(rec, windows):
    """Where the windows of 1 ms begin, and the end: the number of accesses is given, so the last window takes what is left."""
    edges = torch.searchsorted(rec[:, 1].contiguous(), torch.arange(windows, device="cuda") * WINDOW_NS)
    return edges.tolist() + [rec.shape[0]]


def _retention(ppb, bpp, disturb_limit, accel):
    return dict(pages_per_block=ppb, blocks_per_plane=bpp, blocks_per_zone=8, max_pec=3000, disturb_limit=disturb_limit,
                l_ref_s=3.15e7, t_ref_c=40.0, ea_ev=1.04, accel=accel, lead_threshold=0.8)


def _accesses_per_window(case):
    return case["rho"] * 32 * 8 * 4 * WINDOW_NS / (0.02 * 375_000 + 0.98 * 80_000 if case["stream"] == "prefix" else 80_000)


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    s = dict(kind=kind)
    if kind in ("windows", "online"):
        per = _accesses_per_window(case)
        n = int(per * case["windows"])
        if case["stream"] == "prefix":                     # the first sixth of the run programs the end of the prefix
            prof, ranges, rec = _prefix(n, case["rho"], g, lead=int(per * case["windows"] / 6))
        else:
            prof, ranges, rec = _STREAMS[case["stream"]](n, case["rho"], g)
        edges = _window_edges(rec, case["windows"])
        ctx, fp = _context(prof, ranges, case)
        sizes = [b - a for a, b in zip(edges, edges[1:])]
        s.update(ctx=ctx, ext=fp["ext_power_w"], n=n)
        if kind == "online":
            rom, kinds = _rom(ctx.n_regions, g)
            ctx.attach_rom(rom, kinds, WINDOW_NS)
            host = [torch.empty(k, dtype=torch.int64, pin_memory=True) for k in (3 * n, n, n, ctx.n_dies * 6)]
            host[0].copy_(rec.reshape(-1))
            acc, comp, stall, stats = host
            s.update(rom=rom, comp=comp, stall=stall, stats=stats,
                     calls=[(acc[3 * a:3 * b], b - a, comp[a:b], stall[a:b]) for a, b in zip(edges, edges[1:])])
            return s
        comp, stall = (torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(2))
        s.update(full=case["full"], rec=rec, comp=comp, stall=stall, stats=torch.empty((case["windows"], ctx.n_dies * 6), dtype=torch.int64, device="cuda"),
                 temps=torch.empty(ctx.n_cells, dtype=torch.float32, device="cuda"))
        if case["full"]:
            ctx.enable_energy_bins(WINDOW_NS, 64)
            ctx.enable_retention(**_retention(64, 64, 256, 2.0e6))
        s["ws"] = ctx.workspace(max(sizes))
        s["calls"] = [(rec[a:b], b - a, comp[a:b], stall[a:b], s["stats"][k]) for k, (a, b) in enumerate(zip(edges, edges[1:]))]
        return s

    prof, ranges, rec = _STREAMS[case["stream"]](case["n"], case["rho"], g)
    prof.update(BATCH_THRESHOLDS)
    rec = _ordered(rec, case.get("order", "issue"), g)
    n = rec.shape[0]
    ctx, fp = _context(prof, ranges, case)
    s.update(ctx=ctx, n=n, rec=rec, ext=None if fp is None else fp["ext_power_w"])
    s["comp"], s["stall"] = (torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(2))
    s["status"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    s["stats"] = torch.empty((2 if kind == "retention" else 1, ctx.n_dies * 6), dtype=torch.int64, device="cuda")
    if kind == "batch":
        if case["bus"]:
            ctx.enable_channel_bus()
        s["ws"] = ctx.workspace(n)
    elif kind == "paged":                                  # room for every access's pages (what a caller that knows its sizes asks for)
        s["parts"] = int(n * 1.7) if case["stream"] == "capacity" else int(n * 4) if case["stream"] == "decode" else int(n * 2.5)
        s["ws"] = torch.empty(ctx.workspace_bytes_paged(n, s["parts"]), dtype=torch.uint8, device="cuda")
    else:
        half = n // 2
        # page reads per block in the first half, on average, times "limit": which blocks the epoch makes eligible
        blocks = 64 * 8 * 4 * 64
        ctx.enable_retention(**_retention(256, 64, max(1, int(case["limit"] * half * 1.4 / blocks)), 1.0))
        s["temps"] = np.full(ctx.n_regions, 60.0)
        s["ws"] = ctx.workspace(n - half)
        s["calls"] = [(rec[a:b], b - a, s["comp"][a:b], s["stall"][a:b], s["status"][a:b], s["stats"][k]) for k, (a, b) in enumerate(((0, half), (half, n)))]
    return s


# ---- one pass ------------------------------------------------------------------------------------------------------------

def _took(rc):
    if rc != 0:
        raise RuntimeError("refused: %s" % hbf.lib().hbf_strerror(rc).decode())


def run(s):
    ctx, kind = s["ctx"], s["kind"]
    ctx.reset()
    if kind == "online":
        s["rom"].reset()
        hot, stats = [], []
        for acc, n, comp, stall in s["calls"]:
            rc, summary = ctx.submit_pinned(acc, n, comp, stall, s["stats"])
            _took(rc)
            stats.append(s["stats"].clone())
            hot.append(ctx.thermal_step(WINDOW_NS, s["ext"]))
        return dict(comp=s["comp"], stall=s["stall"], stats=torch.stack(stats), hot=np.stack(hot), last=summary)
    if kind == "windows":
        last = len(s["calls"]) - 1
        for k, (acc, n, comp, stall, stats) in enumerate(s["calls"]):
            _took(ctx.submit_batch(acc, n, comp, stall, None, stats, s["ws"]))
            ctx.thermal_step(WINDOW_NS, s["ext"], s["temps"] if k == last else None, want_hot=False)
            if s["full"]:
                ctx.retention_advance(WINDOW_NS)
        out = dict(comp=s["comp"], stall=s["stall"], stats=s["stats"], temps=s["temps"], last=ctx.last_result(), busy=ctx.get_busy_until())
        if s["full"]:
            out.update(retention=ctx.retention_totals(), bins=ctx.energy_bins()[1])
        return out
    if kind == "retention":
        for k, (acc, n, comp, stall, status, stats) in enumerate(s["calls"]):
            _took(ctx.submit_batch(acc, n, comp, stall, status, stats, s["ws"]))
            if k == 0:
                ctx.retention_advance(1_000_000_000, s["temps"])
        return dict(comp=s["comp"], stall=s["stall"], status=s["status"], stats=s["stats"], last=ctx.last_result(), retention=ctx.retention_totals())
    if kind == "paged":
        _took(ctx.submit_batch_paged(s["rec"], s["n"], s["parts"], s["comp"], s["stall"], s["status"], s["stats"], s["ws"]))
    else:
        _took(ctx.submit_batch(s["rec"], s["n"], s["comp"], s["stall"], s["status"], s["stats"], s["ws"]))
    if s["ext"] is not None:
        ctx.thermal_step(WINDOW_NS, s["ext"], None, want_hot=False)
    return dict(comp=s["comp"], stall=s["stall"], status=s["status"], stats=s["stats"], last=ctx.last_result())


# ---- what a pass cannot do without ---------------------------------------------------------------------------------------

def work(case):
    """24 B of record in, 8 B of completion and 8 B of stall out, 1 B of status where it is asked for; per thermal step the
    field and its compensation in and out, the cells' five constants and power in, 14 operations per cell and substep; the
    model's matrices once, per model step a multiply and an add per matrix entry."""
    kind = case["kind"]
    if kind in ("windows", "online"):
        n, w = _accesses_per_window(case) * case["windows"], case["windows"]
        if kind == "online":
            entries = (ROM_STATES + ROM_OUTPUTS) * (ROM_STATES + 63)
            return dict(bytes=40.0 * n + 8.0 * entries, flops=2.0 * entries * w)
        blocks = 32 * 8 * 4 * 64 if case["full"] else 0
        return dict(bytes=40.0 * n + w * (GRID_CELLS * 4.0 * 10 + blocks * 17.0), flops=w * GRID_CELLS * 16 * 14.0)
    if kind == "retention":
        return dict(bytes=41.0 * case["n"] + 64 * 8 * 4 * 64 * 20.0, flops=0.0)
    return dict(bytes=41.0 * case["n"], flops=0.0)


def tolerance(case):
    """Times, bytes, counts and energies are whole numbers: the same whatever the order of the work.  Temperatures are float32 with
    a compensation term over some hundred substeps: after 24 and 48 windows they differ from the same steps in float64 by
    3e-8 of their norm and by 8e-8 of a temperature at most."""
    return dict(rel=1.5e-7, max=5e-7, differ=0.0)

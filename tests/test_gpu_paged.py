"""Parity of the page-granular submit (hbf_submit_batch_paged) with the oracle's, through the C ABI, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import hbfo
from paper_2609_09800_b200 import workloads as wl


@pytest.fixture(scope="module")
def hbf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_09800_b200 import build, hbf as mod
    build.build()
    return mod


def contexts(hbf, profile, ranges, path=None):
    g, o = hbf.Context(profile), hbfo.Oracle(profile)
    for r in ranges:
        g.register_range(*r)
        o.register_range(*r)
    if path is not None:
        g.set_path(path)
    return g, o


def capacity_for(acc, page):
    return int((acc["bytes"].astype(np.int64) // page + 2).sum()) if acc.shape[0] else 0


def compare(g, o, acc, page=16384):
    rc_o, c_o, s_o, st_o, ds_o = o.submit(acc, check=False, paged=True)
    rc_g, c_g, s_g, st_g, ds_g = g.submit_host(acc, check=False, parts_capacity=capacity_for(acc, page))
    assert rc_g == rc_o
    if rc_o not in (0, hbfo.E_ACCESS_FAULT):               # refused for the mode: not classified, outputs not defined
        assert np.array_equal(g.get_busy_until(), o.busy_until())
        return rc_g
    assert np.array_equal(st_g, st_o)
    bad = np.flatnonzero(c_g != c_o)
    assert bad.size == 0, "first mismatch at %d: gpu %d oracle %d (%d mismatches)" % (bad[0], c_g[bad[0]], c_o[bad[0]], bad.size)
    assert np.array_equal(s_g, s_o)
    for k in hbfo.DIE_STATS_DTYPE.names:
        assert np.array_equal(ds_g[k], ds_o[k]), k
    assert np.array_equal(g.get_busy_until(), o.busy_until())
    assert np.array_equal(g.get_pending_energy(), o.pending_energy())
    assert g.last_result() == o.last_result()
    return rc_g


@pytest.mark.parametrize("path", ["auto", "sort"])
@pytest.mark.parametrize("n", [1, 2, 2047, 2048, 2049, 50_000, 300_001])
def test_capacity_mode_reads_of_one_to_five_pages(hbf, n, path):
    w = wl.capacity_mode(n=n, seed=n)
    g, o = contexts(hbf, w.profile, w.ranges, hbf.PATH_AUTO if path == "auto" else hbf.PATH_SORT)
    cut = n // 3
    compare(g, o, w.acc[:cut])
    compare(g, o, w.acc[cut:])


@pytest.mark.parametrize("stripe", [16384, 65536])
def test_mixed_sizes_programs_and_unaligned_spans(hbf, stripe):
    rng = np.random.default_rng(stripe)
    n = 40_000
    acc = np.zeros(n, hbfo.ACCESS_DTYPE)
    acc["addr"] = wl.RANGE_BASE + rng.integers(0, 1 << 26, n).astype(np.uint64)
    acc["issue_ns"] = np.sort(rng.integers(0, 400_000_000, n))
    acc["bytes"] = rng.choice([1, 64, 100, 4096, 16384, 20000, 65536, 200_000, 1 << 20], n)
    acc["flags"] = rng.random(n) < 0.1
    prof = wl.load_profile("nominal", **wl.GEOMETRY["tiny"]); prof["stripe_bytes"] = stripe
    for path in (hbf.PATH_AUTO, hbf.PATH_SORT):
        g, o = contexts(hbf, prof, [(wl.RANGE_BASE, wl.GIB, 3, 0, 0, 0)], path)
        compare(g, o, acc[:25_000])
        compare(g, o, acc[25_000:])
    shuffled = acc[rng.permutation(n)]                       # any record order: the sort path
    g, o = contexts(hbf, prof, [(wl.RANGE_BASE, wl.GIB, 3, 0, 0, 0)])
    compare(g, o, shuffled)


def test_statuses_refusal_and_modes(hbf):
    wf, w = wl.mixed_status(9000, seed=6, faults=True), wl.mixed_status(9000, seed=6)
    g, o = contexts(hbf, w.profile, w.ranges)
    assert compare(g, o, wf.acc) == hbfo.E_ACCESS_FAULT    # refused: nothing changes
    compare(g, o, w.acc)                                     # natives, two ranges with gaps
    g.force_mode(hbf.MODE_LIGHT, 700_001); o.force_mode(hbfo.MODE_LIGHT, 700_001)
    compare(g, o, w.acc)
    g.force_mode(hbf.MODE_SEVERE, 700_001); o.force_mode(hbfo.MODE_SEVERE, 700_001)
    assert compare(g, o, w.acc) == hbfo.E_THROTTLED


def test_empty_batch_and_too_small_a_capacity(hbf):
    w = wl.capacity_mode(n=5000, seed=1)
    g, o = contexts(hbf, w.profile, w.ranges)
    compare(g, o, w.acc[:0])
    rc, *_ = g.submit_host(w.acc, check=False, parts_capacity=5000)     # these 5,000 reads have about 7,000 pages
    assert rc == hbf.E_WORKSPACE and not g.get_busy_until().any()
    compare(g, o, w.acc)


# ---- with the energy ledger, the channel bus and retention on: the list of parts is served like any batch of records ----

RET = dict(pages_per_block=4, blocks_per_plane=8, blocks_per_zone=2, max_pec=3, disturb_limit=40,
           l_ref_s=1000.0, t_ref_c=40.0, ea_ev=1.04, accel=1.0, lead_threshold=0.02)


def same_extras(g, o, bins, bus, ret):
    if bins:
        fg, bg = g.energy_bins(); fo, bo = o.energy_bins()
        assert fg == fo
        bad = np.argwhere(bg != bo)
        assert bad.size == 0, "bins: first difference at bin %d die %d: gpu %d oracle %d" % (bad[0][0], bad[0][1], bg[tuple(bad[0])], bo[tuple(bad[0])])
    if bus:
        assert np.array_equal(g.get_bus_busy_until(), o.bus_busy_until())
    if ret:
        bg, bo = g.retention_blocks(), o.retention_blocks()
        for k in ("disturb", "pec", "epoch"):
            assert np.array_equal(bg[k], bo[k]), k
        assert np.allclose(bg["damage"], bo["damage"], rtol=1e-12, atol=0.0)
        assert g.retention_totals() == o.retention_totals()
        assert np.array_equal(g.retention_plan(), o.retention_plan())


def busy_stream(rng, n, t0, gap):
    acc = np.zeros(n, hbfo.ACCESS_DTYPE)
    acc["addr"] = wl.RANGE_BASE + rng.integers(0, 1 << 24, n).astype(np.uint64)
    acc["issue_ns"] = t0 + np.sort(rng.integers(0, gap * n + 1, n))
    acc["bytes"] = rng.choice([64, 4096, 16384, 20000, 65536, 200_000], n)
    acc["flags"] = rng.random(n) < 0.1
    nat = rng.random(n) < 0.05
    acc["addr"][nat] = 0x2000 + 64 * np.arange(int(nat.sum()), dtype=np.uint64)
    return acc


@pytest.mark.parametrize("path", ["auto", "sort"])
@pytest.mark.parametrize("extras", ["bins", "bus", "retention", "bins+bus+retention"])
def test_parts_with_the_ledger_the_bus_and_retention(hbf, extras, path):
    bins, bus, ret = "bins" in extras, "bus" in extras, "retention" in extras
    prof = wl.load_profile("nominal", **wl.GEOMETRY["tiny"])
    g, o = contexts(hbf, prof, [(wl.RANGE_BASE, wl.GIB, 3, 0, 0, 0)], hbf.PATH_AUTO if path == "auto" else hbf.PATH_SORT)
    for x in (g, o):
        if bins:
            x.enable_energy_bins(250_000, 64)
        if bus:
            x.enable_channel_bus()
        if ret:
            x.enable_retention(**RET)
    rng = np.random.default_rng(len(extras))
    t0 = 0
    for n in (1, 4000, 30_000, 2049):
        acc = busy_stream(rng, n, t0, gap=4000)
        assert compare(g, o, acc) == 0
        same_extras(g, o, bins, bus, ret)
        t0 = int(acc["issue_ns"][-1]) + 1
        if ret:                                              # an epoch: disturbed blocks come due, the next batch's parts claim
            g.retention_advance(10**9, np.array([50.0])); o.retention_advance(10**9, np.array([50.0]))
            same_extras(g, o, bins, bus, ret)
    if ret:
        assert o.retention_totals()["claimed"] > 500
    if bus:
        assert o.bus_busy_until().any()
    if bins:
        assert o.energy_bins()[1].any()


def test_a_refused_paged_batch_changes_nothing_with_everything_on(hbf):
    wf = wl.mixed_status(6000, seed=4, faults=True)
    g, o = contexts(hbf, wf.profile, wf.ranges)
    for x in (g, o):
        x.enable_energy_bins(100_000, 64); x.enable_channel_bus(); x.enable_retention(**RET)
    assert compare(g, o, wf.acc) == hbfo.E_ACCESS_FAULT
    same_extras(g, o, True, True, True)
    assert not g.energy_bins()[1].any() and not g.get_bus_busy_until().any() and not g.retention_blocks()["disturb"].any()


# ---- batches in issue order are cut at stripe units, their pages served as one entry (above 8,192 accesses) ----------------

@pytest.mark.parametrize("n", [8_193, 40_003])
@pytest.mark.parametrize("kind", ["inside", "crossing", "programs", "native", "fault", "odd geometry", "queue per die", "one page units", "scaled", "load", "unordered"])
def test_stripe_units_match_the_oracle(hbf, kind, n):
    rng = np.random.default_rng(n)
    geo = dict(channels=8, dies=4, planes=2, page_bytes=16384, stripe_bytes=131072)
    if kind == "odd geometry": geo.update(channels=5, dies=3, planes=3)
    if kind == "queue per die": geo.update(queue_level=1)
    if kind == "one page units": geo.update(stripe_bytes=16384)
    prof = wl.load_profile("nominal", **geo)
    prof.update(read_granule=256)
    ranges = [(wl.RANGE_BASE, 1 << 30, 3, 0, 0, 5 * 16384)]
    g, o = contexts(hbf, prof, ranges)
    acc = np.zeros(n, hbfo.ACCESS_DTYPE)
    cross = kind in ("crossing", "one page units", "native", "fault", "unordered")
    size = rng.choice([1, 300, 16384, 40_000, 65_536, 131_072], n)
    unit = rng.integers(0, 8000, n)
    # inside: a place in the unit that leaves room for the access (the media begins 5 pages into its first unit)
    place = rng.integers(0, 131_072, n) if cross else (rng.random(n) * (131_072 - size + 1)).astype(np.int64)
    acc["addr"] = (wl.RANGE_BASE + (3 + 8 * unit.astype(np.int64)) * 16384 + place).astype(np.uint64)
    acc["bytes"] = size
    acc["flags"] = rng.random(n) < (0.6 if kind == "programs" else 0.1)
    gap = 2000 if kind == "load" else 40_000
    acc["issue_ns"] = np.sort(rng.integers(0, gap * n, n))
    if kind == "unordered": acc["issue_ns"][n // 2] = 0
    if kind == "native": acc["addr"][rng.random(n) < 0.3] = 77
    if kind == "fault": acc["bytes"][n - 3] = 0
    if kind == "scaled":
        g.force_mode(1, 333_333); hbfo.lib().hbfo_force_mode(o._h, 1, 333_333)
    for _ in range(2):
        compare(g, o, acc)
        acc["issue_ns"] += 1000


@pytest.mark.parametrize("kind", ["inside", "last crosses", "natives", "fault", "unordered", "scaled", "several ranges"])
@pytest.mark.parametrize("n", [70_001, 400_003])             # (the pass counts from 400,000 on)
def test_the_first_pass_counts(hbf, kind, n):
    """A batch whose samples all lie inside their stripe units: the pass counts, and where something else turns up in it (or too many pages
    for the caller's room), the call goes on, or is refused, as if that pass had not been."""
    import torch
    rng = np.random.default_rng(n)
    prof = wl.load_profile("nominal", channels=8, dies=4, planes=2, page_bytes=16384, stripe_bytes=65536)
    ranges = [(wl.RANGE_BASE, wl.GIB, 3, 0, 0, 0)] + ([(wl.RANGE_BASE + 2 * wl.GIB, wl.GIB, 1, 0, 1, wl.GIB)] if kind == "several ranges" else [])
    g, o = contexts(hbf, prof, ranges)
    acc = np.zeros(n, hbfo.ACCESS_DTYPE)
    acc["bytes"] = rng.choice([1, 16384, 40_000, 65_536], n)
    acc["addr"] = wl.RANGE_BASE + rng.integers(0, 16_000, n).astype(np.uint64) * np.uint64(65536) + (rng.random(n) * (65_537 - acc["bytes"])).astype(np.uint64)
    acc["issue_ns"] = np.sort(rng.integers(0, 30_000 * n, n))
    acc["flags"] = rng.random(n) < 0.1
    odd = n - 3                                              # (between two of the samples)
    if kind == "last crosses": acc["addr"][odd] = wl.RANGE_BASE + 65_535; acc["bytes"][odd] = 2
    if kind == "natives": acc["addr"][rng.random(n) < 0.3] = 64
    if kind == "fault": acc["bytes"][odd] = 0
    if kind == "unordered": acc["issue_ns"][odd] = 0
    if kind == "scaled": g.force_mode(1, 333_333); hbfo.lib().hbfo_force_mode(o._h, 1, 333_333)
    first = np.zeros(300, hbfo.ACCESS_DTYPE)                 # a small batch before it, whose summary lies on the device
    first["addr"] = wl.RANGE_BASE; first["bytes"] = 64
    compare(g, o, first)
    before = g.get_busy_until()
    d = torch.from_numpy(acc.view(np.int64).reshape(-1)).cuda()
    comp, stall = (torch.full((n,), -1, dtype=torch.int64, device="cuda") for _ in range(2))
    status = torch.full((n,), 9, dtype=torch.uint8, device="cuda")
    off = acc["addr"].astype(np.int64) % 16384
    pages = int(np.where(acc["addr"] < wl.RANGE_BASE, 1, np.maximum(1, (off + acc["bytes"] + 16383) // 16384)).sum())
    last = g.last_result()
    assert g.submit_batch_paged(d, n, pages - 1, comp, stall, status) == hbf.E_WORKSPACE
    assert (comp == -1).all() and (stall == -1).all() and (status == 9).all()
    assert np.array_equal(g.get_busy_until(), before) and g.last_result() == last
    for _ in range(2):
        compare(g, o, acc)
        acc["issue_ns"] += 1000


@pytest.mark.parametrize("n", [400_003, 2_000_001])
@pytest.mark.parametrize("where", ["first tile", "early and in the middle", "everywhere"])
def test_crossings_that_the_samples_miss(hbf, n, where):
    """The blocks of the pass that counts leave on what the 1,024 samples showed, not on what other blocks of it find meanwhile: crossings in
    tiles that are served first, between the samples, a batch twice on one context and one without crossings behind it."""
    rng = np.random.default_rng(n)
    prof = wl.load_profile("nominal", channels=8, dies=4, planes=2, page_bytes=16384, stripe_bytes=65536)
    g, o = contexts(hbf, prof, [(wl.RANGE_BASE, wl.GIB, 3, 0, 0, 0)])
    acc = np.zeros(n, hbfo.ACCESS_DTYPE)
    acc["bytes"] = rng.choice([1, 16384, 40_000, 65_536], n)
    acc["addr"] = wl.RANGE_BASE + rng.integers(0, 16_000, n).astype(np.uint64) * np.uint64(65536) + (rng.random(n) * (65_537 - acc["bytes"])).astype(np.uint64)
    acc["issue_ns"] = np.sort(rng.integers(0, 30_000 * n, n))
    inside = acc.copy()
    odd = {"first tile": np.array([1, 2]), "early and in the middle": np.concatenate([np.arange(5, 3_000, 97), n // 2 + np.arange(0, 3_000, 97)]),
           "everywhere": rng.choice(n, n // 50, replace=False)}[where]
    odd = np.setdiff1d(odd, np.arange(1024) * (n - 1) // 1024)
    acc["addr"][odd] = wl.RANGE_BASE + rng.integers(0, 16_000, len(odd)).astype(np.uint64) * np.uint64(65536) + np.uint64(65_535)
    acc["bytes"][odd] = 2
    for batch in (acc, inside, acc):
        batch = batch.copy()
        batch["issue_ns"] += 1000
        compare(g, o, batch)


@pytest.mark.parametrize("cross", [False, True])
def test_two_threads_share_a_stream_and_a_workspace(hbf, cross):
    """A page-granular batch keeps state in its workspace over its own wait for the device (the first pass's maps of the queues, or where every
    access's parts begin): another context's call, from another thread, on the same stream and scratch comes before or behind all of it."""
    import threading
    import time
    import torch
    n = 500_000
    prof = wl.load_profile("nominal", channels=8, dies=4, planes=2, page_bytes=16384, stripe_bytes=65536)
    sides = []
    for seed, gap in ((1, 30_000), (2, 3_000)):
        rng = np.random.default_rng(seed)
        acc = np.zeros(n, hbfo.ACCESS_DTYPE)
        acc["bytes"] = 65_536 if cross else 16_384
        acc["addr"] = wl.RANGE_BASE + rng.integers(0, 16_000, n).astype(np.uint64) * np.uint64(65536) + (rng.integers(0, 4, n) * 16_384).astype(np.uint64)
        acc["issue_ns"] = np.sort(rng.integers(0, gap * n, n))
        g, o = contexts(hbf, prof, [(wl.RANGE_BASE, wl.GIB, 3, 0, 0, 0)])
        rec = torch.from_numpy(acc.view(np.int64).reshape(-1)).cuda()
        comp, stall = (torch.zeros(n, dtype=torch.int64, device="cuda") for _ in range(2))
        sides.append((g, o, acc, rec, comp, stall))
    ws = torch.empty(sides[0][0].workspace_bytes_paged(n, 5 * n), dtype=torch.uint8, device="cuda")
    codes = [None, None]

    def call(k):
        g, _, _, rec, comp, stall = sides[k]
        codes[k] = g.submit_batch_paged(rec, n, 5 * n, comp, stall, None, None, ws)

    for _ in range(2):
        torch.cuda.synchronize()
        torch.cuda._sleep(400_000_000)                       # (a fifth of a second in which the first call waits and the second comes)
        threads = [threading.Thread(target=call, args=(k,)) for k in range(2)]
        for t in threads:
            t.start()
            time.sleep(0.05)
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        assert codes == [0, 0]
        for g, o, acc, _, comp, stall in sides:
            _, c_o, s_o, *_ = o.submit(acc, paged=True)
            assert np.array_equal(comp.cpu().numpy(), c_o) and np.array_equal(stall.cpu().numpy(), s_o)
            assert np.array_equal(g.get_busy_until(), o.busy_until()) and g.last_result() == o.last_result()


@pytest.mark.parametrize("cross", [False, True])             # (no access crosses a stripe unit: the batch's own records are served)
@pytest.mark.parametrize("n", [5_000, 12_000])
def test_a_throttled_paged_batch_leaves_zeros(hbf, n, cross):
    import torch
    rng = np.random.default_rng(n)
    prof = wl.load_profile("nominal", channels=8, dies=4, planes=2, page_bytes=16384, stripe_bytes=65536)
    g, o = contexts(hbf, prof, [(wl.RANGE_BASE, wl.GIB, 3, 0, 0, 0)])
    acc = np.zeros(n, hbfo.ACCESS_DTYPE)
    acc["addr"] = wl.RANGE_BASE + rng.integers(0, 8_000, n).astype(np.uint64) * np.uint64(65536) + np.uint64(60_000 if cross else 0)
    acc["bytes"] = 40_000
    acc["issue_ns"] = 1000 * np.arange(n)
    compare(g, o, acc)
    d = torch.from_numpy(acc.view(np.int64).reshape(-1)).cuda()
    comp, stall = (torch.full((n,), -1, dtype=torch.int64, device="cuda") for _ in range(2))
    g.force_mode(2, 1_000_000)
    assert g.submit_batch_paged(d, n, 4 * n, comp, stall) == 0 and g.last_result()["code"] == hbf.E_THROTTLED
    assert not comp.any() and not stall.any()


def test_a_stripe_unit_of_pages_whose_service_passes_64_bits(hbf):
    """2^30 pages of one byte per stripe unit at 17 s each: the time of a whole unit has no place in 64 bits, a batch of
    accesses of a few bytes is served all the same."""
    n = 9_000
    prof = wl.load_profile("nominal", channels=2, dies=1, planes=1, page_bytes=1, stripe_bytes=1 << 30)
    prof.update(t_read_ns=1 << 34)
    g, o = contexts(hbf, prof, [(wl.RANGE_BASE, 1 << 34, 3, 0, 0, 0)])
    acc = np.zeros(n, hbfo.ACCESS_DTYPE)
    acc["addr"] = wl.RANGE_BASE + np.random.default_rng(0).integers(0, 1 << 33, n).astype(np.uint64)
    acc["bytes"] = 1 + np.arange(n) % 3
    acc["issue_ns"] = np.arange(n)
    compare(g, o, acc, page=1)

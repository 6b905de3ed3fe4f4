"""The 32-bit form of the in-order pass at the edges of what it holds, against the oracle, bit for bit: a gap in the stream and a
backlog that do not fit 2^31 ns (the tile is served in the 64-bit form), accesses at the end of the range and larger than the
form takes inline, one-way ranges, a record array that does not begin on a 16-byte boundary, refresh claims on top."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import hbfo
from paper_2609_09800_b200 import workloads as wl

BASE, MIB = wl.RANGE_BASE, wl.MIB


@pytest.fixture(scope="module")
def hbf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_09800_b200 import build, hbf as mod
    build.build()
    return mod


def stream(kind, n, rng):
    acc = np.zeros(n, hbfo.ACCESS_DTYPE)
    acc["addr"] = BASE + rng.integers(0, 4096, n).astype(np.uint64) * np.uint64(65536)
    acc["issue_ns"] = 1000 + np.sort(rng.integers(0, 40 * n, n))
    acc["bytes"] = rng.choice([1, 64, 4096, 16384, 40_000], n)
    acc["flags"] = rng.random(n) < 0.2
    if kind == "gap":                                       # inside a tile, and again at its first record
        acc["issue_ns"][n // 2 + 100:] += 5_000_000_000
        acc["issue_ns"][n // 1024 * 1024:] += 3_000_000_000
    elif kind == "backlog":                                 # 3 ms programs on one queue: a tile's 1,024 of them pass 2^31 ns
        hot = np.arange(n) % 8 != 0
        acc["addr"][hot] = BASE; acc["bytes"][hot] = 131_072; acc["flags"][hot] = 1
    elif kind == "edge":                                    # the last 256 KiB of the range, and sizes around the inline bound
        acc["bytes"] = rng.choice([64, 131_071, 131_072, 131_073, 200_000], n)
        acc["addr"] = np.uint64(BASE + 256 * MIB) - acc["bytes"].astype(np.uint64) - (rng.integers(0, 1000, n).astype(np.uint64) if n else 0)
    elif kind == "native":
        out = rng.random(n) < 0.3
        acc["addr"][out] = rng.integers(0, 1 << 40, int(out.sum())).astype(np.uint64)
    return acc


@pytest.mark.parametrize("entries", [0, 2, 6])              # 0: served twice (batches of this size); else the fix-up, with so many head entries
@pytest.mark.parametrize("n", [8_193, 20_001, 65_536])
@pytest.mark.parametrize("kind", ["plain", "gap", "backlog", "edge", "native", "offset", "read only", "program only", "claims", "claims backlog", "neighbours", "queue per die", "claims queue per die", "several ranges", "throttled"])
def test_32_bit_form_matches_the_oracle(hbf, kind, n, entries):
    import torch
    rng = np.random.default_rng(n)
    prof = wl.load_profile("nominal", channels=8, dies=4, planes=2, page_bytes=16384, stripe_bytes=65536, queue_level=int("queue per die" in kind))
    perms = {"read only": 1, "program only": 2}.get(kind, 3)
    g, o = hbf.Context(prof), hbfo.Oracle(prof)
    for c in (g, o):
        c.register_range(BASE, 256 * MIB, perms, 0, 0, 3 * 65536)
        if kind == "several ranges": c.register_range(BASE + 512 * MIB, 64 * MIB, 3, 0, 0, 512 * MIB)
        if kind == "throttled": c.force_mode(hbfo.MODE_LIGHT, 600_000)
        if "claims" in kind:
            c.enable_retention(pages_per_block=16, blocks_per_plane=32, blocks_per_zone=8, max_pec=3000, disturb_limit=0,
                               l_ref_s=1.0, t_ref_c=40.0, ea_ev=1.04, accel=1.0, lead_threshold=0.5)
            c.retention_advance(1_000_000_000, [40.0])      # every block becomes eligible: 32,768 quanta
    if entries: g.set_head_entries(entries)
    acc = stream(kind.split()[-1] if "backlog" in kind else kind, n, rng)
    if kind == "neighbours":                                # walks along the stripe units; nearly every tile is served again
        acc["addr"] = BASE + (np.arange(n) % 4000).astype(np.uint64) * np.uint64(65536)
    if perms != 3:
        acc["flags"] = perms - 1
    for batch in range(2):                                  # the second one enters on the queues the first one left
        _, c_o, s_o, st_o, ds_o = o.submit(acc)
        if kind == "offset":
            d = torch.zeros(3 * n + 1, dtype=torch.int64, device="cuda")
            d[1:] = torch.from_numpy(acc.view(np.int64).reshape(-1)).cuda()
            comp, stall = (torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(2))
            status = torch.empty(n, dtype=torch.uint8, device="cuda"); ds = torch.empty(g.n_dies * 6, dtype=torch.int64, device="cuda")
            assert g.submit_batch(d[1:], n, comp, stall, status, ds) == 0 and g.last_result()["code"] == 0
            c_g, s_g, st_g, ds_g = comp.cpu().numpy(), stall.cpu().numpy(), status.cpu().numpy(), ds.cpu().numpy().view(hbf.DIE_STATS_DTYPE)
        else:
            _, c_g, s_g, st_g, ds_g = g.submit_host(acc)
        assert np.array_equal(st_g, st_o) and np.array_equal(c_g, c_o) and np.array_equal(s_g, s_o)
        assert all(np.array_equal(ds_g[f], ds_o[f]) for f in hbfo.DIE_STATS_DTYPE.names)
        assert np.array_equal(g.get_busy_until(), o.busy_until()) and g.last_result() == o.last_result()
        if "claims" in kind:
            bg, bo = g.retention_blocks(), o.retention_blocks()
            assert np.array_equal(bg["disturb"], bo["disturb"]) and g.retention_totals() == o.retention_totals()
        acc["issue_ns"] += 50_000


@pytest.mark.parametrize("declared", [False, True])
def test_large_batches_of_changing_loads(hbf, declared):
    """Too large for the host to tell whether their tiles are served twice: far behind, nearly idle and back, on queues that
    start idle and on what the batch before left; the same as without measurements, where nothing is decided."""
    import torch
    n = 19_600_001                                           # fills a wave; 64 queues: above what is always served twice
    prof = wl.load_profile("nominal", **wl.GEOMETRY["tiny"])
    gen = torch.Generator(device="cuda"); gen.manual_seed(3)
    rec = torch.empty((n, 3), dtype=torch.int64, device="cuda")
    rec[:, 0] = BASE + 4096 * torch.randint(0, 1 << 18, (n,), device="cuda", generator=gen)
    gaps = torch.randint(0, 1250, (n,), device="cuda", generator=gen)
    rec[:, 2] = 4096
    sides = []
    for measured in (True, False):
        g = hbf.Context(prof)
        g.register_range(BASE, 1 << 30)
        g.set_tile_balance(measured)
        if declared: g.set_path(hbf.PATH_INORDER)
        sides.append((g, [torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(2)], torch.empty(n, dtype=torch.uint8, device="cuda")))
    for turn, (load, reset) in enumerate([(3, True), (0.3, True), (3, True), (3, True), (0.3, False), (0.3, False), (0.9, True), (0.3, True), (3, True)]):
        rec[:, 1] = torch.cumsum((gaps.double() / load).long(), 0) + (0 if reset else 10_000_000)
        for g, out, status in sides:
            if reset: g.reset()
            assert g.submit_batch(rec, n, *out, status) == 0
        (a, oa, sa), (b, ob, sb) = sides
        assert a.last_result() == b.last_result() and a.last_result()["code"] == 0
        assert torch.equal(oa[0], ob[0]) and torch.equal(oa[1], ob[1]) and torch.equal(sa, sb), turn
        assert np.array_equal(a.get_busy_until(), b.get_busy_until()) and np.array_equal(a.get_pending_energy(), b.get_pending_energy())

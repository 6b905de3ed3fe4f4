"""Batches out of issue order on the automatic path: brought into order in buckets by issue time and served by the in-order
kernels, or handed to the radix sort where the times do not spread; against the oracle, bit for bit."""
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


@pytest.mark.parametrize("n", [8_193, 24_575, 24_577, 100_003, 200_003])
@pytest.mark.parametrize("kind", ["shuffled", "rings", "ties", "bunched", "one time", "long span", "negative", "natives", "fault", "late", "long service", "three ranges"])
def test_unordered_batches_match_the_oracle(hbf, kind, n):
    rng = np.random.default_rng(n)
    w = wl.capacity_mode(n=n, seed=n, rho=0.6)
    ranges = w.ranges if kind != "three ranges" else [(wl.RANGE_BASE, 1 << 39, 3, 0, 0, 0), (wl.RANGE_BASE + (1 << 39), 1 << 38, 3, 0, 0, 1 << 40), (wl.RANGE_BASE + (3 << 38), 1 << 39, 1, 0, 0, 1 << 41)]
    g, o = hbf.Context(w.profile), hbfo.Oracle(w.profile)
    for r in ranges:
        g.register_range(*r); o.register_range(*r)
    acc = w.acc.copy()
    acc["flags"][:n // 2] = (rng.random(n // 2) < 0.1) & (acc["addr"][:n // 2] < wl.RANGE_BASE + (1 << 39))
    if kind == "ties": acc["issue_ns"] //= 40_000                    # about forty records at a time and 1/64 of the bins of a bucket
    if kind == "bunched": acc["issue_ns"][n // 2:] = acc["issue_ns"][n // 2] + np.arange(n - n // 2) // 500
    if kind == "one time": acc["issue_ns"][1:] = 77
    if kind == "long span": acc["issue_ns"] *= 1 + (1 << 46) // int(acc["issue_ns"][-1]) // 2
    order = rng.permutation(n) if kind != "rings" else np.argsort(rng.integers(0, 148, n), kind="stable")
    if kind == "late":                                              # one record out of place: the samples do not see it
        order = np.arange(n); order[[n // 3, n // 3 + 700]] = order[[n // 3 + 700, n // 3]]
    acc = acc[order]
    if kind == "negative": acc["issue_ns"][5] = -3
    if kind == "natives": acc["addr"][rng.random(n) < 0.3] = 4096
    if kind == "fault": acc["bytes"][n - 2] = 0
    if kind == "long service": acc["bytes"][n // 2] = 1 << 31; acc["flags"][n // 2] = 1; acc["addr"][n // 2] = wl.RANGE_BASE
    for batch in range(2):
        rc_o, c_o, s_o, st_o, ds_o = o.submit(acc, check=False)
        rc_g, c_g, s_g, st_g, ds_g = g.submit_host(acc, check=False)
        assert rc_g == rc_o and np.array_equal(st_g, st_o) and np.array_equal(c_g, c_o) and np.array_equal(s_g, s_o)
        assert all(np.array_equal(ds_g[f], ds_o[f]) for f in hbfo.DIE_STATS_DTYPE.names)
        assert np.array_equal(g.get_busy_until(), o.busy_until()) and g.last_result() == o.last_result()
        assert np.array_equal(g.get_pending_energy(), o.pending_energy())
        if rc_o == 0:
            assert np.array_equal(g.queue_order(n), o.last_order())
        acc["issue_ns"] += 10_000


@pytest.mark.parametrize("reset", [False, True])
def test_the_served_order_after_batches_of_other_routes(hbf, reset):
    """A large batch out of order, then small ones: the order asked for is that of the last batch, or there is none."""
    w = wl.capacity_mode(n=28_000, seed=5, rho=0.6)
    g, o = hbf.Context(w.profile), hbfo.Oracle(w.profile)
    for r in w.ranges:
        g.register_range(*r); o.register_range(*r)
    ws = g.workspace(20_000)
    rng = np.random.default_rng(1)
    for lo, hi, ordered in ((0, 20_000, False), (20_000, 24_000, False), (24_000, 28_000, True), (0, 20_000, False), (0, 20_000, True)):
        acc = w.acc[lo:hi] if ordered else w.acc[lo:hi][rng.permutation(hi - lo)]
        o.submit(acc); g.submit_host(acc)
        if ordered:
            with pytest.raises(hbf.HbfError):
                g.queue_order(hi - lo, ws)
        else:
            assert np.array_equal(g.queue_order(hi - lo, ws), o.last_order())
            assert np.array_equal(g.queue_order(hi - lo, ws), o.last_order())       # (asking does not spoil it)
        if reset:
            g.reset(); o.reset()


@pytest.mark.parametrize("n", [8_193, 100_003])
@pytest.mark.parametrize("kind", ["any 64 bits", "both ends", "one negative sample", "one late sample"])
def test_issue_times_outside_their_limits_are_refused(hbf, kind, n):
    """Records that the begin kernel's samples hold: their span has no place in the arithmetic that spreads a batch."""
    w = wl.capacity_mode(n=n, seed=n, rho=0.6)
    g, o = hbf.Context(w.profile), hbfo.Oracle(w.profile)
    for r in w.ranges:
        g.register_range(*r); o.register_range(*r)
    rng = np.random.default_rng(n)
    good = w.acc[rng.permutation(n)]
    acc = good.copy()
    if kind == "any 64 bits": acc["issue_ns"] = rng.integers(-(1 << 63), (1 << 63) - 1, n, endpoint=True)
    if kind == "both ends": acc["issue_ns"][[0, 1]] = (1 << 63) - 1, -(1 << 63)
    if kind == "one negative sample": acc["issue_ns"][0] = -1
    if kind == "one late sample": acc["issue_ns"][0] = 1 << 47
    bad = (acc["issue_ns"] < 0) | (acc["issue_ns"] >= 1 << 47)
    rc, c, s, st, ds = g.submit_host(acc, check=False)
    assert rc == hbfo.E_ACCESS_FAULT and g.last_result()["n_fault"] == int(bad.sum()) and not c.any() and not s.any()
    assert np.array_equal(st, np.where(bad, 4, 1)) and not g.get_busy_until().any()      # 4: unsupported, 1: modeled
    _, c_o, s_o, *_ = o.submit(good)
    _, c, s, *_ = g.submit_host(good)
    assert np.array_equal(c, c_o) and np.array_equal(s, s_o)


@pytest.mark.parametrize("n", [9_000, 100_003])
@pytest.mark.parametrize("stage", [1, 2])
def test_a_wait_that_runs_out_gives_the_batch_up(hbf, stage, n):
    """One share of the records (or of the results) is silent (test support of the library: nothing stalls for real): outputs are
    zeroed, queues and energies untouched, the context refuses batches until it is reset."""
    w = wl.capacity_mode(n=n, seed=n, rho=0.6)
    g, o = hbf.Context(w.profile), hbfo.Oracle(w.profile)
    for r in w.ranges:
        g.register_range(*r); o.register_range(*r)
    acc = w.acc[np.random.default_rng(n).permutation(n)]
    g.submit_host(w.acc[:5000]); o.submit(w.acc[:5000])
    busy0, pend0 = g.get_busy_until(), g.get_pending_energy()
    g.debug_wait_test(poll_limit=200, stage=stage, tile=3)
    for silent in (True, False):                             # the switch off again: the context stays poisoned
        rc, c, s, _, ds = g.submit_host(acc, check=False)
        assert rc == hbf.E_TIMEOUT and not c.any() and not s.any() and not any(ds[f].any() for f in hbfo.DIE_STATS_DTYPE.names)
        assert np.array_equal(g.get_busy_until(), busy0) and np.array_equal(g.get_pending_energy(), pend0)
        with pytest.raises(hbf.HbfError):
            g.queue_order(n)
        g.debug_wait_test()
    g.reset(); o.reset()
    for _ in range(2):
        _, c_o, s_o, _, ds_o = o.submit(acc)
        _, c, s, _, ds = g.submit_host(acc)
        assert np.array_equal(c, c_o) and np.array_equal(s, s_o) and all(np.array_equal(ds[f], ds_o[f]) for f in hbfo.DIE_STATS_DTYPE.names)
        assert np.array_equal(g.get_busy_until(), o.busy_until()) and g.last_result() == o.last_result()
        assert np.array_equal(g.queue_order(n), o.last_order())


def test_a_bus_that_cannot_take_a_batch_out_of_order(hbf):
    """Its last completion passes 2^47 ns: refused before anything is given back or committed."""
    w = wl.capacity_mode(n=30_000, seed=9, rho=0.6)
    g, o = hbf.Context(w.profile), hbfo.Oracle(w.profile)
    for r in w.ranges:
        g.register_range(*r); o.register_range(*r)
    g.enable_channel_bus(); o.enable_channel_bus()
    acc = w.acc[np.random.default_rng(3).permutation(30_000)]
    late = acc.copy(); late["issue_ns"] += (1 << 47) - 1 - int(late["issue_ns"].max())
    rc, c, s, _, ds = g.submit_host(late, check=False)
    assert rc == -1 and not c.any() and not s.any() and not ds["n_read"].any() and not g.get_busy_until().any() and not g.get_bus_busy_until().any()
    _, c_o, s_o, *_ = o.submit(acc)
    _, c, s, *_ = g.submit_host(acc)
    assert np.array_equal(c, c_o) and np.array_equal(s, s_o) and np.array_equal(g.get_bus_busy_until(), o.bus_busy_until())


@pytest.mark.parametrize("n", [9_000, 60_001, 300_000])
@pytest.mark.parametrize("per", [2, 63, 65, 300, 699, 1_100, 2_047, 5_000])
def test_records_that_share_their_issue_times(hbf, per, n):
    """Ticks of so many records each, around what a bin once held, what a bucket holds, and where the radix sort takes over."""
    w = wl.capacity_mode(n=n, seed=n, rho=0.6)
    g, o = hbf.Context(w.profile), hbfo.Oracle(w.profile)
    for r in w.ranges:
        g.register_range(*r); o.register_range(*r)
    acc = w.acc.copy()
    acc["issue_ns"] = np.arange(n) // per * (per * 40) + 7
    acc = acc[np.random.default_rng(per).permutation(n)]
    for _ in range(2):
        _, c_o, s_o, st_o, _ = o.submit(acc)
        _, c, s, st, _ = g.submit_host(acc)
        assert np.array_equal(c, c_o) and np.array_equal(s, s_o) and np.array_equal(st, st_o) and g.last_result() == o.last_result()
        assert np.array_equal(g.queue_order(n), o.last_order())

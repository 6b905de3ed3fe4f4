"""Workspaces of the size that the sort path needs are taken on every path, whatever more hbf_workspace_bytes asks for."""
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


def up(v):
    return (v + 255) // 256 * 256


def least(g, hbf, n, capacity=None):
    """The smallest workspace of a context without the bus, as the declared path asks for it."""
    g.set_path(hbf.PATH_INORDER)
    b = g.workspace_bytes(n) if capacity is None else g.workspace_bytes_paged(n, capacity)
    g.set_path(hbf.PATH_AUTO)
    return b


@pytest.mark.parametrize("order", ["issue", "shuffled", "late"])
@pytest.mark.parametrize("bus", [False, True])
@pytest.mark.parametrize("n", [4_000, 8_193, 60_001])
def test_least_workspace(hbf, n, bus, order):
    import torch
    w = wl.capacity_mode(n=n, seed=n, rho=0.6)
    g, o = hbf.Context(w.profile), hbfo.Oracle(w.profile)
    for r in w.ranges:
        g.register_range(*r); o.register_range(*r)
    need = least(g, hbf, n)
    assert (g.workspace_bytes(n) > need) == (n > 8_192)     # small batches have no use for the arrays that order a batch
    if bus:
        g.enable_channel_bus(); o.enable_channel_bus()
        need += up(4 * n)
    acc = w.acc
    if order == "shuffled": acc = acc[np.random.default_rng(n).permutation(n)]
    if order == "late": acc = acc.copy(); acc[[n // 3, n // 3 + 700]] = acc[[n // 3 + 700, n // 3]]
    rec = torch.from_numpy(acc.view(np.int64).reshape(-1).copy()).cuda()
    comp, stall = (torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(2))
    status = torch.empty(n, dtype=torch.uint8, device="cuda")
    guard = torch.full((need + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    assert g.submit_batch(rec, n, comp, stall, status, None, guard[:need - 256]) == -5
    for _ in range(2):
        assert g.submit_batch(rec, n, comp, stall, status, None, guard[:need]) == 0
        _, c_o, s_o, st_o, _ = o.submit(acc)
        assert g.last_result() == o.last_result()
        assert np.array_equal(comp.cpu().numpy(), c_o) and np.array_equal(stall.cpu().numpy(), s_o) and np.array_equal(status.cpu().numpy(), st_o)
        if order != "issue" and not bus:
            assert np.array_equal(g.queue_order(n, guard[:need]), o.last_order())
    assert bool((guard[need:] == 0xA5).all())               # nothing past its end
    assert np.array_equal(g.get_busy_until(), o.busy_until())
    if bus:
        assert np.array_equal(g.get_bus_busy_until(), o.bus_busy_until())


@pytest.mark.parametrize("order", ["issue", "shuffled"])
def test_least_workspace_of_the_page_granular_submit(hbf, order):
    import torch
    n = 20_001
    w = wl.capacity_mode(n=n, seed=3, rho=0.4)
    g, o = hbf.Context(w.profile), hbfo.Oracle(w.profile)
    for r in w.ranges:
        g.register_range(*r); o.register_range(*r)
    acc = w.acc if order == "issue" else w.acc[np.random.default_rng(1).permutation(n)]
    need = least(g, hbf, n, 3 * n)
    assert g.workspace_bytes_paged(n, 3 * n) > need
    rec = torch.from_numpy(acc.view(np.int64).reshape(-1).copy()).cuda()
    comp, stall = (torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(2))
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    assert g.submit_batch_paged(rec, n, 3 * n, comp, stall, None, None, ws[:need - 256]) == -5
    for _ in range(2):
        assert g.submit_batch_paged(rec, n, 3 * n, comp, stall, None, None, ws) == 0
        _, c_o, s_o, *_ = o.submit(acc, paged=True)
        assert g.last_result() == o.last_result() and np.array_equal(comp.cpu().numpy(), c_o) and np.array_equal(stall.cpu().numpy(), s_o)


@pytest.mark.parametrize("order", ["issue", "shuffled"])
@pytest.mark.parametrize("n", [500, 8_192])
def test_small_batches_that_the_cluster_does_not_take(hbf, n, order):
    """One die of 300 planes: more queues than a block of the small route serves, fewer records than are ordered in buckets."""
    prof = wl.load_profile("nominal", channels=1, dies=1, planes=300, page_bytes=16384, stripe_bytes=16384)
    g, o = hbf.Context(prof), hbfo.Oracle(prof)
    g.register_range(wl.RANGE_BASE, wl.GIB, 3, 0, 0, 0); o.register_range(wl.RANGE_BASE, wl.GIB, 3, 0, 0, 0)
    rng = np.random.default_rng(n)
    acc = np.zeros(n, hbfo.ACCESS_DTYPE)
    acc["addr"] = wl.RANGE_BASE + rng.integers(0, 1 << 29, n).astype(np.uint64)
    acc["issue_ns"], acc["bytes"] = 500 * np.arange(n), 4096
    if order == "shuffled": acc = acc[rng.permutation(n)]
    for _ in range(2):
        _, c_o, s_o, *_ = o.submit(acc)
        _, c, s, *_ = g.submit_host(acc)
        assert np.array_equal(c, c_o) and np.array_equal(s, s_o) and g.last_result() == o.last_result()

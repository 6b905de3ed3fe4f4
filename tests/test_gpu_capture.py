"""Batches captured into a CUDA graph: every replay serves the batch again on the queues the one before left."""
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


class Captured:
    """A context on a stream of its own, a device copy of a batch, and the batch as a graph."""

    def __init__(self, hbf, acc, profile, ranges):
        import torch
        self.torch, self.n = torch, len(acc)
        self.stream = torch.cuda.Stream()
        self.g, self.o = hbf.Context(profile, stream=self.stream), hbfo.Oracle(profile)
        for r in ranges:
            self.g.register_range(*r); self.o.register_range(*r)
        self.acc = torch.from_numpy(acc.view(np.int64).reshape(-1).copy()).cuda()
        self.comp, self.stall = (torch.zeros(self.n, dtype=torch.int64, device="cuda") for _ in range(2))
        self.ws = self.g.workspace(self.n)
        self.graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()

    def submit(self):
        assert self.g.submit_batch(self.acc, self.n, self.comp, self.stall, None, None, self.ws) == 0

    def capture(self):
        with self.torch.cuda.graph(self.graph, stream=self.stream):
            self.submit()

    def replay(self):
        with self.torch.cuda.stream(self.stream):
            self.graph.replay()


@pytest.mark.parametrize("n", [4_000, 20_000])
def test_the_summary_is_that_of_the_last_replay(hbf, n):
    w = wl.capacity_mode(n=n, seed=n)
    t = Captured(hbf, w.acc, w.profile, w.ranges)
    t.capture()
    for turn in range(4):
        t.submit() if turn == 2 else t.replay()             # (one of them not from the graph)
        _, c_o, s_o, *_ = t.o.submit(w.acc)
        assert t.g.last_result() == t.o.last_result()
        assert np.array_equal(t.comp.cpu().numpy(), c_o) and np.array_equal(t.stall.cpu().numpy(), s_o)


@pytest.mark.parametrize("n", [4_000, 20_000])
def test_a_capture_between_two_calls(hbf, n):
    """The batch before it is sorted by its last kernel: what is captured does not follow that one, the call behind the capture does."""
    import torch
    w = wl.capacity_mode(n=n, seed=n)
    t = Captured(hbf, w.acc, w.profile, w.ranges)
    wl_late = wl.capacity_mode(n=150_000, seed=1)
    late = wl_late.acc.copy(); late[[70_000, 70_900]] = late[[70_900, 70_000]]
    rec = torch.from_numpy(late.view(np.int64).reshape(-1).copy()).cuda()
    comp, stall = (torch.empty(150_000, dtype=torch.int64, device="cuda") for _ in range(2))
    ws = torch.empty(t.g.workspace_bytes(150_000), dtype=torch.uint8, device="cuda")
    t.ws = ws
    torch.cuda.synchronize()
    for turn in range(3):
        assert t.g.submit_batch(rec, 150_000, comp, stall, None, None, ws) == 0
        t.o.submit(late)
        t.graph = torch.cuda.CUDAGraph()
        t.capture()
        t.submit()
        _, c_o, s_o, *_ = t.o.submit(w.acc)
        assert t.g.last_result() == t.o.last_result() and np.array_equal(t.comp.cpu().numpy(), c_o) and np.array_equal(t.stall.cpu().numpy(), s_o)
        t.replay()
        _, c_o, *_ = t.o.submit(w.acc)
        assert t.g.last_result() == t.o.last_result() and np.array_equal(t.comp.cpu().numpy(), c_o)


@pytest.mark.parametrize("entries", [0, 4])
def test_a_captured_batch_that_fills_a_wave(hbf, entries):
    """Large enough for tile sizes from measurements, which come from the host: replays agree with a context that is not captured."""
    import torch
    n = 19_600_003
    w = wl.capacity_mode(n=n, seed=7, rho=0.5)
    t = Captured(hbf, w.acc, w.profile, w.ranges)
    with torch.cuda.stream(t.stream):
        other = hbf.Context(w.profile, stream=t.stream)
    for r in w.ranges:
        other.register_range(*r)
    if entries:
        t.g.set_head_entries(entries)
    comp, stall = (torch.zeros(n, dtype=torch.int64, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    t.capture()
    for turn in range(3):
        t.replay()
        assert other.submit_batch(t.acc, n, comp, stall, None, None, other.workspace(n)) == 0
        torch.cuda.synchronize()
        assert torch.equal(t.comp, comp) and torch.equal(t.stall, stall) and t.g.last_result() == other.last_result()
        t.submit()                                          # and one that is not from the graph, on the queues the replay left
        other.submit_batch(t.acc, n, comp, stall, None, None, other.workspace(n))
        torch.cuda.synchronize()
        assert torch.equal(t.comp, comp) and np.array_equal(t.g.get_busy_until(), other.get_busy_until())


@pytest.mark.parametrize("paged", [0, 1, 2])
def test_the_served_order_of_a_replay_behind_page_granular_batches(hbf, paged):
    """What hbf_queue_order reads of a batch lies where a graph captured before left it, whatever page-granular batches (large enough that
    their first pass counts) came between the capture and the replay."""
    import torch
    n, m = 20_000, 400_003
    w = wl.capacity_mode(n=n, seed=n, rho=0.6)
    shuffled = w.acc[np.random.default_rng(4).permutation(n)]
    t = Captured(hbf, shuffled, w.profile, w.ranges)
    inside = wl.capacity_mode(n=m, seed=5, rho=0.4).acc.copy()
    inside["addr"] -= inside["addr"] % np.uint64(w.profile["stripe_bytes"])
    inside["bytes"] = 4096
    rec = torch.from_numpy(inside.view(np.int64).reshape(-1).copy()).cuda()
    comp, stall = (torch.empty(m, dtype=torch.int64, device="cuda") for _ in range(2))
    ws = torch.empty(t.g.workspace_bytes_paged(m, m), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    t.capture()
    for turn in range(2):
        for _ in range(paged):
            assert t.g.submit_batch_paged(rec, m, m, comp, stall, None, None, ws) == 0
            t.o.submit(inside, paged=True)
            with pytest.raises(hbf.HbfError):
                t.g.queue_order(m, ws)                       # (served in order)
        t.replay()
        _, c_o, *_ = t.o.submit(shuffled)
        assert t.g.last_result() == t.o.last_result() and np.array_equal(t.comp.cpu().numpy(), c_o)
        assert np.array_equal(t.g.queue_order(n, t.ws), t.o.last_order())

"""The fused kernels clear the workspace's control block themselves: whatever is in it before a call, the call is exact."""
import numpy as np
import pytest
import torch

import helpers
import oracle
import test_gpu_threshold as thr
from paper_2104_01981_b200 import api
from helpers import GpuWorker, bits, check_topk_against_oracle, to_np_u32
from test_gpu_threshold import _built, randn   # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu

ONE, MANY = [5_000_003], [300_000, 5, 1_500_001, 0, 64, 700_003, 4097]


class DirtyWorker(GpuWorker):
    def step(self, g):
        self.ws.view(torch.uint8).random_(0, 256)
        super().step(g)


@pytest.fixture
def dirty(monkeypatch):
    monkeypatch.setattr(helpers, "GpuWorker", DirtyWorker)
    monkeypatch.setattr(thr, "GpuWorker", DirtyWorker)


@pytest.mark.parametrize("sizes", [[1], [4096], [70_001], ONE, [12_000_000], MANY], ids=lambda s: "%d_%d" % (len(s), sum(s)))
@pytest.mark.parametrize("options", [{}, {api.GC_OPT_SAMPLE_RANK_PERMILLE: 30}, {api.GC_OPT_CANDIDATE_CAPACITY: 100}],
                         ids=["plain", "starved", "overflow"])
def test_topk_from_a_dirty_workspace(dirty, sizes, options):
    n = sum(sizes)
    check_topk_against_oracle(sizes, 0.01, [randn(n, 31 * n + s) for s in range(2)], options=options)


@pytest.mark.parametrize("sizes", [[70_001], ONE, MANY], ids=lambda s: "%d_%d" % (len(s), sum(s)))
@pytest.mark.parametrize("ties", [False, True], ids=["plain", "overflow"])
def test_threshold_from_a_dirty_workspace(dirty, sizes, ties):
    n = sum(sizes)
    # (equal magnitudes everywhere: every element is a hit, the hit lists overflow)
    grads = [torch.full((n,), 0.25) if ties else randn(n, 37 * n + s) for s in range(2)]
    thr.check_threshold(sizes, 0.01, grads, cap_factor=2.0)


# (plans of these sizes are taken fold first; starved: the redo starts from whatever is in the workspace, too)
FOLD_ONE, FOLD_MANY = [13_000_003], [300_000, 5, 1_500_001, 0, 64, 11_000_003, 4097]


@pytest.mark.parametrize("sizes", [FOLD_ONE, FOLD_MANY], ids=["one", "many"])
@pytest.mark.parametrize("opts", [{}, {api.GC_OPT_SAMPLE_RANK_PERMILLE: 30}, {api.GC_OPT_CANDIDATE_CAPACITY: 100}],
                         ids=["plain", "starved", "overflow"])
def test_threshold_fold_first_from_a_dirty_workspace(dirty, monkeypatch, sizes, opts):
    class WithOptions(api.Plan):
        def __init__(self, *a, **k):
            super().__init__(*a, **k)
            for opt, value in opts.items():
                self.set_option(opt, value)
    monkeypatch.setattr(thr.api, "Plan", WithOptions)
    plan, w = thr.check_threshold(sizes, 0.002, [randn(sum(sizes), 41 + s) for s in range(2)])
    assert (plan.last_counters(w.ws)[1:] == (0, 0)) == (not opts)


@pytest.mark.parametrize("mode,MANY,starved", [(api.GC_TOPK, MANY, False), (api.GC_THRESHOLD, MANY, False), (api.GC_THRESHOLD, FOLD_MANY, False),
                                               (api.GC_THRESHOLD, FOLD_MANY, True)], ids=["topk", "threshold", "fold_first", "fold_first_starved"])
def test_workers_from_dirty_workspaces(mode, MANY, starved):
    """Three workers in one launch on dirty workspaces give what three calls on zeroed ones give."""
    plan, n = api.Plan(MANY, 0.01 if MANY is not FOLD_MANY else 0.002, mode=mode, device=0), sum(MANY)
    if starved:
        plan.set_option(api.GC_OPT_SAMPLE_RANK_PERMILLE, 30)
    a, b = ([GpuWorker(plan) for _ in range(3)] for _ in range(2))
    for step in range(2):
        gs = [randn(n, 1000 * step + w).cuda() for w in range(3)]
        for wk in a:
            wk.ws.view(torch.uint8).random_(0, 256)
        plan.compress_workers(gs, [w.residual for w in a], [w.idx for w in a], [w.val for w in a], [w.count for w in a], [w.ws for w in a])
        for w in range(3):
            b[w].ws.zero_()
            plan.compress(gs[w], b[w].residual, b[w].idx, b[w].val, b[w].count, b[w].ws)
            a[w].check_status()
            assert torch.equal(a[w].count, b[w].count) and torch.equal(a[w].residual, b[w].residual)
            live = torch.cat([torch.arange(o, o + c) for o, c in zip(plan.tensor_out_offset(), b[w].count.tolist())])
            assert torch.equal(a[w].idx.cpu()[live], b[w].idx.cpu()[live])
            assert np.array_equal(to_np_u32(a[w].val.cpu()[live]), to_np_u32(b[w].val.cpu()[live]))


@pytest.mark.parametrize("sizes", [[300_000], ONE, MANY[:3]], ids=["direct", "one", "many"])
def test_call_that_clears_captured_in_a_graph(sizes):
    plan, n = api.Plan(sizes, 0.01, device=0), sum(sizes)
    wk, ks, r_cpu = GpuWorker(plan), plan.tensor_k(), np.zeros(sum(sizes), np.float32)
    g_dev, side, graph = torch.zeros(n, device="cuda"), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    GpuWorker(plan).step(g_dev)                             # (kernels are loaded)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        plan.compress(g_dev, wk.residual, wk.idx, wk.val, wk.count, wk.ws, side)
    for s in range(2):
        g = randn(n, 50 + s)
        g_dev.copy_(g)
        wk.ws.view(torch.uint8).random_(0, 256)
        graph.replay()
        wk.check_status()
        oi, ov = oracle.topk_compress_tensors(sizes, ks, g.numpy(), r_cpu)
        assert np.array_equal(to_np_u32(wk.idx[:sum(ks)]), oi) and np.array_equal(to_np_u32(wk.val[:sum(ks)]), bits(ov))
        assert np.array_equal(to_np_u32(wk.residual[:n]), bits(r_cpu))

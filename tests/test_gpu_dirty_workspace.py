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


@pytest.mark.parametrize("mode", [api.GC_TOPK, api.GC_THRESHOLD], ids=["topk", "threshold"])
def test_workers_from_dirty_workspaces(mode):
    """Three workers in one launch on dirty workspaces give what three calls on zeroed ones give."""
    plan, n = api.Plan(MANY, 0.01, mode=mode, device=0), sum(MANY)
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

"""Threshold mode, several tensors, fold first: the definition's sample is picked out of the stream; every way out of it."""
import pytest
import torch

import test_gpu_threshold as thr
from paper_2104_01981_b200 import api
from test_gpu_threshold import _built, randn   # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu

# (large enough, and the largest one's sample long enough at small strides, that the plans are taken this way)
SIZES = [300_000, 5, 1_500_001, 0, 4096, 64, 11_000_003, 4097, 65_537]


@pytest.fixture
def options(request, monkeypatch):
    class WithOptions(api.Plan):
        def __init__(self, *a, **k):
            super().__init__(*a, **k)
            for opt, value in request.param.items():
                self.set_option(opt, value)
    monkeypatch.setattr(thr.api, "Plan", WithOptions)


@pytest.mark.parametrize("options", [{}, {api.GC_OPT_SAMPLE_RANK_PERMILLE: 30}, {api.GC_OPT_CANDIDATE_CAPACITY: 100},
                                     {api.GC_OPT_SAMPLE_RANK_PERMILLE: 700}], ids=["plain", "starved", "overflow", "tight"], indirect=True)
@pytest.mark.parametrize("density", [0.0005, 0.01, 0.06])
@pytest.mark.parametrize("stride,cap_factor", [(0, 0.0), (1, 1.0), (7, 1.5), (1000, 2.0)])
def test_strides_densities_and_redo(options, density, stride, cap_factor):
    n = sum(SIZES)
    thr.check_threshold(SIZES, density, [randn(n, 7 * stride + s) for s in range(2)], stride=stride, cap_factor=cap_factor)


@pytest.mark.parametrize("what", ["blind", "biased", "grid", "constant", "zeros", "nonfinite", "sorted"])
def test_samples_that_mislead(what):
    """The definition's sample and the one that sets the bracket see different tensors, or equal keys by the thousand."""
    g = randn(sum(SIZES), 8)
    off = 0
    for n in SIZES:
        v, grp = g[off:off + n], torch.arange(n) // 4
        if what == "blind":
            v[(grp % 64) == 0] *= 1e-3
        elif what == "biased":
            v[(grp % 64) == 0] *= 1e3
        elif what == "grid":
            v.copy_((v * 8).round() / 8)
        elif what == "constant":
            v.fill_(0.25)
        elif what == "zeros":
            v[: n - n // 200] = 0.0
        elif what == "nonfinite" and n > 100:
            v[::97] = float("inf")
            v[1::1009] = float("nan")
        elif what == "sorted":
            v.copy_(v[v.abs().argsort()])
        off += n
    thr.check_threshold(SIZES, 0.01, [g, g], cap_factor=3.0)


def test_tensors_with_long_samples():
    """Samples of more than 128 sample tiles: such plans took the staged route before."""
    sizes = [20_000_003, 70_000, 9_000_000]
    assert api.Plan(sizes, 0.01, mode=api.GC_THRESHOLD, device=0).query(api.GC_Q_COMPRESS_ROUTE) == api.GC_ROUTE_THRESHOLD_MANY
    thr.check_threshold(sizes, 0.01, [randn(sum(sizes), s) for s in range(2)])


@pytest.mark.parametrize("W,density", [(2, 0.01), (8, 0.001), (3, 0.05)])
def test_workers(W, density):
    sizes = [9_300_000, 3, 70_001, 4097, 3_400_000, 513]
    thr.check_threshold_workers(sizes, density, W, lambda w, s: randn(sum(sizes), 100 * s + w))


@pytest.mark.parametrize("cap_factor", [8.0, 1.0], ids=["all", "truncated"])
@pytest.mark.parametrize("bad", [0, 2, 6])
@pytest.mark.parametrize("what", ["ties", "blind"])
def test_one_tensor_fails_and_the_others_do_not(what, bad, cap_factor):
    """A tensor whose short list is too long, or that leaves no room in a region of the candidate list, is redone by itself,
    in front of, between or behind others that are not."""
    g = randn(sum(SIZES), 9)
    t = g[sum(SIZES[:bad]):sum(SIZES[:bad + 1])]
    if what == "ties":
        t[t.abs() > 2.0] = 2.0                         # equal keys from above the threshold to below it
    else:
        t[(torch.arange(t.numel()) // 4) % 64 == 0] *= 1e-3      # the sample meets small ones only: nearly every element is a hit
    plan, w = thr.check_threshold(SIZES, 0.01, [g], cap_factor=cap_factor)
    # (what such a tensor lists in a region that it shares may leave no room for the head of the next one)
    assert plan.last_counters(w.ws)[1:] in ([(0, 1)] if what == "ties" else [(0, 1), (0, 2)])


def test_workers_that_fail_in_one_tensor():
    """The same in a launch that several workers share, another tensor for each of them; calls of their own give the same."""
    plan = api.Plan(SIZES, 0.002, mode=api.GC_THRESHOLD, device=0)
    a, b = ([thr.GpuWorker(plan) for _ in range(4)] for _ in range(2))
    gs = [randn(sum(SIZES), 70 + w).cuda() for w in range(4)]
    for w, bad in enumerate((0, 2, 6)):
        t = gs[w][sum(SIZES[:bad]):sum(SIZES[:bad + 1])]
        t[(torch.arange(t.numel(), device="cuda") // 4) % 64 == 0] *= 1e-3
    plan.compress_workers(gs, [w.residual for w in a], [w.idx for w in a], [w.val for w in a], [w.count for w in a], [w.ws for w in a])
    seen = [plan.last_counters(w.ws)[1:] for w in a]
    assert all(c in ((0, 1), (0, 2)) for c in seen[:3]) and seen[3] == (0, 0)
    for w in range(4):
        b[w].step(gs[w])
        assert torch.equal(a[w].count, b[w].count) and torch.equal(a[w].residual, b[w].residual)
        for o, c in zip(plan.tensor_out_offset(), b[w].count.tolist()):
            assert torch.equal(a[w].idx[o:o + c], b[w].idx[o:o + c]) and torch.equal(a[w].val[o:o + c], b[w].val[o:o + c])


def test_more_tensors_than_the_tables_in_shared_memory_hold():
    """Above 1024 tensors the owners of tiles and sample tiles are searched in the device tables."""
    sizes = [9000] * 550 + [9_000_003] + [9001] * 550            # (the long sample: no other fused kernel takes the plan)
    assert api.Plan(sizes, 0.002, mode=api.GC_THRESHOLD, device=0).query(api.GC_Q_COMPRESS_ROUTE) == api.GC_ROUTE_THRESHOLD_MANY
    plan, w = thr.check_threshold(sizes, 0.002, [randn(sum(sizes), s) for s in range(2)])
    assert plan.last_counters(w.ws)[1:] == (0, 0)

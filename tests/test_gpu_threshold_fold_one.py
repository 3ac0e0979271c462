"""Threshold mode, one tensor, fold first: sizes on both sides of its line, strides, redo, samples that mislead."""
import pytest
import torch

import test_gpu_threshold as thr
from paper_2104_01981_b200 import api
from test_gpu_threshold import _built, randn   # noqa: F401  (the module's build fixture)
from test_gpu_threshold_fold import options    # noqa: F401

pytestmark = pytest.mark.gpu

N = 13_000_003                                     # (12M elements and 2 % are the line)


@pytest.mark.parametrize("options", [{}, {api.GC_OPT_SAMPLE_RANK_PERMILLE: 30}, {api.GC_OPT_CANDIDATE_CAPACITY: 100}],
                         ids=["plain", "starved", "overflow"], indirect=True)
@pytest.mark.parametrize("density,stride,cap_factor", [(0.0003, 0, 0.0), (0.001, 7, 1.0), (0.01, 0, 1.0), (0.01, 1, 1.5), (0.02, 1000, 4.0)])
def test_strides_densities_and_redo(options, density, stride, cap_factor):
    thr.check_threshold([N], density, [randn(N, 7 * stride + s) for s in range(2)], stride=stride, cap_factor=cap_factor)


@pytest.mark.parametrize("n", [(12 << 20) - 1, 12 << 20, (12 << 20) + 1, 40_000_001])
def test_sizes_around_the_line(n):
    thr.check_threshold([n], 0.005, [randn(n, s) for s in range(2)])


@pytest.mark.parametrize("what", ["blind", "biased", "grid", "constant", "zeros", "nonfinite", "sorted"])
def test_samples_that_mislead(what):
    g, grp = randn(N, 8), torch.arange(N) // 4
    if what == "blind":
        g[(grp % 64) == 0] *= 1e-3
    elif what == "biased":
        g[(grp % 64) == 0] *= 1e3
    elif what == "grid":
        g = (g * 8).round() / 8
    elif what == "constant":
        g.fill_(0.25)
    elif what == "zeros":
        g[: N - N // 200] = 0.0
    elif what == "nonfinite":
        g[::97] = float("inf")
        g[1::1009] = float("nan")
    elif what == "sorted":
        g = g[g.abs().argsort()].contiguous()
    thr.check_threshold([N], 0.01, [g, g], cap_factor=3.0)


@pytest.mark.parametrize("what,n,density", [("bfloat16", N, 0.01), ("bfloat16", N, 0.02), ("grid", 40_000_001, 0.01), ("grid", 40_000_001, 0.003)])
@pytest.mark.parametrize("cap_factor", [8.0, 1.0], ids=["all", "truncated"])
def test_ties_by_the_thousand_are_counted(what, n, density, cap_factor):
    """More equal keys at the threshold than a short list is worth, or than it holds: no redo."""
    g = randn(n, 5)
    g = g.to(torch.bfloat16).float() if what == "bfloat16" else (g * 8).round() / 8
    plan, w = thr.check_threshold([n], density, [g], cap_factor=cap_factor)
    assert plan.last_counters(w.ws)[1:] == (0, 0)


@pytest.mark.parametrize("density", [0.001, 0.03])
def test_samples_beyond_the_rounds_of_the_other_kernel(density):
    """A definition that samples everything: more than 64 groups per thread, formerly four launches, now fold first at any density."""
    n = 31_000_001
    assert api.Plan([n], density, mode=api.GC_THRESHOLD, device=0, sample_stride=1).query(api.GC_Q_COMPRESS_ROUTE) == api.GC_ROUTE_THRESHOLD_ONE
    plan, w = thr.check_threshold([n], density, [randn(n, s) for s in range(2)], stride=1)
    assert plan.last_counters(w.ws)[1:] == (0, 0)

"""Threshold mode on gradients whose scale varies along rows: the definition's sample then sees a few columns over and over,
and the bracket of the fold-first kernels has to come from the same places.  No redo, and the oracle's result."""
import numpy as np
import pytest
import torch

import test_gpu_threshold as thr
from paper_2104_01981_b200 import api
from test_gpu_threshold import _built   # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


def columns(rows, cols, repeat, spread, gen):
    """rows x (cols x repeat) normal entries times a log-normal scale per column (a channel's `repeat` entries share it)."""
    scale = torch.exp(torch.randn(cols, generator=gen) * spread).repeat_interleave(repeat)
    return (torch.randn(rows, cols * repeat, generator=gen) * scale).flatten()


def check_without_redo(sizes, density, g, stride=0):
    plan, w = thr.check_threshold(sizes, density, [g], stride=stride, cap_factor=4.0)
    assert plan.last_counters(w.ws)[1:] == (0, 0)


@pytest.mark.parametrize("cols", [768, 1024, 4608])
@pytest.mark.parametrize("spread,density,stride", [(0.1, 0.01, 0), (0.4, 0.01, 0), (0.4, 0.001, 0), (0.2, 0.02, 16), (0.4, 0.01, 1)])
def test_one_tensor(cols, spread, density, stride):
    gen = torch.Generator().manual_seed(cols + int(100 * spread))
    for _ in range(2):
        g = columns(13_000_003 // cols + 1, cols, 1, spread, gen)[:13_000_003].contiguous()
        check_without_redo([13_000_003], density, g, stride)


# layers of a convolutional network, 1 x 1 and 3 x 3, and a dense one that takes the plan over 12M elements
LAYERS = [(64, 64, 1), (64, 64, 9), (256, 64, 1), (128, 128, 9), (512, 128, 1), (3, 1, 1), (256, 256, 9), (1024, 256, 1), (512, 512, 9),
          (2048, 512, 1), (2048, 3072, 1), (1000, 2048, 1)]


def layers(spread, gen):
    return torch.cat([columns(o, i, k, spread, gen) for o, i, k in LAYERS])


@pytest.mark.parametrize("spread", [0.1, 0.2, 0.4])
@pytest.mark.parametrize("density,stride", [(0.001, 0), (0.005, 0), (0.001, 8)])
def test_layers(spread, density, stride):
    sizes, gen = [o * i * k for o, i, k in LAYERS], torch.Generator().manual_seed(int(100 * spread))
    for _ in range(2):
        check_without_redo(sizes, density, layers(spread, gen), stride)


def test_workers():
    sizes, gen = [o * i * k for o, i, k in LAYERS], torch.Generator().manual_seed(3)
    plan = api.Plan(sizes, 0.001, mode=api.GC_THRESHOLD, device=0, cap_factor=4.0)
    ws = [thr.GpuWorker(plan) for _ in range(4)]
    plan.compress_workers([layers(0.4, gen).cuda() for _ in ws], [w.residual for w in ws], [w.idx for w in ws], [w.val for w in ws],
                          [w.count for w in ws], [w.ws for w in ws])
    assert [plan.last_counters(w.ws)[1:] for w in ws] == [(0, 0)] * 4
    assert all(np.all(w.count.cpu().numpy()[:len(sizes)] > 0) for w in ws)

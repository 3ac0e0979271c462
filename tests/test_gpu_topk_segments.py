"""Many-tensor plans at the lines between their forms: lengths of the short list, unequal shares of several workers."""
import pytest
import torch

from paper_2104_01981_b200 import api
from helpers import GpuWorker, check_topk_against_oracle
from test_gpu_topk_dense import _built   # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c", [1, 31, 32, 33, 64, 128, 255, 256, 257, 511, 512, 513, 1025])
@pytest.mark.parametrize("equal", [0, 1, 3], ids=["distinct", "equal", "threes"])
def test_short_lists_of_given_length(c, equal):
    """Two tensors whose threshold lies in the middle of `c` magnitudes within 1e-4 of each other, with nothing else
    near: the band bin holds these.  Distinct, all equal, or three of a kind (the lowest indices win)."""
    density, sizes = 0.01, [400_000, 1_000_003]
    parts = []
    for t, n in enumerate(sizes):
        gen = torch.Generator().manual_seed(100 * c + t)
        k = -(-n // 100)
        v = torch.rand(n, generator=gen) * 0.5                       # the rest
        top = k - (c + 1) // 2
        v[:top] = 4.0 + torch.rand(top, generator=gen) * 8.0         # sent for sure
        step = torch.arange(c, dtype=torch.float32) // max(equal, 1) if equal != 1 else torch.zeros(c)
        v[top:top + c] = 1.0 + step * (1e-4 / max(c, 1))
        v *= torch.where(torch.rand(n, generator=gen) < 0.5, -1.0, 1.0)
        parts.append(v[torch.randperm(n, generator=gen)])
    check_topk_against_oracle(sizes, density, [torch.cat(parts)])


@pytest.mark.parametrize("W", [2, 3, 5, 8, 12])
def test_unequal_shares_of_several_workers(W):
    """Workers whose CTAs have some sixty tiles: one launch gives what calls of their own give."""
    n = 444 * 4096 * 62 // W
    sizes = [n // 2 + 3, 1000, n // 3, 5, n - n // 2 - n // 3]
    plan = api.Plan(sizes, 0.01, device=0)
    gen = torch.Generator(device="cuda").manual_seed(W)
    a, b = ([GpuWorker(plan) for _ in range(W)] for _ in range(2))
    gs = [torch.randn(plan.total_n, device="cuda", generator=gen) for _ in range(W)]
    for _ in range(2):
        plan.compress_workers(gs, [w.residual for w in a], [w.idx for w in a], [w.val for w in a], [w.count for w in a], [w.ws for w in a])
        for w in range(W):
            plan.compress(gs[w], b[w].residual, b[w].idx, b[w].val, b[w].count, b[w].ws)
            a[w].check_status()
            assert torch.equal(a[w].idx, b[w].idx) and torch.equal(a[w].val, b[w].val) and torch.equal(a[w].count, b[w].count)
            assert torch.equal(a[w].residual, b[w].residual)

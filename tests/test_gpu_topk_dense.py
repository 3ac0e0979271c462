"""GPU parity of the fused top-k kernels where lists get long -- densities of several per cent, thousands of
ties at the threshold -- against the CPU oracle (bit for bit)."""
import pytest
import torch

from paper_2104_01981_b200 import api, build
from helpers import check_topk_against_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    api.lib()


@pytest.mark.parametrize("sizes,density,route", [
    ([30_000_001], 0.05, api.GC_ROUTE_TOPK_ONE),
    ([7_000_003], 0.1, api.GC_ROUTE_TOPK_ONE),
    ([9_000_000, 4097, 3_000_001, 130_000, 17], 0.05, api.GC_ROUTE_TOPK_MANY),
    ([5_000_000, 5_000_001], 0.0099, api.GC_ROUTE_TOPK_MANY),      # sample read once: tau is a bin edge
    ([5_000_000, 5_000_001], 0.0101, api.GC_ROUTE_TOPK_MANY),      # sample ranked twice
    ([60_000_000, 1000], 0.04, api.GC_ROUTE_TOPK_MANY),
])
@pytest.mark.parametrize("kind", ["normal", "ties"])
def test_dense_plans_match_the_oracle(sizes, density, route, kind):
    """Two error-feedback steps; `ties`: magnitudes on a grid, so that the short list of the threshold
    holds thousands of equal keys (and may send the tensor to the exact redo)."""
    assert api.Plan(sizes, density, device=0).query(api.GC_Q_COMPRESS_ROUTE) == route
    gen = torch.Generator(device="cuda").manual_seed(7)
    grads = []
    for _ in range(2):
        g = torch.randn(sum(sizes), device="cuda", generator=gen)
        grads.append((torch.round(g * 4096.0) / 4096.0 if kind == "ties" else g).cpu())
    check_topk_against_oracle(sizes, density, grads)


@pytest.mark.parametrize("n,density,step", [(12_000_003, 0.01, 1 / 64), (12_000_003, 0.01, 1 / 4), (9_000_000, 0.002, 1 / 16),
                                            (20_000_001, 0.05, 1 / 32), (2_000_000, 0.01, 1.0), (6_000_000, 0.3, 1 / 8)])
def test_thousands_of_ties_at_the_threshold(n, density, step):
    """Magnitudes on a coarse grid: the band bin of the threshold holds 4,000 to a million candidates with one
    or a few keys, and the lowest indices among the equal ones win."""
    gen = torch.Generator(device="cuda").manual_seed(n)
    grads = [(torch.round(torch.randn(n, device="cuda", generator=gen) / step) * step).cpu() for _ in range(2)]
    check_topk_against_oracle([n], density, grads)


def test_ties_in_one_region_only():
    """All candidates at the threshold key lie in one stretch of the tensor: the cut falls inside a chunk of it."""
    n = 8_000_001
    for lo, hi, density in ((0, 30_000, 0.002), (n - 30_000, n, 0.002), (4_000_000, 4_100_000, 0.01)):
        g = torch.randn(n, generator=torch.Generator().manual_seed(hi)) * 0.01
        g[lo:hi] = 3.0
        g[lo + 5:hi:7] = -3.0
        check_topk_against_oracle([n], density, [g])

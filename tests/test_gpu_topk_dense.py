"""GPU parity of the fused top-k kernels at densities of several per cent, where a CTA's candidate region
holds tens of thousands of entries, against the CPU oracle (bit for bit)."""
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

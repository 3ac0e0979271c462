"""One-tensor top-k on both sides of the lines between its two ways to rank a chunk's candidates."""
import pytest
import torch

from helpers import check_topk_against_oracle
from test_gpu_topk_dense import _built   # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu

TILES = 16_000 * 4096


@pytest.mark.parametrize("n,density", [(TILES - 4096, 0.005), (TILES - 4095, 0.005), (70_000_001, 0.0021), (70_000_001, 0.0089),
                                       (70_000_001, 0.0091), (70_000_001, 0.0124), (70_000_001, 0.0126), (70_000_001, 0.021), (20_000_001, 0.021), (5_000_001, 0.003)])
def test_both_ways_match_the_oracle(n, density):
    gen = torch.Generator(device="cuda").manual_seed(n % 1000 + int(density * 1e5))
    check_topk_against_oracle([n], density, [torch.randn(n, device="cuda", generator=gen).cpu() for _ in range(2)])

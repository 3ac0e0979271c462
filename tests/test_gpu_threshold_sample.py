"""The one-tensor threshold's sample: a block counts its keys above a floor of its own, and below it on demand."""
import pytest
import torch

from test_gpu_threshold import _built, check_threshold, randn   # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [70_001, 3_000_001])
@pytest.mark.parametrize("stride", [1, 7, 64])
@pytest.mark.parametrize("layout", ["sorted", "one_block_large", "one_block_huge", "constant"])
def test_sample_floor(n, stride, layout):
    # magnitudes gathered in one place: the floors of the blocks that sample it lie above the wanted rank's bin,
    # and the keys of that bin that they left out are counted afterwards
    grads = []
    for s in range(2):
        g = randn(n, 11 * n + stride + s)
        if layout == "sorted":
            g = g[g.abs().argsort()]
        elif layout == "one_block_large":
            g[n // 2:n // 2 + n // 8] *= 3.0
        elif layout == "one_block_huge":
            g[:n // 300] *= 1e4
        else:
            g = torch.full((n,), 0.25)
        grads.append(g.contiguous())
    check_threshold([n], 0.01, grads, stride=stride, cap_factor=4.0)

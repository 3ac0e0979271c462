"""Decode kernels are launched while the kernel in front of them ends: what that kernel wrote last is what they read."""
import pytest
import torch

from paper_2104_01981_b200 import api
from test_gpu_topk_dense import _built   # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,W,density", [(4097, 1, 0.05), (300_001, 1, 0.01), (300_001, 5, 0.01), (2_000_003, 8, 0.02), (14_000_000, 2, 0.01)])
@pytest.mark.parametrize("apply", ["dense", "add", "momentum"])
@pytest.mark.parametrize("captured", [False, True])
def test_lists_written_by_the_kernel_in_front(n, W, density, apply, captured):
    """Rounds without a wait: lists, buffers and parameters are overwritten by copies, the decode follows at once."""
    plan = api.Plan([n], density, device=0)
    k, rounds = plan.total_cap, 12
    gen = torch.Generator(device="cuda").manual_seed(n + W)
    src_i = [[torch.randperm(n, device="cuda", generator=gen)[:k].sort().values.to(torch.int32) for _ in range(W)] for _ in range(rounds)]
    src_v = [[torch.randint(-8, 9, (k,), device="cuda", generator=gen).float() for _ in range(W)] for _ in range(rounds)]      # (sums are exact)
    start = torch.randint(-8, 9, (n,), device="cuda", generator=gen).float()
    idx = [torch.zeros(k, dtype=torch.int32, device="cuda") for _ in range(W)]
    val = [torch.zeros(k, device="cuda") for _ in range(W)]
    buf, vel, ws, got = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda"), plan.alloc_workspace(), []
    side = torch.cuda.Stream()

    def round_(r, stream):
        buf.copy_(start)
        if apply == "momentum":
            vel.copy_(start)
        for w in range(W):
            idx[w].copy_(src_i[r][w])
            val[w].copy_(src_v[r][w])
        if apply == "momentum":
            plan.decompress_apply_momentum(idx, val, None, buf, vel, 0.5, 0.5, 1.0, ws, stream)
        else:
            plan.decompress_accumulate(idx, val, None, buf, apply == "dense", ws, stream)

    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        round_(0, side)
        graphs = []
        if captured:
            side.synchronize()
            for r in range(rounds):
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=side):
                    round_(r, side)
                graphs.append(g)
        for r in range(rounds):
            graphs[r].replay() if captured else round_(r, side)
            got.append((buf.clone(), vel.clone()))
    side.synchronize()
    for r in range(rounds):
        total = torch.zeros(n, device="cuda")
        for w in range(W):
            total.index_add_(0, src_i[r][w].long(), src_v[r][w])
        if apply == "momentum":
            v = 0.5 * start + total
            assert torch.equal(got[r][1], v) and torch.equal(got[r][0], start - 0.5 * v), r
        else:
            assert torch.equal(got[r][0], total if apply == "dense" else start + total), r
    assert plan.last_status(ws)[0] == api.GC_OK

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


@pytest.mark.parametrize("sizes,W,mode", [([70_001, 5, 300_000, 0, 64, 4097], 1, api.GC_THRESHOLD), ([70_001, 5, 300_000, 0, 64, 4097], 3, api.GC_THRESHOLD),
                                          ([2_000_003], 1, api.GC_THRESHOLD), ([13_000_003], 1, api.GC_THRESHOLD),
                                          ([300_000, 11_000_003, 1_500_001], 2, api.GC_THRESHOLD), ([1_000_001], 1, api.GC_TOPK)],
                         ids=["several", "several_workers", "one", "one_fold_first", "fold_first_workers", "topk"])
@pytest.mark.parametrize("apply", ["dense", "add", "momentum"])
def test_lists_and_counts_written_by_the_compress_in_front(sizes, W, mode, apply):
    """Steps in a row without a wait, another gradient each: as with a wait behind every call."""
    n, rounds = sum(sizes), 8
    plan = api.Plan(sizes, 0.002 if n > 12_000_000 else 0.01, mode=mode, device=0)
    gen = torch.Generator(device="cuda").manual_seed(n + W)
    # (magnitudes differ from round to round, so the lengths of the lists do)
    grads = [[torch.randn(n, device="cuda", generator=gen) * (1 + r % 3) for _ in range(W)] for r in range(rounds)]

    def steps(wait):
        out = [plan.alloc_outputs() for _ in range(W)]
        idx, val, cnt = ([o[i] for o in out] for i in range(3))
        ws, res = [plan.alloc_workspace() for _ in range(W)], [torch.zeros(n, device="cuda") for _ in range(W)]
        buf, vel, got = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda"), []
        counts = cnt if mode == api.GC_THRESHOLD else None
        torch.cuda.synchronize()
        for r in range(rounds):
            if W == 1:
                plan.compress(grads[r][0], res[0], idx[0], val[0], cnt[0], ws[0])
            else:
                plan.compress_workers(grads[r], res, idx, val, cnt, ws)
            if wait:
                torch.cuda.synchronize()
            if apply == "momentum":
                plan.decompress_apply_momentum(idx, val, counts, buf, vel, 0.5, 0.5, 1.0, ws[0])
            else:
                plan.decompress_accumulate(idx, val, counts, buf, apply == "dense", ws[0])
            if wait:
                torch.cuda.synchronize()
            got.append((buf.clone(), vel.clone()))
        torch.cuda.synchronize()
        return got, res
    (a, ra), (b, rb) = steps(False), steps(True)
    assert all(torch.equal(x, y) for p, q in zip(a, b) for x, y in zip(p, q))
    assert all(torch.equal(x, y) for x, y in zip(ra, rb)) and float(a[-1][0].abs().max()) > 0.0

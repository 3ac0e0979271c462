"""GPU parity of the fused top-k kernels where lists get long -- densities of several per cent, thousands of
ties at the threshold -- against the CPU oracle (bit for bit)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2104_01981_b200 import api, build
from helpers import bits, check_topk_against_oracle, to_np_u32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    api.lib()


@pytest.mark.parametrize("sizes,density,route", [
    ([30_000_001], 0.05, api.GC_ROUTE_TOPK_ONE),
    ([7_000_003], 0.1, api.GC_ROUTE_TOPK_ONE),
    ([9_000_000, 4097, 3_000_001, 130_000, 17], 0.05, api.GC_ROUTE_TOPK_MANY),
    ([5_000_000, 5_000_001], 0.00049, api.GC_ROUTE_TOPK_MANY),     # sample read once: tau is a bin edge
    ([5_000_000, 5_000_001], 0.00051, api.GC_ROUTE_TOPK_MANY),     # sample ranked twice
    ([5_000_000, 5_000_001], 0.0199, api.GC_ROUTE_TOPK_MANY),      # below and above the forms for dense plans
    ([5_000_000, 5_000_001], 0.0201, api.GC_ROUTE_TOPK_MANY),
    ([9_000_001], 0.0199, api.GC_ROUTE_TOPK_ONE),
    ([9_000_001], 0.0201, api.GC_ROUTE_TOPK_ONE),
    ([60_000_000, 1000], 0.04, api.GC_ROUTE_TOPK_MANY),
])
@pytest.mark.parametrize("kind", ["normal", "ties", "repeated"])
def test_dense_plans_match_the_oracle(sizes, density, route, kind):
    """Two error-feedback steps; `ties`: magnitudes on a grid, so that the short list of the threshold
    holds thousands of equal keys (and may send the tensor to the exact redo); `repeated`: five steps with one
    gradient, whose unsent entries pile up below the threshold."""
    assert api.Plan(sizes, density, device=0).query(api.GC_Q_COMPRESS_ROUTE) == route
    gen = torch.Generator(device="cuda").manual_seed(7)
    grads = []
    for _ in range(2 if kind != "repeated" else 1):
        g = torch.randn(sum(sizes), device="cuda", generator=gen)
        grads.append((torch.round(g * 4096.0) / 4096.0 if kind == "ties" else g).cpu())
    check_topk_against_oracle(sizes, density, grads if kind != "repeated" else grads * 5)


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


STAMPS = 16                                              # word of the workspace header: phases of the last launch + 1


def check_bf16(n, density, grads, r0, redo=False):
    """compress_bf16 on one plan, step after step, against the oracle on the widened values.  Returns the phases of
    each step: a counted band has one more than a listed one."""
    plan = api.Plan([n], density, device=0)
    assert plan.query(api.GC_Q_COMPRESS_ROUTE) == api.GC_ROUTE_TOPK_ONE and n > 1 << 22
    k, ws = plan.total_cap, plan.alloc_workspace()
    idx, val, cnt = plan.alloc_outputs()
    r, r_cpu, phases = r0.cuda(), r0.numpy().copy(), []
    for g in grads:
        idx.fill_(-1)
        plan.compress_bf16(g.cuda(), r, idx, val, cnt, ws)
        oi, ov = oracle.topk_compress_tensors([n], [k], g.float().numpy(), r_cpu)
        assert plan.last_status(ws)[0] == api.GC_OK and (redo or plan.last_counters(ws)[1:] == (0, 0))
        assert np.array_equal(to_np_u32(idx), oi) and np.array_equal(to_np_u32(val), bits(ov))
        assert np.array_equal(to_np_u32(r), bits(r_cpu)) and cnt.tolist() == [k, k]
        phases.append(ws.view(torch.int32)[STAMPS].item())
    return phases


# (n x step x twice the normal density at the threshold, over sqrt(2) with the second residual, entries share the
# threshold's magnitude: at least 5,000 here, counting begins at 4,097)
@pytest.mark.parametrize("n,density,step", [(12_000_003, 0.01, 1 / 32), (4_194_305, 0.01, 1 / 16), (9_000_000, 0.002, 1 / 4),
                                            (20_000_001, 0.05, 1 / 32), (12_000_003, 0.02, 1 / 64)])
@pytest.mark.parametrize("residual", ["zero", "grid"])
def test_thousands_of_bfloat16_ties_are_counted(n, density, step, residual):
    """bfloat16 gradients on a residual of zero, or on one of few distinct values: the band bin of the threshold
    holds more candidates than are listed, so they are counted and cut by tile.  The next step, on a residual with
    few ties, lists them."""
    gen = torch.Generator(device="cuda").manual_seed(n % 1000)
    grads = [(torch.round(torch.randn(n, device="cuda", generator=gen) / step) * step).to(torch.bfloat16).cpu() for _ in range(2)]
    r0 = torch.zeros(n) if residual == "zero" else torch.round(torch.randn(n, generator=torch.Generator().manual_seed(1)) * 4) / 4
    counted = check_bf16(n, density, grads, r0)
    listed = check_bf16(n, density, [torch.randn(n, device="cuda", generator=gen).to(torch.bfloat16).cpu()],
                        torch.randn(n, generator=torch.Generator().manual_seed(2)))
    assert counted[0] == listed[0] + 1, (counted, listed)


@pytest.mark.parametrize("lo,hi,density,redo", [(0, 30_000, 0.002, True), (8_000_001 - 30_000, 8_000_001, 0.002, True),
                                                (4_000_000, 4_100_000, 0.01, True), (1_000_123, 1_400_124, 0.03, False),
                                                (0, 400_000, 0.04, False), (8_000_001 - 600_000, 8_000_001, 0.05, False)])
def test_bfloat16_ties_in_one_region_only(lo, hi, density, redo):
    """All candidates at the threshold key lie in one stretch of the tensor: the cut falls inside a chunk of it.  (The
    tiles of a short stretch lie with few CTAs, whose regions they may overflow: then the exact redo settles it.)"""
    n = 8_000_001
    g = torch.randn(n, generator=torch.Generator().manual_seed(hi)) * 0.01
    g[lo:hi] = 3.0
    g[lo + 5:hi:7] = -3.0
    check_bf16(n, density, [g.to(torch.bfloat16)], torch.zeros(n), redo)

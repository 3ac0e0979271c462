"""GPU parity of the direct (radix-select) top-k kernel -- small one-tensor plans and the call without a
plan -- at the edges of its geometry, against the CPU oracle (bit for bit)."""
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


# one CTA, one more element than it takes, a ragged last vector, the largest plan of the kernel and the
# first that is not
@pytest.mark.parametrize("n", [4098, 8192, 8193, 606_207, 606_209, 1_212_419, (1 << 22) - 1, 1 << 22, (1 << 22) + 1])
@pytest.mark.parametrize("density,step", [(0.01, 0.0), (0.0005, 0.0), (0.2, 0.0), (0.01, 1 / 8), (0.01, 4.0)])
def test_plans_match_the_oracle(n, density, step):
    """Three error-feedback steps; step > 0 puts the values on a grid, so that from a handful to all of the
    entries around the threshold share their key."""
    gen = torch.Generator(device="cuda").manual_seed(n)
    grads = []
    for _ in range(3 if n < 2_000_000 else 2):
        g = torch.randn(n, device="cuda", generator=gen)
        grads.append((torch.round(g / step) * step if step else g).cpu())
    check_topk_against_oracle([n], density, grads)


@pytest.mark.parametrize("n,k", [(1, 1), (3, 2), (2049, 1), (2049, 2049), (7_274_000, 72_740), (7_290_001, 3), (9_000_003, 900_000)])
@pytest.mark.parametrize("ties", [False, True])
def test_call_without_a_plan_matches_the_oracle(n, k, ties):
    """Shares in shared memory and, beyond 7.2M elements, read back from L2."""
    gen = torch.Generator(device="cuda").manual_seed(n + k)
    status = torch.full((1,), 77, dtype=torch.int32, device="cuda")
    r = torch.randn(n + 4, device="cuda", generator=gen)[:n]
    r_cpu = r.cpu().numpy().copy()
    for _ in range(2):
        g = torch.randn(n + 4, device="cuda", generator=gen)[:n]
        if ties:
            g, r = torch.round(g * 4) / 4, torch.round(r * 4) / 4
            r_cpu = r.cpu().numpy().copy()
        idx = torch.full((k,), -1, dtype=torch.int32, device="cuda")
        val = torch.full((k,), float("nan"), device="cuda")
        oi, ov = oracle.topk_compress_tensors([n], [k], g.cpu().numpy(), r_cpu)
        assert api.compress_noalloc(g, r, n, k, idx, val, status) == api.GC_OK
        torch.cuda.synchronize()
        assert status.item() == api.GC_OK
        assert np.array_equal(to_np_u32(idx), oi) and np.array_equal(to_np_u32(val), bits(ov))
        assert np.array_equal(to_np_u32(r), bits(r_cpu))


def test_bfloat16_and_a_private_workspace():
    n = 500_003
    plan = api.Plan([n], 0.01, device=0)
    plan.set_option(api.GC_OPT_WORKSPACE_PRIVATE, 1)
    ws = plan.alloc_workspace()
    idx, val, cnt = plan.alloc_outputs()
    r, r_cpu = torch.zeros(n, device="cuda"), np.zeros(n, np.float32)
    before = plan.launches()
    for step in range(4):
        g = torch.randn(n, generator=torch.Generator().manual_seed(step)).to(torch.bfloat16)
        plan.compress_bf16(g.cuda(), r, idx, val, cnt, ws)
        oi, ov = oracle.topk_compress_tensors([n], plan.tensor_k(), g.to(torch.float32).numpy(), r_cpu)
        assert np.array_equal(to_np_u32(idx), oi) and np.array_equal(to_np_u32(val), bits(ov))
        assert np.array_equal(to_np_u32(r), bits(r_cpu))
    assert plan.launches() - before == 5                  # one clearing launch, then one launch per call
    assert plan.last_status(ws) == (api.GC_OK, 0)


# word ranges of the scratch behind its header: the three histograms, the length of the list
@pytest.mark.parametrize("words,value", [((64, 64 + 2048), 40), ((64 + 2047, 64 + 2048), 1), ((64, 65), 1 << 20),
                                         ((2112, 2112 + 1024), 500), ((4160, 4161), 40), ((4160, 4161), 1 << 30)])
def test_scratch_that_others_wrote_to_is_reported_and_writes_stay_in_bounds(words, value):
    """A private workspace in which somebody raised counts and left the header's mark alone: the call ends with
    GC_E_INVALID, nothing is written behind the k entries, and after the status has been read the next call is
    exact again."""
    n, k, slack = 1_000_003, 10_001, 4096
    plan = api.Plan([n], 0.01, device=0)
    plan.set_option(api.GC_OPT_WORKSPACE_PRIVATE, 1)
    assert plan.total_cap == k
    ws = plan.alloc_workspace()
    idx = torch.full((k + slack,), -7, dtype=torch.int32, device="cuda")
    val = torch.full((k + slack,), -7.0, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(value & 0xFFFF)
    r = torch.zeros(n, device="cuda")
    for step in range(3):
        g = torch.randn(n, device="cuda", generator=gen)
        if step == 1:
            ws.view(torch.int32)[words[0]:words[1]] += value
        r_cpu = r.cpu().numpy().copy()
        plan.compress(g, r, idx, val, None, ws)
        assert plan.last_status(ws)[0] == (api.GC_E_INVALID if step == 1 else api.GC_OK)
        assert bool((idx[k:] == -7).all()) and bool((val[k:] == -7.0).all())
        if step != 1:
            oi, ov = oracle.topk_compress_tensors([n], [k], g.cpu().numpy(), r_cpu)
            assert np.array_equal(to_np_u32(idx[:k]), oi) and np.array_equal(to_np_u32(val[:k]), bits(ov))
            assert np.array_equal(to_np_u32(r), bits(r_cpu))

"""Rows of every length class -- 8, 16 or 32 lanes a row, full and ragged -- against the oracle, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import ecrm_oracle as eo
from paper_2104_01981_b200 import ecrm, synth
from test_gpu_ecrm import _built, same   # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [4, 28, 32, 36, 64, 68, 128, 132, 260])
@pytest.mark.parametrize("m", [1, 5, 37, 20_003])
@pytest.mark.parametrize("optimizer,lr,hyper", [(ecrm.ECRM_ADAGRAD, 0.05, 1e-8), (ecrm.ECRM_MOMENTUM, 0.01, 0.9)])
def test_rows_of_any_length(dim, m, optimizer, lr, hyper):
    n = 2 * m + 3
    k = 6
    shards = synth.ecrm_tables(n, dim, k, seed=dim + m)
    parity = eo.encode([s.numpy() for s in shards])
    rows, g = synth.ecrm_batch(n, m, dim, seed=dim * m)
    rows_np = rows.numpy().view(np.uint32)
    prow = torch.from_numpy(np.random.default_rng(m).permutation(n)[:m].astype(np.uint32).view(np.int32))
    prow_np = prow.numpy().view(np.uint32)
    bad = torch.zeros(1, dtype=torch.int32, device="cuda")

    # reads of a lost shard's rows, every surviving shard with rows of its own or all with the parity's
    for srow in (None, [prow.roll(s) for s in range(k - 1)]):
        out = torch.full((m, dim), float("nan"), device="cuda")
        ecrm.degraded_read(prow.cuda(), None if srow is None else [s.cuda() for s in srow],
                           [s.cuda() for s in shards[1:]], torch.from_numpy(parity).cuda(), out, bad)
        want = parity[prow_np].copy()
        for s in range(1, k):
            at = prow_np if srow is None else srow[s - 1].numpy().view(np.uint32)
            want = (want - shards[s].numpy()[at]).astype(np.float32)
        assert same(out, want)

    # optimizer step with differences, parity update; then both in one pass on copies: the same bits
    state, p_state = torch.rand(n, dim), torch.rand(n, dim)
    first = [t.cuda() for t in (shards[0], state, torch.from_numpy(parity), p_state)]
    fused = [t.clone() for t in first]
    h = [t.cpu().numpy().copy() for t in first]
    rows_bad = rows.clone()
    if m > 1:
        rows_bad[m // 2] = n                                # out of range: skipped and counted
    keep = np.arange(m) != (m // 2 if m > 1 else -1)
    de, ds = torch.zeros(m, dim, device="cuda"), torch.zeros(m, dim, device="cuda")
    ecrm.rows_step(optimizer, rows_bad.cuda(), g.cuda(), first[0], first[1], lr, hyper, de, ds, bad)
    wde, wds = eo.rows_step(optimizer, rows_np[keep], g.numpy()[keep], h[0], h[1], lr, hyper)
    assert same(de[torch.from_numpy(keep).cuda()], wde) and same(ds[torch.from_numpy(keep).cuda()], wds)
    ecrm.parity_add(prow.cuda(), de, ds, first[2], first[3], bad)
    eo.parity_add(prow_np[keep], wde, wds, h[2], h[3])
    ecrm.rows_step_parity(optimizer, rows_bad.cuda(), prow.cuda(), g.cuda(), *fused, lr, hyper, bad)
    for a, b, c in zip(first, fused, h):
        assert same(a, c) and same(b, c)
    assert bad.item() == (2 if m > 1 else 0)

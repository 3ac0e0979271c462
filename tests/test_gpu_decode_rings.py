"""GPU parity of the ring decode kernel at the edges of its geometry, against the CPU oracle (bit for bit)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2104_01981_b200 import api, build, synth
from helpers import bits, to_np_u32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    api.lib()


# n around one and several groups of eight sub-tiles (sub-tiles are multiples of 128 elements);
# densities from lists that leave most sub-tiles empty to lists whose rings cannot hold a tile's share
@pytest.mark.parametrize("n", [1, 1023, 16384, 16385, 300_001])
@pytest.mark.parametrize("W,density", [(1, 0.2), (2, 0.01), (5, 0.02), (16, 0.05), (32, 0.01), (33, 0.003), (64, 0.4)])
@pytest.mark.parametrize("offset", [0, 1])
def test_ring_decode_matches_the_oracle(n, W, density, offset):
    """Both modes of the plain decode and the momentum step.  `offset` = 1: lists that start 4 bytes
    past a 16-byte boundary; half of the workers share their indices."""
    plan = api.Plan([n], density, device=0)
    plan.set_option(api.GC_OPT_DECODE_ROUTE, api.GC_DECODE_WIDE)
    ws = plan.alloc_workspace()
    k = plan.total_cap
    pairs, d_idx, d_val = [], [], []
    for w in range(W):
        idx, _ = synth.sparse_set([n], [k], 100 + (w // 2 if w < W // 2 else w))
        _, val = synth.sparse_set([n], [k], 900 + w, scale=10.0 ** (w % 5 - 2))
        pairs.append((idx, val))
        for host, out in ((idx.view(np.int32), d_idx), (val, d_val)):
            buf = torch.zeros(k + 8, dtype=torch.from_numpy(host).dtype, device="cuda")
            buf[offset:offset + k] = torch.from_numpy(host).cuda()
            out.append(buf[offset:offset + k])
    out = torch.full((n,), 2.5, device="cuda")
    for zero_first in (True, False):
        want = oracle.decode_accumulate(pairs, out.cpu().numpy().copy(), zero_first)
        plan.decompress_accumulate(d_idx, d_val, None, out, zero_first, ws)
        assert np.array_equal(to_np_u32(out), bits(want)), zero_first
    p0 = np.random.default_rng(n).standard_normal(n).astype(np.float32)
    v0 = (p0 * np.float32(0.1)).astype(np.float32)
    d_p, d_v = (torch.zeros(n + 4, device="cuda")[:n] for _ in range(2))
    d_p.copy_(torch.from_numpy(p0)); d_v.copy_(torch.from_numpy(v0))
    plan.decompress_apply_momentum(d_idx, d_val, None, d_p, d_v, 0.05, 0.9, 0.25, ws)
    oracle.decode_apply_momentum(pairs, p0, v0, 0.05, 0.9, 0.25)
    assert np.array_equal(to_np_u32(d_p), bits(p0)) and np.array_equal(to_np_u32(d_v), bits(v0))
    st, det = plan.last_status(ws)
    assert st == api.GC_OK, (st, det)


@pytest.mark.parametrize("n", [2, 131, 1026, 700_003, 3_000_002])
@pytest.mark.parametrize("W", [1, 40])
def test_momentum_at_the_buffers_end(n, W):
    """The last sub-tile takes the optimizer step like the others, and nothing behind the buffer is written;
    the longer buffers give every CTA one or a few even tiles."""
    plan = api.Plan([n], 0.004, device=0)
    ws = plan.alloc_workspace()
    k = plan.total_cap
    pairs = [synth.sparse_set([n], [k], 40 + w) for w in range(W)]
    d_idx = [torch.from_numpy(i.view(np.int32)).cuda() for i, _ in pairs]
    d_val = [torch.from_numpy(v).cuda() for _, v in pairs]
    p0 = np.random.default_rng(n).standard_normal(n).astype(np.float32)
    v0 = (p0 * np.float32(0.1)).astype(np.float32)
    d_p, d_v = (torch.full((n + 8,), 7.0, device="cuda") for _ in range(2))
    d_p[:n].copy_(torch.from_numpy(p0)); d_v[:n].copy_(torch.from_numpy(v0))
    plan.decompress_apply_momentum(d_idx, d_val, None, d_p[:n], d_v[:n], 0.05, 0.9, 0.25, ws)
    oracle.decode_apply_momentum(pairs, p0, v0, 0.05, 0.9, 0.25)
    assert np.array_equal(to_np_u32(d_p[:n]), bits(p0)) and np.array_equal(to_np_u32(d_v[:n]), bits(v0))
    assert bool((d_p[n:] == 7.0).all()) and bool((d_v[n:] == 7.0).all())
    assert plan.last_status(ws)[0] == api.GC_OK

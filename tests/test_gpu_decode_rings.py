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


@pytest.mark.parametrize("n,density,every", [(300_000, 0.01, 128), (8_000_000, 0.001, 2048)])
@pytest.mark.parametrize("fused", [False, True], ids=["decode", "momentum"])
def test_neighbours_out_of_order_are_reported_or_added(n, density, every, fused):
    """Two neighbouring entries change places across a multiple of `every` (sub-tiles, tiles and the runs of
    the CTAs begin at such places): either both are added all the same, or GC_E_INVALID is recorded."""
    plan = api.Plan([n], density, device=0)
    plan.set_option(api.GC_OPT_DECODE_ROUTE, api.GC_DECODE_WIDE)
    ws = plan.alloc_workspace()
    host, val = synth.sparse_set([n], [plan.total_cap], 5)
    idx, val = torch.from_numpy(host.view(np.int32)).cuda(), torch.from_numpy(val).cuda()
    outs = [torch.zeros(n, device="cuda") for _ in range(2)]

    def call():
        if not fused:
            plan.decompress_accumulate([idx], [val], None, outs[0], True, ws)
            return outs[0]
        for o in outs:
            o.zero_()
        plan.decompress_apply_momentum([idx], [val], None, outs[1], outs[0], 1.0, 0.0, 1.0, ws)
        return outs[0]                                     # the velocity: momentum 0, so the sum itself

    want = call().clone()
    assert plan.last_status(ws)[0] == api.GC_OK
    lost = []
    for p in np.nonzero(np.diff(host // every))[0]:
        for t in (idx, val):
            t[p:p + 2] = t[p:p + 2].flip(0)
        ws[:256].zero_()
        same = torch.equal(call(), want)
        if plan.last_status(ws)[0] != api.GC_E_INVALID and not same:
            lost.append(int(host[p]))
        for t in (idx, val):
            t[p:p + 2] = t[p:p + 2].flip(0)
    assert not lost, lost


@pytest.mark.parametrize("bad", [400_000, 0xFFFFFFFF], ids=["one_beyond", "largest_word"])
@pytest.mark.parametrize("fused", [False, True], ids=["decode", "momentum"])
def test_a_list_with_invalid_entries_does_not_cost_the_others_theirs(bad, fused):
    """The second half of one list is filled with an index beyond the buffer; the other lists crowd into a few
    places, so that their rings end inside a tile.  The bad entries are skipped and reported, everything else
    is added."""
    n, k = 400_000, 4000
    plan = api.Plan([n], k / n, device=0)
    plan.set_option(api.GC_OPT_DECODE_ROUTE, api.GC_DECODE_WIDE)
    assert plan.total_cap == k
    ws = plan.alloc_workspace()
    rng = np.random.default_rng(3)
    crowd = np.concatenate([np.arange(a, a + 1000, dtype=np.uint32) for a in (20_000, 150_000, 200_500, 390_000)])
    spread = np.sort(rng.choice(n // 2, k // 2, replace=False)).astype(np.uint32) + np.uint32(1)
    lists = [crowd, np.concatenate([spread, np.full(k // 2, bad, np.uint32)]), crowd + np.uint32(7)]
    vals = [rng.standard_normal(k).astype(np.float32) for _ in lists]
    pairs = [(i[:k // 2] if w == 1 else i, v[:k // 2] if w == 1 else v) for w, (i, v) in enumerate(zip(lists, vals))]
    d_idx = [torch.from_numpy(i.view(np.int32)).cuda() for i in lists]
    d_val = [torch.from_numpy(v).cuda() for v in vals]
    want = oracle.decode_accumulate(pairs, np.zeros(n, np.float32), True)
    out, other = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
    if fused:
        plan.decompress_apply_momentum(d_idx, d_val, None, other, out, 1.0, 0.0, 1.0, ws)       # the velocity: the sum
    else:
        plan.decompress_accumulate(d_idx, d_val, None, out, True, ws)
    assert plan.last_status(ws)[0] == api.GC_E_INVALID
    assert np.array_equal(to_np_u32(out), bits(want))


@pytest.mark.parametrize("n,density,W", [(300_000, 0.01, 1), ((1 << 20) + 3, 0.02, 2), (2_000_001, 0.2, 2), (3_000_001, 0.003, 16),
                                         (3_000_001, 0.3, 1), (500_001, 1.0, 3), (1_500_000, 0.001, 64), (11_600_000, 0.001, 40),
                                         (11_600_000, 0.001, 3)])
def test_decode_on_both_sides_of_the_route_rules(n, density, W):
    """Sizes, densities and worker counts around the lines between the tile kernel and the rings, dense lists whose
    sub-tiles are bounded by the rings alone, and both kernels on request: plain decode in both modes and the
    momentum step."""
    k = api.Plan([n], density, device=-1).total_cap
    pairs, d_idx, d_val = [], [], []
    for w in range(W):
        idx, _ = synth.sparse_set([n], [k], 300 + (w // 3 if w % 2 else w))
        _, val = synth.sparse_set([n], [k], 700 + w, scale=10.0 ** (w % 5 - 2))
        pairs.append((idx, val))
        d_idx.append(torch.from_numpy(idx.view(np.int32)).cuda())
        d_val.append(torch.from_numpy(val).cuda())
    p0 = np.random.default_rng(n).standard_normal(n).astype(np.float32)
    sums = [oracle.decode_accumulate(pairs, p0.copy(), zero_first) for zero_first in (True, False)]
    p1, v1 = p0.copy(), (p0 * np.float32(0.1)).astype(np.float32)
    v0 = torch.from_numpy(v1.copy())
    oracle.decode_apply_momentum(pairs, p1, v1, 0.05, 0.9, 0.25)
    for route in (api.GC_DECODE_AUTO, api.GC_DECODE_NARROW, api.GC_DECODE_WIDE):
        plan = api.Plan([n], density, device=0)
        plan.set_option(api.GC_OPT_DECODE_ROUTE, route)
        ws = plan.alloc_workspace()
        for want, zero_first in zip(sums, (True, False)):
            out = torch.from_numpy(p0.copy()).cuda()
            plan.decompress_accumulate(d_idx, d_val, None, out, zero_first, ws)
            assert np.array_equal(to_np_u32(out), bits(want)), (route, zero_first)
        d_p, d_v = torch.from_numpy(p0.copy()).cuda(), v0.cuda()
        plan.decompress_apply_momentum(d_idx, d_val, None, d_p, d_v, 0.05, 0.9, 0.25, ws)
        assert np.array_equal(to_np_u32(d_p), bits(p1)) and np.array_equal(to_np_u32(d_v), bits(v1)), route
        assert plan.last_status(ws)[0] == api.GC_OK

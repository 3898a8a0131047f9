"""The append inside a step's attention launch, at the edges of the kernels' tiles: the new
token's rows, position, utility and length, and a sequence without room."""
import math

import pytest
import torch

from paper_2609_03515_gb300 import DecodeCache, ikv

pytestmark = pytest.mark.gpu

LENS = [0, 1, 7, 8, 15, 16, 31, 127, 128, 129, 255, 300]


@pytest.mark.parametrize("gran", [ikv.IKV_GRAN_SEQ, ikv.IKV_GRAN_KVHEAD])
@pytest.mark.parametrize("dtype,d,ps", [(ikv.IKV_BF16, 128, 64), (ikv.IKV_BF16, 128, 24), (ikv.IKV_BF16, 64, 16),
                                        (ikv.IKV_F32, 64, 16), (ikv.IKV_F32, 128, 48)])
def test_step_appends(dtype, d, ps, gran):
    dt = torch.bfloat16 if dtype == ikv.IKV_BF16 else torch.float32
    kvh, G, layers, nb = 2, 4, 3, len(LENS)
    gen = torch.Generator(device="cuda").manual_seed(d + ps)
    c = DecodeCache(nb, layers, G * kvh, kvh, d, max(LENS) + 8, dtype=dtype, page_size=ps, page_perm_seed=2,
                    granularity=gran, value_norms=True)
    c.k.copy_(torch.randn(c.k.shape, generator=gen, device="cuda"))
    c.v.copy_(torch.randn(c.v.shape, generator=gen, device="cuda"))
    c.set_prefill(LENS, [10000] * nb)  # nothing to evict
    c.start.copy_(torch.tensor([(3 * b) % 7 for b in range(nb)], dtype=torch.int32))
    full = nb - 1
    c.start[full] = c.cap - LENS[full]  # no room for its new token
    c.ema.copy_(torch.rand(c.ema.shape, generator=gen, device="cuda"))
    R = c.rows_per_seq
    for b, L in enumerate(LENS):
        for r in range(R):  # every row of a sequence has as many dead slots
            c.pos[b * R + r, torch.randperm(L, generator=gen, device="cuda")[:round(0.15 * L)]] = -1
        if L < c.cap:  # a stale mark in the slot that the new token gets
            c.pos.view(nb, -1, c.cap)[b, :, L] = -1
    q = torch.randn(layers, nb, G * kvh, d, generator=gen, device="cuda").to(dt)
    kn = torch.randn(layers, nb, kvh, d, generator=gen, device="cuda").to(dt)
    vn = torch.randn(layers, nb, kvh, d, generator=gen, device="cuda").to(dt)
    out = torch.full((layers, nb, G * kvh, d), 9.0, device="cuda").to(dt)
    ema0, pos0 = c.ema.clone(), c.pos.clone()
    kv0 = [[[[c.gather(x, b, l, g, L) for g in range(kvh)] for l in range(layers)] for b, L in enumerate(LENS)]
           for x in (c.k, c.v)]
    c.vnorm.copy_(torch.rand(c.vnorm.shape, generator=gen, device="cuda"))
    vnorm0 = c.vnorm.clone()
    holes = 8
    p = c.params(0.5, refresh_period=2, max_holes=holes)
    cch = c.cache(max(LENS), dead_slots=True)
    n = ikv.ikv_step_workspace_size(c.shape(), cch)
    ws = torch.full((n,), 0xAB, dtype=torch.uint8, device="cuda")
    ikv.ikv_step(c.shape(), p, cch, c.ema, 2, q, kn, vn, out, ws, n)  # t = 2: the mean initialisation
    torch.cuda.synchronize()
    assert ikv.ikv_device_status() == 4
    for b, L in enumerate(LENS):
        new = int(b != full)
        dead = round(0.15 * L)
        assert int(c.next_pos[b]) == L + new
        # a sequence compacts only past max_holes dead slots, its order kept
        compacted = dead > holes
        n1 = L + new - (dead if compacted else 0)
        assert int(c.len[b]) == n1, L
        for r in range(R):
            row = b * R + r
            live = pos0[row, :L] >= 0
            mean = float(ema0[row, :L][live].double().mean()) if bool(live.any()) else 0.0
            pos = torch.cat([pos0[row, :L], torch.full((new,), L, dtype=torch.int32, device="cuda")])
            ema = torch.cat([ema0[row, :L], torch.full((new,), mean, device="cuda")])
            lv = pos >= 0
            stay = lv if compacted else torch.ones_like(lv)
            assert torch.equal(c.pos[row, :n1], pos[stay]), (L, r)
            err = (c.ema[row, :n1] - ema[stay]).abs()
            assert float(err.max()) < 1e-5 if n1 else True
            for l in range(layers):
                for g in range(kvh) if R == 1 else [r]:
                    K, V = [torch.cat([x[b][l][g], y[l, b, g][None]][:1 + new]) for x, y in ((kv0[0], kn), (kv0[1], vn))]
                    assert torch.equal(c.gather(c.k, b, l, g, n1), K[stay]), (L, l, g)
                    assert torch.equal(c.gather(c.v, b, l, g, n1), V[stay]), (L, l, g)
                    norm = torch.cat([vnorm0[l, b, g, :L], vn[l, b, g].double().norm().float()[None]][:1 + new])
                    assert torch.allclose(c.vnorm[l, b, g, :n1], norm[stay], rtol=1e-5, atol=0), (L, l, g)
                    z = q[l, b, g * G:(g + 1) * G].double() @ K.double().T / math.sqrt(d)
                    z[:, ~lv] = -math.inf
                    want = torch.softmax(z, -1) @ V.double() if bool(lv.any()) else torch.zeros(G, d, device="cuda")
                    err = (out[l, b, g * G:(g + 1) * G].double() - want).abs().max()
                    assert err < (2e-2 if dtype == ikv.IKV_BF16 else 1e-4), (L, l, g, float(err))


# launches: attention and compaction, and a selection of its own where the bookkeeping CTAs would
# outlast the attention (long rows over few bytes of K and V a slot) or nothing can be deferred
# and the keep list would have left L2
@pytest.mark.parametrize("L,layers,kvh,gran,holes,launches", [
    (300, 3, 2, ikv.IKV_GRAN_KVHEAD, 4, 2), (300, 3, 2, ikv.IKV_GRAN_SEQ, 0, 2),
    (8191, 1, 2, ikv.IKV_GRAN_KVHEAD, 4, 2), (8192, 1, 2, ikv.IKV_GRAN_KVHEAD, 4, 3),
    (8192, 1, 2, ikv.IKV_GRAN_SEQ, 0, 3), (9000, 16, 4, ikv.IKV_GRAN_KVHEAD, 4, 2),
    (2100, 16, 4, ikv.IKV_GRAN_KVHEAD, 0, 3),
])
def test_off_refresh_selection(L, layers, kvh, gran, holes, launches):
    d, G, nb = 128, 2, 2
    gen = torch.Generator(device="cuda").manual_seed(L + layers)
    c = DecodeCache(nb, layers, G * kvh, kvh, d, L + 200, dtype=ikv.IKV_BF16, page_size=64, page_perm_seed=4,
                    granularity=gran)
    c.k.copy_(torch.randn(c.k.shape, generator=gen, device="cuda"))
    c.v.copy_(torch.randn(c.v.shape, generator=gen, device="cuda"))
    c.set_prefill([L] * nb, [L] * nb)
    c.ema.copy_(torch.rand(c.ema.shape, generator=gen, device="cuda"))
    c.ema[:, 17] = c.ema[:, 5]
    c.ema[0, 5] = c.ema[0, 17] = 0.0  # a tie: the higher slot goes
    ema0, pos0 = c.ema.clone(), c.pos.clone()
    k0 = c.gather(c.k, 0, layers - 1, kvh - 1, L)
    q = torch.randn(layers, nb, G * kvh, d, generator=gen, device="cuda").bfloat16()
    kn = torch.randn(layers, nb, kvh, d, generator=gen, device="cuda").bfloat16()
    out = torch.zeros_like(q)
    cch = c.cache(L)
    ws = c.step_workspace()
    before = ikv.ikv_launch_count()
    p = c.params(0.9, refresh_period=4, max_holes=holes)
    ikv.ikv_step(c.shape(), p, cch, c.ema, 2, q, kn, kn, out, ws, ws.numel())
    torch.cuda.synchronize()
    assert ikv.ikv_launch_count() - before == launches
    assert ikv.ikv_device_status() == 0
    assert c.next_pos.tolist() == [L + 1] * nb and c.len.tolist() == [L + (holes > 0)] * nb
    for r in range(c.rows):
        mean = float(ema0[r, :L].double().mean())
        if holes:
            assert abs(float(c.ema[r, L]) - mean) < 1e-5 and int(c.pos[r, L]) == L
        util = torch.cat([ema0[r, :L], torch.tensor([mean], device="cuda")])
        victim = int((util == util.min()).nonzero().max())
        want = torch.cat([pos0[r, :L], torch.tensor([L], dtype=torch.int32, device="cuda")])
        if holes:
            want[victim] = -1
        else:
            want = want[want != victim]
        assert torch.equal(c.pos[r, :want.numel()], want), r
        if r == (kvh if gran == ikv.IKV_GRAN_KVHEAD else 1) - 1:  # the last KV head of sequence 0
            rows = torch.cat([k0, kn[layers - 1, 0, kvh - 1][None]])
            keep = torch.arange(L + 1, device="cuda")
            keep = keep if holes else keep[keep != victim]
            assert torch.equal(c.gather(c.k, 0, layers - 1, kvh - 1, keep.numel()), rows[keep])


@pytest.mark.parametrize("dtype,d", [(ikv.IKV_BF16, 128), (ikv.IKV_F32, 64)])
def test_step_lengths_without_eviction(dtype, d):
    """Lengths and positions over steps that evict nothing, then defer, then compact."""
    dt = torch.bfloat16 if dtype == ikv.IKV_BF16 else torch.float32
    for mode in (ikv.IKV_COMPACT_STABLE, ikv.IKV_COMPACT_STABLE_SHORT, ikv.IKV_COMPACT_HOLEFILL):
        lens, budget, holes = [5, 40, 130], [9, 38, 130], 3
        c = DecodeCache(3, 2, 4, 2, d, 400, dtype=dtype, page_size=16, page_perm_seed=2)
        c.k.normal_()
        c.v.normal_()
        c.set_prefill(lens, budget)
        ws = c.step_workspace()
        L, live = list(lens), list(lens)
        z = torch.randn(2, 3, 2, d, device="cuda").to(dt)
        q = torch.randn(2, 3, 4, d, device="cuda").to(dt)
        out = torch.empty_like(q)
        for t in range(1, 12):
            p = c.params(0.9, refresh_period=2, max_holes=holes, compact_mode=mode, ws_zeroed=t > 1)
            ikv.ikv_step(c.shape(), p, c.cache(max(L)), c.ema, t, q, z, z, out, ws, ws.numel())
            L = [x + 1 for x in L]
            live = [x + 1 for x in live]
            for b in range(3):
                kept = min(live[b], budget[b])
                if not L[b] - kept <= holes:
                    L[b] = kept
                live[b] = kept
            assert c.len.cpu().tolist() == L, (mode, t)
            assert c.next_pos.cpu().tolist() == [x + t for x in lens]
            for b in range(3):
                pos = c.pos[b, :L[b]].cpu()
                assert int((pos >= 0).sum()) == live[b]
                assert pos[pos >= 0].unique().numel() == live[b]
        assert ikv.ikv_device_status() == 0

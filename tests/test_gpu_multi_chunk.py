"""Units of 2 to 8 chunks in launches of two waves or more: a step's utilities and outputs
against fp64 PyTorch, with ragged lengths, start offsets and dead slots; and the outputs do
not depend on whether the step scores."""
import math

import pytest
import torch

from paper_2609_03515_gb300 import DecodeCache, ikv

pytestmark = pytest.mark.gpu

LAYERS = 19  # batch x kv heads x 19 layers x chunks fills whole waves of 2 x 152 CTAs


@pytest.mark.parametrize("lens,kvh,G,ps,gran", [
    ([1921, 3600, 1, 200, 0, 1920, 3000, 1793], 4, 8, 128, ikv.IKV_GRAN_SEQ),   # 2 chunks at most
    ([3713, 1920, 5500, 129, 128, 4000, 17, 5376], 4, 7, 64, ikv.IKV_GRAN_KVHEAD),  # 3
    ([7400, 2000, 0, 3841], 2, 7, 128, ikv.IKV_GRAN_SEQ),          # 4
    ([15000, 1700], 2, 7, 256, ikv.IKV_GRAN_KVHEAD),              # 8
    ([14000, 13441], 2, 8, 64, ikv.IKV_GRAN_SEQ),                 # 8
])
def test_multi_chunk_units(lens, kvh, G, ps, gran):
    d, nb, H = 128, len(lens), kvh * G
    gen = torch.Generator(device="cuda").manual_seed(sum(lens))
    c = DecodeCache(nb, LAYERS, H, kvh, d, max(lens) + 130, dtype=ikv.IKV_BF16, page_size=ps, page_perm_seed=2,
                    granularity=gran)
    c.k.copy_(torch.randn(c.k.shape, generator=gen, device="cuda"))
    c.v.copy_(torch.randn(c.v.shape, generator=gen, device="cuda"))
    c.set_prefill(lens, [10 ** 6] * nb)  # nothing to evict
    c.start.copy_(torch.tensor([(29 * b) % 97 for b in range(nb)], dtype=torch.int32))
    c.ema.copy_(1e-3 * torch.rand(c.ema.shape, generator=gen, device="cuda"))
    R = c.rows_per_seq
    # the same number of dead slots in every row of a sequence, below the compaction limit
    for b, L in enumerate(lens):
        for r in range(R):
            c.pos[b * R + r, torch.randperm(L, generator=gen, device="cuda")[:L // 10]] = -1
    pos0, ema0 = c.pos.clone(), c.ema.clone()
    q = (2.0 * torch.randn(LAYERS, nb, H, d, generator=gen, device="cuda")).bfloat16()
    kn = torch.randn(LAYERS, nb, kvh, d, generator=gen, device="cuda").bfloat16()
    vn = torch.randn(LAYERS, nb, kvh, d, generator=gen, device="cuda").bfloat16()
    out = torch.full((LAYERS, nb, H, d), 9.0, device="cuda").bfloat16()
    alpha = 0.9
    p = c.params(alpha, refresh_period=1, max_holes=10 ** 6)
    cch = c.cache(max(lens), dead_slots=True)
    n = ikv.ikv_step_workspace_size(c.shape(), cch)
    ws = torch.full((n,), 0xAB, dtype=torch.uint8, device="cuda")
    for rep in range(2):  # the same step twice: the counters are left ready
        c.set_prefill(lens, [10 ** 6] * nb)
        c.start.copy_(torch.tensor([(29 * b) % 97 for b in range(nb)], dtype=torch.int32))
        c.pos.copy_(pos0)
        c.ema.copy_(ema0)
        ikv.ikv_step(c.shape(), p, cch, c.ema, 1, q, kn, vn, out, ws, n)
    torch.cuda.synchronize()
    assert ikv.ikv_device_status() == 0
    # the same token in a step that does not score: the same attention, bit for bit
    got_ema, got_len, out1 = c.ema.clone(), c.len.clone(), torch.zeros_like(out)
    c.set_prefill(lens, [10 ** 6] * nb)
    c.start.copy_(torch.tensor([(29 * b) % 97 for b in range(nb)], dtype=torch.int32))
    c.pos.copy_(pos0)
    c.ema.copy_(ema0)
    ikv.ikv_step(c.shape(), c.params(alpha, refresh_period=2, max_holes=10 ** 6), cch, c.ema, 2, q, kn, vn, out1, ws, n)
    torch.cuda.synchronize()
    assert ikv.ikv_device_status() == 0
    assert torch.equal(out, out1)
    c.ema.copy_(got_ema)
    assert torch.equal(c.len, got_len)
    for b, L in enumerate(lens):
        assert int(c.len[b]) == L + 1
        want = torch.cat([ema0.view(nb, R, -1)[b, :, :L].double(), torch.zeros(R, 1, device="cuda").double()], 1)
        lv = torch.cat([pos0.view(nb, R, -1)[b, :, :L] >= 0, torch.ones(R, 1, dtype=torch.bool, device="cuda")], 1)
        for l in range(LAYERS):
            s = torch.zeros_like(want)
            for g in range(kvh):
                r = 0 if R == 1 else g
                K = c.gather(c.k, b, l, g, L + 1).double()
                V = c.gather(c.v, b, l, g, L + 1).double()
                assert torch.equal(K[L], kn[l, b, g].double())
                z = q[l, b, g * G:(g + 1) * G].double() @ K.T / math.sqrt(d)
                z[:, ~lv[r]] = -math.inf
                a = torch.softmax(z, -1)
                s[r] += a.sum(0) / (H if R == 1 else G)
                err = (out[l, b, g * G:(g + 1) * G].double() - a @ V).abs().max()
                assert err < 2e-2, (L, l, g, float(err))
            want = alpha * want + (1 - alpha) * s
        got = c.ema.view(nb, R, -1)[b, :, :L + 1].double()
        # fp32 logits of magnitude < 2^6 and their exponentials: 2^-24 * 2^6 relative, times the
        # sums' rounding; 2e-5 leaves a factor of four
        err = ((got - want).abs() / (want.abs() + 1e-7))[lv].max()
        assert err < 2e-5, (L, float(err))

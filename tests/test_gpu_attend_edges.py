"""Single-layer attention, scores and the merge of its splits at the edges of their tiles.

A plain PyTorch fp64 softmax attention over the same rows is the reference.  Bounds: the
utilities' and scores' 2e-5 and the outputs' 1e-4 (fp32) and 2e-2 (bf16 output rounding) are
those of the other attention tests."""
import math

import pytest
import torch

from paper_2609_03515_gb300 import DecodeCache, ikv

pytestmark = pytest.mark.gpu


def _reference(c, layer, q, b, g, L, live):
    """fp64 output [G][D] and probabilities [G][L] of sequence b, KV head g."""
    G = c.q_heads // c.kv_heads
    K = c.gather(c.k, b, layer, g, L).double()
    V = c.gather(c.v, b, layer, g, L).double()
    z = q[b, g * G:(g + 1) * G].double() @ K.T / math.sqrt(c.head_dim)
    z[:, ~live] = -math.inf
    p = torch.softmax(z, -1) if bool(live.any()) else torch.zeros_like(z)
    return p @ V, p


# one token, a warp's group (8 / 16 tokens) and the CTA's four of them, a tile, splits: each
# less one, exact and one more; an empty sequence
EDGES = [0, 1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 129, 511, 513, 2049]


@pytest.mark.parametrize("dtype", [ikv.IKV_F32, ikv.IKV_BF16])
@pytest.mark.parametrize("d,G,ps", [(64, 1, 64), (64, 2, 7), (64, 4, 16), (64, 7, 1), (64, 8, 48), (128, 1, 12),
                                    (128, 2, 80), (128, 4, 3), (128, 7, 48), (128, 8, 100), (128, 4, 64),
                                    (128, 7, 16)])
def test_attention_edges(dtype, d, G, ps):
    dt = torch.bfloat16 if dtype == ikv.IKV_BF16 else torch.float32
    kvh = 2
    gen = torch.Generator(device="cuda").manual_seed(d + G + ps)
    for lens in (EDGES, [5000]):
        starts = [(5 * i) % 23 for i in range(len(lens))]
        c = DecodeCache(len(lens), 2, G * kvh, kvh, d, max(lens) + 40, dtype=dtype, page_size=ps, page_perm_seed=3)
        tc = ikv.ikv_attend_path(c.shape(), c.cache(max(lens))) == ikv.IKV_PATH_TENSOR_CORE
        assert tc == (dtype == ikv.IKV_BF16 and d == 128 and ps in (16, 64))
        if not tc:  # rows no sequence holds are NaN: nothing past a sequence's end may be used
            c.k.fill_(math.nan)
            c.v.fill_(math.nan)
        c.len.copy_(torch.tensor(lens, dtype=torch.int32))
        c.start.copy_(torch.tensor(starts, dtype=torch.int32))
        layer = 1
        for b, L in enumerate(lens):
            for g in range(kvh):
                c.scatter(c.k, b, layer, g, torch.randn(L, d, generator=gen, device="cuda"))
                c.scatter(c.v, b, layer, g, torch.randn(L, d, generator=gen, device="cuda"))
        c.pos.copy_(torch.arange(c.cap, dtype=torch.int32, device="cuda").expand(c.rows, c.cap))
        c.pos[torch.rand(c.pos.shape, generator=gen, device="cuda") < 0.1] = -1
        if len(lens) > 9:
            c.pos[8] = -1  # every slot of a sequence dead
        q = (2.0 * torch.randn(len(lens), G * kvh, d, generator=gen, device="cuda")).to(dt)
        for dead in (False, True):
            out = torch.full((len(lens), G * kvh, d), 9.0, dtype=dt, device="cuda")
            score = torch.full((c.rows, c.cap), -7.0, device="cuda")
            cch = c.cache(max(lens), dead_slots=dead)
            n = ikv.ikv_attend_workspace_size(c.shape(), cch)
            ws = torch.full((n,), 0xAB, dtype=torch.uint8, device="cuda")  # needs no initialisation
            ikv.ikv_decode_attend_score(c.shape(), cch, layer, q, out, score, None, 0.0, ws, n)
            torch.cuda.synchronize()
            assert ikv.ikv_device_status() == 0
            for b, L in enumerate(lens):
                live = c.pos[b, :L] >= 0 if dead else torch.ones(L, dtype=torch.bool, device="cuda")
                pooled = torch.zeros(L, dtype=torch.float64, device="cuda")
                for g in range(kvh):
                    o, p = _reference(c, layer, q, b, g, L, live)
                    pooled += p.sum(0) / (G * kvh)
                    err = (out[b, g * G:(g + 1) * G].double() - o).abs().max()
                    assert err < (2e-2 if dtype == ikv.IKV_BF16 else 1e-4), (L, g, dead, float(err))
                if L:
                    assert (score[b, :L].double() - pooled).abs().max() < 2e-5, (L, dead)
                assert torch.all(score[b, L:] == -7.0)

"""Per-layer eviction's fold over positions: every lane split of the layers, against fp64."""
import math

import pytest
import torch

from paper_2609_03515_gb300 import DecodeCache, ikv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers", [1, 3, 8, 32, 33, 64, 65, 128, 129, 300, 512])
@pytest.mark.parametrize("some", [False, True])
def test_layer_fold(layers, some):
    """The state after a step and every layer's victim (the lowest utility as of its update);
    `some`: every third layer is ineligible, and an off-refresh step follows."""
    n, prefill, d, alpha, nb = 40, 90, 64, 0.7, 2
    gen = torch.Generator(device="cuda").manual_seed(layers)
    c = DecodeCache(nb, layers, 2, 1, d, n + 9, dtype=ikv.IKV_F32, page_size=16, pos_cap=prefill + 8)
    c.k.normal_(generator=gen)
    c.v.normal_(generator=gen)
    c.set_prefill([n] * nb, [n] * nb)
    c.next_pos.fill_(prefill)
    for r in range(nb * layers):
        at = torch.randperm(prefill, generator=gen, device="cuda")[:n]
        c.pos[r, :n] = torch.sort(at).values.to(torch.int32)
    c.pos_state[:, :prefill] = torch.rand(nb, prefill, generator=gen, device="cuda")
    eligible = [not some or l % 3 != 1 for l in range(layers)]
    q = torch.randn(layers, nb, 2, d, generator=gen, device="cuda")
    kn = torch.randn(layers, nb, 1, d, generator=gen, device="cuda")
    out = torch.empty_like(q)
    ws = c.step_workspace()
    for t in ((1, 2) if some else (1,)):
        state, pos = c.pos_state.double().clone(), c.pos.clone()
        K = c.k.double().clone()
        p = c.params(alpha, refresh_period=2, layer_eligible=eligible, evict_mode=ikv.IKV_EVICT_LAYER,
                     compact_mode=ikv.IKV_COMPACT_STABLE, ws_zeroed=t > 1)
        ikv.ikv_step(c.shape(), p, c.cache(n), c.pos_state, t, q, kn, kn, out, ws, ws.numel())
        torch.cuda.synchronize()
        assert ikv.ikv_device_status() == 0
        new = prefill + t - 1
        for b in range(nb):
            m = state[b].clone()
            held = [torch.cat([pos[b * layers + l, :n].long(), torch.tensor([new], device="cuda")]) for l in range(layers)]
            live = torch.zeros(m.shape[0], dtype=torch.bool, device="cuda")
            live[torch.cat(held)] = True
            live[new] = False
            m[new] = 0.0 if t == 1 else m[live].mean()
            live[new] = True
            for l in range(layers):
                if t == 1 and eligible[l]:
                    slots = torch.arange(n, device="cuda")
                    keys = K[l, c.block_table[b, slots // 16].long(), 0, slots % 16]
                    keys = torch.cat([keys, kn[l, b].double()])
                    s = torch.softmax(q[l, b].double() @ keys.T / math.sqrt(d), -1).mean(0)
                    full = torch.zeros_like(m)
                    full[held[l]] = s
                    m = torch.where(live, alpha * m + (1 - alpha) * full, m)
                util = m[held[l]]
                order = torch.sort(util).values
                if order[1] - order[0] > 1e-6:  # (a gap that fp32 keeps)
                    want = held[l][torch.arange(n + 1, device="cuda") != int(util.argmin())]
                    assert torch.equal(c.pos[b * layers + l, :n].long(), want), (t, b, l)
            assert (c.pos_state[b].double() - m).abs().max() < 1e-6, (t, b)

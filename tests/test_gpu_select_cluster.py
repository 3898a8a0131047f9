"""Budgeted selection by clusters of CTAs: bit-exact against a stable sort at the sizes where
the row's parts, the warps' parts and the keys in shared memory begin and end."""
import threading

import pytest
import torch

from paper_2609_03515_gb300 import ikv

pytestmark = pytest.mark.gpu


def _want(util, pos, L, B):
    """Slots kept, ascending: the B largest live utilities, lower slot first among equals."""
    u = util[:L].clone()
    u[u.isnan()] = -float("inf")
    u = u + 0.0  # -0 == +0
    live = torch.arange(L) if pos is None else torch.nonzero(pos[:L] >= 0).flatten()
    nan = util[:L][live].isnan()
    key = u[live]
    # NaN below -inf: two stable sorts, least significant criterion first
    order = torch.sort(key, descending=True, stable=True).indices
    order = order[torch.sort(nan[order].int(), stable=True).indices]
    return torch.sort(live[order[:min(B, live.numel())]]).values


LENS = [0, 1, 2, 31, 33, 511, 512, 513, 1024, 1025, 4095, 4096, 4097, 8191, 8192, 8193, 16385]


LONG = [24576, 24575, 12288, 3071, 6143, 6144, 6145, 9216, 18431, 21504, 1, 0]  # eight CTAs down to one


@pytest.mark.parametrize("rows,cap,lens,ctas", [
    (17, 16448, LENS, 4),
    (19, 24576, LONG, 8),
    (70, 6144, LENS[:13] + [6143, 6144], 2),
    (60, 3000, LENS[:10] + [3000], 1),
    (400, 1500, LENS[:10], 1),
    (1, 70000, [70000], 8),            # one long row
    (400, 70000, [60000, 33], 1),      # more keys than a CTA keeps in shared memory
    (3, 400000, [400000, 70000], 8),   # the same in a cluster
])
@pytest.mark.parametrize("dead", [False, True])
def test_select_cluster_bit_exact(rows, cap, lens, ctas, dead):
    assert ikv.ikv_select_plan(rows, cap)["ctas"] == ctas
    # clusters: every row once with each budget and kind of utility
    for shift in range(1 if ctas == 1 else 28 if cap < 100000 else 7):
        _bit_exact(rows, cap, lens, dead, shift)


def _bit_exact(rows, cap, lens, dead, shift):
    assert max(lens) <= cap
    gen = torch.Generator().manual_seed(rows + cap + shift)
    ln = torch.tensor([lens[r % len(lens)] for r in range(rows)], dtype=torch.int32)
    kinds = ["spread", "ties", "special", "low"]
    util = torch.empty(rows, cap)
    for r in range(min(rows, 40)):
        kind = kinds[(r // len(lens) + r + shift) % 4]
        x = torch.randn(cap, generator=gen)
        if kind == "spread":
            x = torch.exp(4 * x - 9)
        elif kind == "ties":
            x = (x * 2).round() / 4
        elif kind == "special":
            x[torch.rand(cap, generator=gen) < 0.05] = float("nan")
            x[torch.rand(cap, generator=gen) < 0.05] = float("inf")
            x[torch.rand(cap, generator=gen) < 0.05] = -float("inf")
            x[torch.rand(cap, generator=gen) < 0.2] = -0.0
            x[torch.rand(cap, generator=gen) < 0.05] = torch.finfo(torch.float32).min
        else:
            x[:] = 0.0
        util[r] = x
    for r in range(40, rows):
        util[r] = util[r % 40]
    pos = torch.arange(cap, dtype=torch.int32).repeat(rows, 1)
    if dead:
        pos[torch.rand(pos.shape, generator=gen) < 0.1] = -1
    live = [(int((pos[r, :int(ln[r])] >= 0).sum())) for r in range(rows)]
    # none, one, a tenth, all but two, all but one, all, more than there are
    pick = [lambda n: 0, lambda n: 1, lambda n: n // 10, lambda n: max(0, n - 2), lambda n: max(0, n - 1), lambda n: n,
            lambda n: n + 5]
    budget = torch.tensor([pick[(3 * r + r // len(lens) + shift) % 7](live[r]) for r in range(rows)], dtype=torch.int32)
    keep = torch.full((rows, cap), -9, dtype=torch.int32, device="cuda")
    keep_len = torch.full((rows,), -9, dtype=torch.int32, device="cuda")
    ikv.ikv_select_budget(rows, cap, util.cuda(), ln.cuda(), 1, budget.cuda(), pos.cuda() if dead else None, keep,
                          keep_len)
    torch.cuda.synchronize()
    keep, keep_len = keep.cpu(), keep_len.cpu()
    for r in list(range(min(rows, 120))) + [rows - 1]:
        want = _want(util[r], pos[r] if dead else None, int(ln[r]), int(budget[r]))
        assert int(keep_len[r]) == want.numel(), (r, int(ln[r]), int(budget[r]))
        assert torch.equal(keep[r, :want.numel()].long(), want), (r, int(ln[r]), int(budget[r]))
        assert torch.all(keep[r, want.numel():] == -9)


def test_select_sizes_on_two_threads():
    """Selections of different capacities at the same time: the larger is not refused for a
    shared-memory limit that the smaller one set (400 rows: one CTA a row, of the same kernel)."""
    errors = []

    def loop(cap):
        try:
            rows, s = 400, torch.cuda.Stream()
            with torch.cuda.stream(s):
                util = torch.rand(rows, cap, device="cuda")
                ln = torch.full((rows,), 100, dtype=torch.int32, device="cuda")
                keep = torch.zeros(rows, cap, dtype=torch.int32, device="cuda")
                keep_len = torch.zeros(rows, dtype=torch.int32, device="cuda")
                budget = ln - 7
                for _ in range(2000):
                    ikv.ikv_select_budget(rows, cap, util, ln, 1, budget, None, keep, keep_len, s)
            s.synchronize()
            assert int(keep_len.min()) == int(keep_len.max()) == 93
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=loop, args=(cap,)) for cap in (11000, 48000)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors

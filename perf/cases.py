"""The decode-step work this library is used for, as cases that can be timed and compared.

A case is one of four kinds:
  step    whole decode steps (ikv_step, or ikv_step_begin / _layer / _end), in the steady
          state after the prefill was evicted to its budget, or the first step after it;
  attend  ikv_decode_attend_score, layer by layer, folding each layer's score into the utility;
  select  ikv_select_budget on utilities;
  layer   steps under per-layer eviction (every layer keeps its own tokens).

Inputs follow the synthetic decode workloads of gen/: keys and values N(0, 1), a share of
heavy tokens whose keys lie around a per-KV-head direction, the first four positions scaled
(attention sinks), queries around the same directions.
"""
import math

import torch

from paper_2609_03515_gb300 import DecodeCache, ikv

DTYPES = {"bf16": (ikv.IKV_BF16, torch.bfloat16), "f32": (ikv.IKV_F32, torch.float32)}
COMPACT = {"stable": ikv.IKV_COMPACT_STABLE, "short": ikv.IKV_COMPACT_STABLE_SHORT,
           "holefill": ikv.IKV_COMPACT_HOLEFILL}


def _step(name, **kw):
    c = {"name": name, "kind": "step", "batch": 1, "layers": 32, "q_heads": 32, "kv_heads": 8, "head_dim": 128,
         "dtype": "bf16", "page": 64, "prefill_lo": 32768, "prefill_hi": 32768, "budget": 0.1, "refresh": 1,
         "max_holes": 128, "compact": "short", "first": False, "api": "step", "graph": False, "alpha": 0.9}
    c.update(kw)
    return c


def listed():
    return [
        # the tiny fp32 loop (2 layers, 512-token prefill): launches and latency only; the
        # step is replayed from a CUDA graph, as a decode loop of small steps is run
        _step("step_tiny_f32", layers=2, q_heads=4, kv_heads=2, head_dim=64, dtype="f32", prefill_lo=512,
              prefill_hi=512, max_holes=0, graph=True),
        # single-stream decode of the Llama-3.1-8B shape at 32k, 10% budget, full refresh:
        # the headline workload in its steady state
        _step("step_b1_32k"),
        # its first step: the whole prefill is scored, 90% of it evicted, the rest compacted
        _step("first_b1_32k", first=True),
        # the same steady state driven layer by layer, as a model that has layer l's q, k, v
        # only after layer l - 1 does it, captured in the model's step graph
        _step("layers_b1_32k", api="layers", graph=True),
        # batched serving, ragged lengths, Lazy4: one pass is one period (a refresh step and
        # three attention-only steps)
        _step("lazy4_b16_ragged", batch=16, prefill_lo=4096, prefill_hi=8192, refresh=4),
        # the largest: Qwen-2.5-7B shape (group of 7), b = 32, 16k prefill, 25% budget
        _step("step_qwen_b32_25", batch=32, layers=28, q_heads=28, kv_heads=4, prefill_lo=16384, prefill_hi=16384,
              budget=0.25),
        # bf16 heads of 64 dims (the other head size the library takes), small pages
        _step("step_d64_bf16", batch=8, layers=16, head_dim=64, page=16, prefill_lo=8192, prefill_hi=8192,
              budget=0.25, max_holes=64),
        # fp32 caches (accuracy studies): 128-dim heads, half budget
        _step("step_f32_b4", batch=4, layers=8, q_heads=16, kv_heads=4, dtype="f32", prefill_lo=4096, prefill_hi=4096,
              budget=0.5, max_holes=64),
        # one layer at a time through the workspace entry point, utility updated after each
        # layer; single stream, inside the model's graph
        {"name": "attend_b1", "kind": "attend", "batch": 1, "layers": 32, "q_heads": 32, "kv_heads": 8,
         "head_dim": 128, "dtype": "bf16", "page": 64, "len_lo": 3277, "len_hi": 3277, "gran": "seq", "graph": True,
         "alpha": 0.8},
        # the same at a long context and a large batch, one utility row per KV head
        {"name": "attend_b32_16k", "kind": "attend", "batch": 32, "layers": 2, "q_heads": 28, "kv_heads": 4,
         "head_dim": 128, "dtype": "bf16", "page": 128, "len_lo": 12000, "len_hi": 16384, "gran": "kvhead",
         "graph": False, "alpha": 0.9},
        # the eviction decision of a batch after a 16k prefill
        {"name": "select_32x16k", "kind": "select", "rows": 32, "len_lo": 16385, "len_hi": 16385, "budget": 0.1},
        # per-layer eviction: every layer scores, then evicts from its own token set
        {"name": "layer_evict_b1", "kind": "layer", "batch": 1, "layers": 32, "q_heads": 32, "kv_heads": 8,
         "head_dim": 128, "dtype": "bf16", "page": 64, "prefill": 32768, "budget": 0.1, "compact": "holefill",
         "alpha": 0.9},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    return work(c)["bytes"]


_LIMIT = 7.0e9  # bytes of a drawn pass: below the largest listed case's


def draw(rng):
    while True:
        c = _draw(rng)
        if _cost(c) <= _LIMIT:
            return c


def _heads(rng):
    g = rng.choice([1, 2, 4, 4, 7, 8])
    hkv = rng.choice([2, 4, 8])
    return g * hkv, hkv


def _draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "step", "attend", "attend", "select", "layer"])
    qh, kvh = _heads(rng)
    if kind == "select":
        hi = _logint(rng, 600, 66000)
        return {"kind": "select", "rows": _logint(rng, 1, 64), "len_lo": max(1, int(hi * rng.uniform(0.5, 1.0))),
                "len_hi": hi, "budget": rng.choice([0.1, 0.25, 0.5])}
    if kind == "attend":
        hi = _logint(rng, 300, 20000)
        return {"kind": "attend", "batch": _logint(rng, 1, 32), "layers": rng.choice([2, 8, 32]), "q_heads": qh,
                "kv_heads": kvh, "head_dim": rng.choice([128, 128, 128, 64]),
                "dtype": rng.choice(["bf16", "bf16", "bf16", "f32"]), "page": rng.choice([16, 64, 128]),
                "len_lo": max(1, int(hi * rng.uniform(0.5, 1.0))), "len_hi": hi,
                "gran": rng.choice(["seq", "kvhead"]), "graph": True, "alpha": rng.choice([0.5, 0.8, 0.9, 0.99])}
    if kind == "layer":
        return {"kind": "layer", "batch": rng.choice([1, 1, 2, 4]), "layers": rng.choice([16, 28, 32]), "q_heads": qh,
                "kv_heads": kvh, "head_dim": 128, "dtype": "bf16", "page": rng.choice([16, 64]),
                "prefill": _logint(rng, 4096, 33000), "budget": rng.choice([0.1, 0.25]), "compact": "holefill",
                "alpha": 0.9}
    hi = _logint(rng, 512, 33000)
    c = _step("", batch=_logint(rng, 1, 32), layers=rng.choice([2, 8, 16, 28, 32]), q_heads=qh, kv_heads=kvh,
              head_dim=rng.choice([128, 128, 128, 64]), dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]),
              page=rng.choice([16, 64, 128]), prefill_lo=max(64, int(hi * rng.uniform(0.5, 1.0))), prefill_hi=hi,
              budget=rng.choice([0.1, 0.25, 0.5]), refresh=rng.choice([1, 1, 2, 4]),
              max_holes=rng.choice([0, 64, 128]), compact=rng.choice(["short", "short", "stable"]),
              first=rng.random() < 0.2, api=rng.choice(["step", "step", "layers"]),
              alpha=rng.choice([0.5, 0.8, 0.9, 0.99]))
    del c["name"]
    c["graph"] = c["refresh"] == 1 and not c["first"] and (c["api"] == "layers" or rng.random() < 0.5)
    if c["first"]:
        c["refresh"], c["api"] = 1, "step"
    elif c["api"] == "layers":
        c["refresh"], c["graph"] = 1, True
    return c


# ---------------------------------------------------------------- sizes
def _spread(lo, hi, n):
    """n lengths over [lo, hi], ragged and fixed by the sizes alone."""
    if lo == hi or n == 1:
        return [hi] * n
    return [lo + (hi - lo) * ((i * 7919 + 3) % 997) // 996 for i in range(n)]


def _lens(case):
    """(prefill lengths, budgets, lengths the pass starts from)"""
    if case["kind"] == "attend":
        n = _spread(case["len_lo"], case["len_hi"], case["batch"])
        return n, n, n
    if case["kind"] == "layer":
        n = [case["prefill"]] * case["batch"]
    else:
        n = _spread(case["prefill_lo"], case["prefill_hi"], case["batch"])
    b = [max(1, int(math.floor(case["budget"] * x + 0.5))) for x in n]
    return n, b, (n if case.get("first") else b)


def work(case):
    if case["kind"] == "select":
        lens = _spread(case["len_lo"], case["len_hi"], case["rows"])
        kept = [max(1, int(n * case["budget"])) for n in lens]
        return {"bytes": 4 * (sum(lens) + sum(kept)), "flops": sum(lens)}
    eb = 4 if case["dtype"] == "f32" else 2
    K, H, G, D, nb = case["layers"], case["q_heads"], case["kv_heads"], case["head_dim"], case["batch"]
    _, budget, lens = _lens(case)
    new = 0 if case["kind"] == "attend" else 1
    tok = sum(n + new for n in lens)
    steps = case.get("refresh", 1)
    by = tok * K * G * D * 2 * eb + 2 * nb * K * H * D * eb + new * 2 * nb * K * G * D * 2 * eb
    fl = 4 * tok * K * H * D
    if case["kind"] == "attend":
        rows = G if case["gran"] == "kvhead" else 1
        st = tok * rows * K * 12  # each call: the utility read and written, the score written
        return {"bytes": by + st, "flops": fl}
    by, fl = by * steps, fl * steps
    by += tok * 8  # the utility, read and written on the refresh step
    if case.get("first"):
        by += sum(budget) * K * G * D * 2 * eb  # the survivors' rows written
    return {"bytes": by, "flops": fl}


def tolerance(case):
    if case["kind"] == "select":
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "differ": 0.002}
    return {"rel": 1e-2, "differ": 0.002}


# ---------------------------------------------------------------- inputs
def _generator(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(seed)


def _cap(case):
    _, budget, lens = _lens(case)
    if case["kind"] == "attend":
        return max(lens) + 1
    if case.get("first"):
        return max(lens) + 1 + case["max_holes"]
    # the pages a server keeps for a sequence once its prefill was evicted
    return max(budget) + max(budget) // 4 + case.get("max_holes", 0) + 256


def _inputs(case, seed):
    """The tensors of a case, from the seed alone: pools, block table, queries, new tokens."""
    gen = _generator(seed)
    dt = DTYPES[case["dtype"]][1]
    K, H, G, D, nb, ps = (case["layers"], case["q_heads"], case["kv_heads"], case["head_dim"], case["batch"],
                          case["page"])
    n0, budget, lens = _lens(case)
    max_pages = (_cap(case) + ps - 1) // ps
    pages = torch.randperm(nb * max_pages, generator=gen, device="cuda").to(torch.int32).view(nb, max_pages)
    shape = (K, nb * max_pages, G, ps, D)
    k = torch.empty(shape, dtype=dt, device="cuda").normal_(generator=gen)
    v = torch.empty(shape, dtype=dt, device="cuda").normal_(generator=gen)
    u = torch.nn.functional.normalize(torch.randn(K, G, D, generator=gen, device="cuda"), dim=-1) * 8.0
    # heavy tokens: 1% of the prefill; eviction keeps them, so their share grows as it shrinks
    share = 0.01 if lens == n0 else min(0.5, 0.01 / case["budget"])
    for b in range(nb):
        n = lens[b]
        m = max(1, int(n * share))
        slots = torch.randperm(n, generator=gen, device="cuda")[:m]
        pg, off = pages[b, slots // ps].long(), slots % ps
        noise = 0.3 * torch.randn(m, K, G, D, generator=gen, device="cuda")
        k[:, pg, :, off] = (3.0 * u + noise).to(dt)
        sink = torch.arange(min(4, n), device="cuda")
        pg, off = pages[b, sink // ps].long(), sink % ps
        k[:, pg, :, off] = (4.0 * k[:, pg, :, off].float()).to(dt)
    sets = 1 if case.get("graph") or case["kind"] == "attend" else max(2, case.get("refresh", 1))
    uq = u.repeat_interleave(H // G, dim=1)
    q, kn, vn = [], [], []
    for _ in range(sets):
        w = uq[:, None] + 0.5 * torch.randn(K, nb, H, D, generator=gen, device="cuda")
        q.append((8.0 * torch.nn.functional.normalize(w, dim=-1)).to(dt))
        kn.append(torch.randn(K, nb, G, D, generator=gen, device="cuda").to(dt))
        vn.append(torch.randn(K, nb, G, D, generator=gen, device="cuda").to(dt))
    return {"k": k, "v": v, "pages": pages, "max_pages": max_pages, "q": q, "kn": kn, "vn": vn, "gen": gen}


def _utility(n_rows, n, gen):
    """Utilities of a steady state: spread over decades, as the softmax leaves them."""
    return torch.exp(3.0 * torch.randn(n_rows, n, generator=gen, device="cuda") - 9.0)


def _positions(n, prefill, gen):
    return torch.sort(torch.randperm(prefill, generator=gen, device="cuda")[:n]).values.to(torch.int32)


def _cache(case, inp, **kw):
    """The caller's cache on those inputs (DecodeCache allocates; the pools are replaced)."""
    cap = inp["max_pages"] * case["page"]
    c = DecodeCache(case["batch"], 1, case["q_heads"], case["kv_heads"], case["head_dim"], cap,
                    dtype=DTYPES[case["dtype"]][0], page_size=case["page"], **kw)
    c.layers = case["layers"]
    c.k, c.v, c.block_table = inp["k"], inp["v"], inp["pages"]
    return c


def _flat(*tensors):
    """The tensors as views of one buffer, so that one copy rewinds them all."""
    sizes = [(t.numel() + 3) // 4 * 4 for t in tensors]
    buf = torch.zeros(sum(sizes), dtype=torch.int32, device="cuda")
    out, at = [], 0
    for t, n in zip(tensors, sizes):
        w = buf[at:at + t.numel()].view(t.dtype).view(t.shape)
        w.copy_(t)
        out.append(w)
        at += n
    return buf, out


def _graph(fn):
    """fn's work captured once; a side stream warms it up, as capture asks for."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            fn(s)
    torch.cuda.current_stream().wait_stream(s)
    return g


def prepare(case, seed):
    return {"select": _prepare_select, "attend": _prepare_attend, "layer": _prepare_layer,
            "step": _prepare_step}[case["kind"]](case, seed)


def run(state):
    return state["run"](state)


# ---------------------------------------------------------------- select
def _prepare_select(case, seed):
    gen = _generator(seed)
    lens = _spread(case["len_lo"], case["len_hi"], case["rows"])
    cap = (max(lens) + 64) // 64 * 64
    util = _utility(case["rows"], cap, gen)
    util[torch.rand(util.shape, generator=gen, device="cuda") < 0.001] = 0.0  # tokens scored 0: ties
    i32 = {"dtype": torch.int32, "device": "cuda"}
    return {"run": _run_select, "rows": case["rows"], "cap": cap, "util": util, "len": torch.tensor(lens, **i32),
            "budget": torch.tensor([max(1, int(n * case["budget"])) for n in lens], **i32),
            "keep": torch.zeros(case["rows"], cap, **i32), "keep_len": torch.zeros(case["rows"], **i32)}


def _run_select(s):
    ikv.ikv_select_budget(s["rows"], s["cap"], s["util"], s["len"], 1, s["budget"], None, s["keep"], s["keep_len"],
                          torch.cuda.current_stream())
    return [s["keep"], s["keep_len"]]


# ---------------------------------------------------------------- attend
def _prepare_attend(case, seed):
    inp = _inputs(case, seed)
    gran = ikv.IKV_GRAN_KVHEAD if case["gran"] == "kvhead" else ikv.IKV_GRAN_SEQ
    c = _cache(case, inp, granularity=gran)
    lens = _lens(case)[2]
    c.set_prefill(lens, lens)
    c.ema.copy_(_utility(c.rows, c.cap, inp["gen"]))
    shape, cache = c.shape(), c.cache()
    nbytes = ikv.ikv_attend_workspace_size(shape, cache)
    s = {"run": _run_attend, "c": c, "shape": shape, "cache": cache, "q": inp["q"][0], "alpha": case["alpha"],
         "ws": torch.empty(nbytes, dtype=torch.uint8, device="cuda"), "nbytes": nbytes,
         "out": torch.zeros_like(inp["q"][0]),
         "score": torch.zeros(case["layers"], c.rows, c.cap, dtype=torch.float32, device="cuda")}
    if case["graph"]:
        s["graph"] = _graph(lambda st: _layers_attend(s, st))
    return s


def _layers_attend(s, stream):
    for layer in range(s["c"].layers):
        ikv.ikv_decode_attend_score(s["shape"], s["cache"], layer, s["q"][layer], s["out"][layer], s["score"][layer],
                                    s["c"].ema, s["alpha"], s["ws"], s["nbytes"], stream)


def _run_attend(s):
    if "graph" in s:
        s["graph"].replay()
    else:
        _layers_attend(s, torch.cuda.current_stream())
    return [s["out"], s["score"], s["c"].ema]


# ---------------------------------------------------------------- steps
def _prepare_step(case, seed):
    inp = _inputs(case, seed)
    c = _cache(case, inp)
    n0, budget, lens = _lens(case)
    c.set_prefill(lens, budget)
    if not case["first"]:
        for b in range(case["batch"]):
            c.ema[b, :lens[b]] = _utility(1, lens[b], inp["gen"])[0]
            c.pos[b, :lens[b]] = _positions(lens[b], n0[b], inp["gen"])
        c.next_pos.copy_(torch.tensor(n0, dtype=torch.int32))
    s = {"run": _run_step, "c": c, "q": inp["q"], "kn": inp["kn"], "vn": inp["vn"], "api": case["api"],
         "out": [torch.zeros_like(inp["q"][0]) for _ in range(case["refresh"])], "steps": case["refresh"], "t": 1}
    if case["first"]:  # the pass starts over from the prefill's bookkeeping
        s["live"], (c.len, c.next_pos, c.start, c.pos, c.ema) = _flat(c.len, c.next_pos, c.start, c.pos, c.ema)
        s["saved"] = s["live"].clone()
    s["shape"] = c.shape()
    # bound on len before a step's append: dead slots included once compaction is deferred
    s["cache"] = c.cache(max(lens) if case["first"] else max(budget) + case["max_holes"])
    s["params"] = c.params(case["alpha"], refresh_period=case["refresh"], compact_mode=COMPACT[case["compact"]],
                           max_holes=case["max_holes"], ws_zeroed=True)
    s["ws"] = torch.zeros(ikv.ikv_step_workspace_size(s["shape"], s["cache"]), dtype=torch.uint8, device="cuda")
    if case["graph"]:
        s["graph"] = _graph(lambda st: _one_step(s, 1, 0, st))
    return s


def _one_step(s, t, i, stream):
    c, ws = s["c"], s["ws"]
    q, kn, vn, out = s["q"][i % len(s["q"])], s["kn"][i % len(s["q"])], s["vn"][i % len(s["q"])], s["out"][i % s["steps"]]
    if s["api"] == "step":
        ikv.ikv_step(s["shape"], s["params"], s["cache"], c.ema, t, q, kn, vn, out, ws, ws.numel(), stream)
        return
    ikv.ikv_step_begin(s["shape"], s["params"], s["cache"], c.ema, t, ws, ws.numel(), stream)
    for layer in range(c.layers):
        ikv.ikv_step_layer(s["shape"], s["params"], s["cache"], c.ema, t, layer, q[layer], kn[layer], vn[layer],
                           out[layer], ws, ws.numel(), stream)
    ikv.ikv_step_end(s["shape"], s["params"], s["cache"], c.ema, t, ws, ws.numel(), stream)


def _run_step(s):
    c = s["c"]
    if "graph" in s:
        s["graph"].replay()
    elif "saved" in s:
        s["live"].copy_(s["saved"])
        _one_step(s, 1, 0, torch.cuda.current_stream())
    else:
        stream = torch.cuda.current_stream()
        for _ in range(s["steps"]):  # a period of the schedule: its refresh step first
            _one_step(s, s["t"], s["t"] - 1, stream)
            s["t"] += 1
    return s["out"] + [c.ema, c.pos, c.len, c.k, c.v]


# ---------------------------------------------------------------- per-layer eviction
def _prepare_layer(case, seed):
    inp = _inputs(case, seed)
    n0, budget, lens = _lens(case)
    pos_cap = case["prefill"] + 64
    c = _cache(case, inp, pos_cap=pos_cap)
    c.pos = torch.zeros(case["batch"] * case["layers"], c.cap, dtype=torch.int32, device="cuda")
    c.set_prefill(lens, budget)
    # every layer holds its own tokens; most are shared, as the layers' utilities agree
    for b in range(case["batch"]):
        shared = torch.randperm(n0[b], generator=inp["gen"], device="cuda")
        for layer in range(case["layers"]):
            most = shared[:lens[b] * 7 // 8]
            rest = shared[lens[b] * 7 // 8:min(n0[b], lens[b] * 5 // 4)]
            rest = rest[torch.randperm(rest.numel(), generator=inp["gen"], device="cuda")[:lens[b] - most.numel()]]
            c.pos[b * case["layers"] + layer, :lens[b]] = torch.sort(torch.cat([most, rest])).values.to(torch.int32)
        c.pos_state[b, :n0[b]] = _utility(1, n0[b], inp["gen"])[0]
    c.next_pos.copy_(torch.tensor(n0, dtype=torch.int32))
    # the positions are bounded by pos_cap, so a pass starts over from the same bookkeeping
    buf, (c.len, c.next_pos, c.pos, c.pos_state) = _flat(c.len, c.next_pos, c.pos, c.pos_state)
    s = {"run": _run_layer, "c": c, "live": buf, "saved": buf.clone(), "q": inp["q"], "kn": inp["kn"], "vn": inp["vn"],
         "out": [torch.zeros_like(inp["q"][0])], "steps": 1, "api": "step", "shape": c.shape(),
         "cache": c.cache(max(budget))}
    s["params"] = c.params(case["alpha"], compact_mode=COMPACT[case["compact"]], evict_mode=ikv.IKV_EVICT_LAYER,
                           ws_zeroed=True)
    s["ws"] = torch.zeros(ikv.ikv_step_workspace_size(s["shape"], s["cache"]), dtype=torch.uint8, device="cuda")
    return s


def _run_layer(s):
    c = s["c"]
    s["live"].copy_(s["saved"])
    ikv.ikv_step(s["shape"], s["params"], s["cache"], c.pos_state, 1, s["q"][0], s["kn"][0], s["vn"][0], s["out"][0],
                 s["ws"], s["ws"].numel(), torch.cuda.current_stream())
    return s["out"] + [c.pos_state, c.pos, c.len, c.k, c.v]


# ---------------------------------------------------------------- the same in 64 bits
def _rows64(pool, pages, layer, b, n, ps):
    slots = torch.arange(n, device="cuda")
    return pool[layer, pages[b, slots // ps].long(), :, slots % ps].double()  # [n][G][D]


def _attend64(q, k, v, dead=None):
    """q [H][D], k / v [n][G][D] -> (out [H][D], probabilities [H][n])"""
    H, D = q.shape
    n, G, _ = k.shape
    z = torch.einsum("grd,ngd->grn", q.double().view(G, H // G, D), k) / math.sqrt(D)
    if dead is not None:
        z[:, :, dead] = -math.inf
    p = torch.softmax(z, dim=-1)
    return torch.einsum("grn,ngd->grd", p, v).reshape(H, D), p.reshape(H, n)


def exact(case, seed):
    return {"select": lambda c, s: None, "attend": _exact_attend, "layer": _exact_layer,
            "step": _exact_step}[case["kind"]](case, seed)


def _exact_attend(case, seed):
    inp = _inputs(case, seed)
    K, H, G, nb, ps = case["layers"], case["q_heads"], case["kv_heads"], case["batch"], case["page"]
    lens = _lens(case)[2]
    rows = nb * G if case["gran"] == "kvhead" else nb
    cap = inp["max_pages"] * ps
    ema = _utility(rows, cap, inp["gen"]).double()
    out = torch.zeros(inp["q"][0].shape, dtype=torch.float64, device="cuda")
    score = torch.zeros(K, rows, cap, dtype=torch.float64, device="cuda")
    per = rows // nb
    for layer in range(K):
        for b in range(nb):
            n = lens[b]
            o, p = _attend64(inp["q"][0][layer, b], _rows64(inp["k"], inp["pages"], layer, b, n, ps),
                             _rows64(inp["v"], inp["pages"], layer, b, n, ps))
            out[layer, b] = o
            score[layer, b * per:(b + 1) * per, :n] = p.view(per, H // per, n).mean(1)
            r = slice(b * per, (b + 1) * per)
            ema[r, :n] = case["alpha"] * ema[r, :n] + (1 - case["alpha"]) * score[layer, r, :n]
    return [out, score, ema]


def _exact_step(case, seed):
    inp = _inputs(case, seed)
    K, nb, ps, cap = case["layers"], case["batch"], case["page"], inp["max_pages"] * case["page"]
    n0, budget, lens = _lens(case)
    ema = torch.zeros(nb, cap, dtype=torch.float64, device="cuda")
    if not case["first"]:
        for b in range(nb):
            ema[b, :lens[b]] = _utility(1, lens[b], inp["gen"])[0].double()
            _positions(lens[b], n0[b], inp["gen"])
    outs = [torch.zeros(inp["q"][0].shape, dtype=torch.float64, device="cuda") for _ in range(case["refresh"])]
    # compaction moves slots between the steps of a pass; deferred, they stay where they are
    if case["refresh"] > 1 and case["max_holes"] < case["refresh"]:
        return None
    for b in range(nb):
        n, dead = lens[b], torch.zeros(cap, dtype=torch.bool, device="cuda")
        new_k, new_v = [[] for _ in range(K)], [[] for _ in range(K)]
        for i in range(case["refresh"]):
            j = i % len(inp["q"])
            live = ~dead[:n]
            ema[b, n] = 0.0 if i == 0 else ema[b, :n][live].mean()
            n += 1
            for layer in range(K):
                new_k[layer].append(inp["kn"][j][layer, b].double())
                new_v[layer].append(inp["vn"][j][layer, b].double())
                k = torch.cat([_rows64(inp["k"], inp["pages"], layer, b, lens[b], ps), torch.stack(new_k[layer])])
                v = torch.cat([_rows64(inp["v"], inp["pages"], layer, b, lens[b], ps), torch.stack(new_v[layer])])
                o, p = _attend64(inp["q"][j][layer, b], k, v, dead[:n])
                outs[i][layer, b] = o
                if i == 0:
                    ema[b, :n] = case["alpha"] * ema[b, :n] + (1 - case["alpha"]) * p.mean(0)
            if case["first"]:
                continue
            m = ema[b, :n].clone()
            m[dead[:n]] = math.inf
            low = int((m == m.min()).nonzero().max())  # the highest slot among equals
            if case["max_holes"] > 0:
                dead[low] = True
            else:
                ema[b, :n - 1] = torch.cat([ema[b, :low], ema[b, low + 1:n]])
                n -= 1
    return outs + [None if case["first"] else ema, None, None, None, None]


def _exact_layer(case, seed):
    inp = _inputs(case, seed)
    K, nb, ps = case["layers"], case["batch"], case["page"]
    n0, budget, lens = _lens(case)
    out = torch.zeros(inp["q"][0].shape, dtype=torch.float64, device="cuda")
    state = torch.zeros(nb, case["prefill"] + 64, dtype=torch.float64, device="cuda")
    for b in range(nb):
        shared = torch.randperm(n0[b], generator=inp["gen"], device="cuda")
        held = []
        for layer in range(K):
            most = shared[:lens[b] * 7 // 8]
            rest = shared[lens[b] * 7 // 8:min(n0[b], lens[b] * 5 // 4)]
            rest = rest[torch.randperm(rest.numel(), generator=inp["gen"], device="cuda")[:lens[b] - most.numel()]]
            held.append(torch.sort(torch.cat([most, rest])).values)
        state[b, :n0[b]] = _utility(1, n0[b], inp["gen"])[0].double()
        live = torch.zeros(state.shape[1], dtype=torch.bool, device="cuda")
        live[torch.cat(held)] = True
        live[n0[b]] = True
        for layer in range(K):
            at = torch.cat([held[layer], torch.tensor([n0[b]], device="cuda")])
            k = torch.cat([_rows64(inp["k"], inp["pages"], layer, b, lens[b], ps),
                           inp["kn"][0][layer, b][None].double()])
            v = torch.cat([_rows64(inp["v"], inp["pages"], layer, b, lens[b], ps),
                           inp["vn"][0][layer, b][None].double()])
            o, p = _attend64(inp["q"][0][layer, b], k, v)
            out[layer, b] = o
            s = torch.zeros(state.shape[1], dtype=torch.float64, device="cuda")
            s[at] = p.mean(0)
            state[b] = torch.where(live, case["alpha"] * state[b] + (1 - case["alpha"]) * s, state[b])
    return [out, state, None, None, None, None]

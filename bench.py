#!/usr/bin/env python3
"""Decode-step throughput of the InertiaKV eviction path on GB300.

Default workload: Llama-3.1-8B-shaped single-stream decode (32 layers, 32 query
heads, 8 KV heads, head_dim 128, bf16 K/V/q, fp32 utilities), prefilled
context 32768, budget 10% (3277 tokens), full-refresh EMA with alpha = 0.9.
Synthetic inputs from the seeded generator (heavy tokens, sinks, drifting
queries).  A step = one ikv_step call: append, attention of all layers,
Eq. 1 score + layer-sequential EMA (refresh steps), budgeted selection, stable
compaction.  Warm-up steps start at decode step 1 (which evicts ~90% of the
prefill); timed steps are the steady state that follows.

One JSON line on stdout (rank 0).  N > 1 (torchrun): every rank runs its own
replica on its own GPU (independent sequences, weak scaling); value = tokens
of all ranks / max time.
  --impl reference : times the CPU oracle on the host cores instead.
"""
from __future__ import annotations

import argparse
import ctypes
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

os.environ.setdefault("OPENBLAS_NUM_THREADS", "1")
os.environ.setdefault("MKL_NUM_THREADS", "1")

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "decode tokens/s at 10% KV budget (full/Lazy4/Score-Free); % of HBM peak"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--config", type=int, default=1)
    ap.add_argument("--layers", type=int, default=0,
                    help="profiling aid: keep the workload's shape but only this many layers (0 = all)")
    ap.add_argument("--no-modes", action="store_true", help="skip the Lazy4 / Score-Free lines")
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU-oracle baseline")
    ap.add_argument("--compact", default="short", choices=["short", "stable", "holefill"],
                    help="short: order-preserving, moves the shorter side (default); stable: always shifts "
                         "the suffix left; holefill: moves survivors into holes (order not kept)")
    ap.add_argument("--max-holes", type=int, default=128,
                    help="deferred compaction: evicted slots stay marked dead until a sequence holds more "
                         "than this many (0 = compact on every eviction; -1 = about 2 sqrt(B), the "
                         "bandwidth model's optimum, which measured no better here)")
    ap.add_argument("--mode-kernels", action="store_true",
                    help="also run every mode eagerly and report its per-kernel times")
    ap.add_argument("--cpu-steps", type=int, default=0, help="oracle steps in the CPU sample (0 = auto)")
    ap.add_argument("--no-trace", action="store_true", help="skip the rank-trace diagnostics")
    ap.add_argument("--no-configs", action="store_true",
                    help="skip the other workloads (per-configuration block and the Qwen-shaped sweep)")
    return ap.parse_args()


def max_over_ranks(ms: float, dist, device=None) -> float:
    """Slowest rank's time: the job's time for weak-scaled replicas (all ranks start
    after the same barrier)."""
    if dist is None:
        return ms
    import torch

    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(tokens_per_rank: int, world: int, ms_max: float) -> float:
    """Whole-job tokens/s: every rank decodes its own sequences."""
    return tokens_per_rank * world / (ms_max / 1e3)


def rank_seed(base_seed: int, rank: int) -> int:
    """Each rank decodes different sequences."""
    return base_seed + 1000 * rank


# revision of each attention kernel; a committed ncu summary counts only for its own revision
ATTEND_KERNEL_REV = {"attend_tc_kernel": "attend_tc_v15", "attend_bf16_kernel": "attend_bf16_v1", "attend_f32_kernel": "attend_f32_v1"}


def schedule_name(w) -> str:
    """The refresh schedule of a workload: full, lazy<r> (Eq. 6) or score_free."""
    if w.score_free:
        return "score_free"
    return "full" if w.refresh_period == 1 else f"lazy{w.refresh_period}"


def profiled_traffic(kernel: str, workload: str):
    """DRAM bytes per launch of the attention kernel from the committed ncu summary,
    or None when that summary was taken on another kernel revision or workload."""
    import re

    path = os.path.join(ROOT, "profiles", f"{kernel}__{workload}.md")
    if not os.path.exists(path):
        return None
    txt = open(path).read()
    rev = re.search(r"^kernel_rev:\s*(\S+)", txt, re.M)
    tb = re.search(r"^traffic_bytes_per_launch:\s*(\d+)", txt, re.M)
    if not rev or not tb or rev.group(1) != ATTEND_KERNEL_REV.get(kernel):
        return None
    return int(tb.group(1))


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


# ---------------------------------------------------------------------------
# CPU oracle sample (reference arm and cpu_baseline)
# ---------------------------------------------------------------------------
class OracleSample:
    """The CPU oracle stepping one sequence of the workload at its steady-state size.

    Sample: a cache of B tokens (the workload's decode budget) drawn from the
    seeded generator, then oracle decode steps from t = 2 on (append, attention
    of every layer, Eq. 1 score + layer-sequential EMA on refresh steps,
    eviction back to B).  Built once; each step() is timed on its own."""

    def __init__(self, w, max_steps: int):
        import numpy as np

        import gen
        import oracle as O

        self.O, self.w = O, w
        u = w.u_table()
        B = w.budgets()[0]
        K, V = [], []
        for l in range(w.layers):
            k, v = w.kv_block(0, l, 0, B, u)
            K.append([k[g].astype(np.float64) for g in range(w.kv_heads)])
            V.append([v[g].astype(np.float64) for g in range(w.kv_heads)])
        self.st = O.prefill_state(K, V, B)
        self.st.m[0] = np.linspace(1e-4, 2e-4, B)
        self.p = O.Params(alpha=w.alpha, refresh_period=w.refresh_period, score_free=w.score_free)
        self.t = 2
        qs = w.queries(2, 2 + max_steps, u)
        self.q64 = gen.bf16_to_f32(qs).astype(np.float64) if w.dtype == gen.BF16 else qs.astype(np.float64)
        self.u = u
        self.B = B

    def step(self) -> float:
        i = self.t - 2
        kn, vn = self.w.new_tokens(self.t, self.u)
        t0 = time.perf_counter()
        self.O.decode_step(self.st, self.t, self.q64[i][:, 0], kn[:, 0], vn[:, 0], self.p)
        dt = time.perf_counter() - t0
        self.t += 1
        return dt

    def describe(self, n: int) -> str:
        w = self.w
        return (f"{n} oracle decode steps of one sequence with a {self.B}-token cache (the decode budget), "
                f"{w.layers} layers x {w.q_heads} q heads / {w.kv_heads} kv heads x d {w.head_dim}, "
                f"fp64 numpy, 1 BLAS thread; tokens/s = steps / summed step time")


def _oracle_worker(w, n_warm: int, n_steps: int, barrier, queue):
    """One host core's share of the all-cores oracle run (a spawned process): one
    sequence's sample, its warm-up steps, then n_steps timed after every worker is ready."""
    s = OracleSample(w, n_warm + n_steps)
    for _ in range(n_warm):
        s.step()
    barrier.wait()
    t0 = time.monotonic()
    for _ in range(n_steps):
        s.step()
    queue.put((t0, time.monotonic()))


def host_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


def oracle_all_cores(w, n_warm: int, n_steps: int, cores: int = 0) -> dict:
    """The oracle on every host core: one process per core (spawned, BLAS on 1 thread
    each), each decoding its own sequence of the workload (a different seed) for n_steps
    steps after n_warm untimed ones; tokens/s = all decoded tokens / the wall time from the
    first worker's start to the last one's end."""
    import multiprocessing as mp

    n = cores or host_cores()
    ctx = mp.get_context("spawn")
    barrier = ctx.Barrier(n)
    queue = ctx.Queue()
    procs = [ctx.Process(target=_oracle_worker, args=(w.with_(seed=w.seed + 7919 * (i + 1)), n_warm, n_steps,
                                                      barrier, queue)) for i in range(n)]
    for p in procs:
        p.start()
    spans = [queue.get(timeout=1800) for _ in range(n)]
    for p in procs:
        p.join()
    wall = max(b for _, b in spans) - min(a for a, _ in spans)
    return {"value": n * n_steps / wall, "unit": "tokens/s", "cores": n, "kind": "oracle",
            "sample": f"{n} processes, one per host core, each {n_steps} oracle decode steps (after {n_warm} "
                      f"untimed) of its own sequence with a {w.budgets()[0]}-token cache, {w.layers} layers x "
                      f"{w.q_heads} q heads / {w.kv_heads} kv heads x d {w.head_dim}, fp64 numpy, 1 BLAS thread "
                      f"each; tokens/s = all steps / wall time", "wall_s": wall}


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import gen

    w = gen.config(args.config)
    if args.layers:
        w = w.with_(layers=args.layers, name=f"{w.name}-{args.layers}layers")
    # every host core runs the oracle on a sequence of its own (the workload's shape)
    cb = oracle_all_cores(w, args.warmup, args.steps)
    value = cb["value"]
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "tokens/s", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * cb["wall_s"] / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": w.name, "prefill": w.prefill[0], "budget": w.budgets()[0],
                                            "alpha": w.alpha, "refresh_period": w.refresh_period},
            "cpu_baseline": cb,
            "e2e": {"value": value, "unit": "tokens/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------------------
# GPU arm
# ---------------------------------------------------------------------------
class ClockSampler:
    def __init__(self, index: int):
        self.f = tempfile.NamedTemporaryFile(mode="w+", suffix=".csv", delete=False)
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.p = subprocess.Popen(["nvidia-smi", f"--id={index}", f"--query-gpu={q}", "--format=csv,noheader,nounits",
                                       "-lms", "100"], stdout=self.f, stderr=subprocess.DEVNULL)
        except OSError:
            self.p = None

    def stop(self):
        if self.p is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.25)
        self.p.terminate()
        self.p.wait()
        self.f.flush()
        self.f.seek(0)
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.f.read().splitlines():
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        os.unlink(self.f.name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "samples": len(sm), "reasons": sorted(reasons)}


def device_inputs(w, u, u_dev, T: int, dev):
    """Every decode step's inputs, resident on the device: q [T][layers][batch][q_heads][d]
    from the host generator, k_new / v_new [T][layers][batch][kv_heads][d] from the device
    generator (bit-identical to the host's)."""
    import numpy as np
    import torch

    import gen

    qs_h = w.queries(1, T + 1, u)
    tdt = torch.bfloat16 if w.dtype == gen.BF16 else torch.float32
    if w.dtype == gen.BF16:
        qs_t = torch.from_numpy(qs_h.view(np.int16)).view(torch.bfloat16)
    else:
        qs_t = torch.from_numpy(qs_h)
    qs_dev = qs_t.to(dev)
    kn_dev = torch.empty((T, w.layers, w.batch, w.kv_heads, w.head_dim), dtype=tdt, device=dev)
    vn_dev = torch.empty_like(kn_dev)
    sp = w.spec()
    L0 = torch.tensor(w.prefill, dtype=torch.int32, device=dev)
    rc = gen.cuda_lib().ikvgen_fill_tokens_cuda(ctypes.byref(sp), u_dev.data_ptr(), L0.data_ptr(), 1, T + 1, w.dtype,
                                                kn_dev.data_ptr(), vn_dev.data_ptr(),
                                                torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    torch.cuda.synchronize()
    return qs_dev, kn_dev, vn_dev


def setup(w, device, compact_mode, steps: int = 0):
    import numpy as np
    import torch

    import gen
    from paper_2609_03515_gb300 import DecodeCache, ikv

    c = DecodeCache(w.batch, w.layers, w.q_heads, w.kv_heads, w.head_dim, w.cap,
                    dtype=ikv.IKV_BF16 if w.dtype == gen.BF16 else ikv.IKV_F32, page_size=w.page_size,
                    device=device, page_perm_seed=1, value_norms=True,
                    pos_cap=max(w.prefill) + steps + 2)  # position state for per-layer eviction
    return c


def reset(c, w, u_dev):
    import torch

    import gen

    c.set_prefill(w.prefill, w.budgets())
    sp = w.spec()
    L0 = torch.tensor(w.prefill, dtype=torch.int32, device=c.k.device)
    rc = gen.cuda_lib().ikvgen_fill_paged_cuda(ctypes.byref(sp), u_dev.data_ptr(), c.k.data_ptr(), c.v.data_ptr(),
                                               c.block_table.data_ptr(), L0.data_ptr(), c.num_pages, c.page_size,
                                               c.max_pages, max(w.prefill), w.dtype,
                                               torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    if c.vnorm is not None:  # value-row norms of the prefill, for the VNorm scorer
        from paper_2609_03515_gb300 import ikv

        ikv.ikv_value_norms(c.shape(), c.cache(max(w.prefill)))
    torch.cuda.synchronize()


def run_mode(args, w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, want_detail: bool, dist, mh: int = 0,
             scorer: int = 0):
    """Warm-up then K timed steps of one schedule, launched eagerly; returns a dict of
    measurements (with per-kernel CUDA-event times when want_detail)."""
    import torch

    from paper_2609_03515_gb300 import ikv, step_lengths

    reset(c, w, u_dev)
    p = c.params(w.alpha, w.refresh_period, w.score_free, compact_mode, max_holes=mh, scorer=scorer)
    budgets = w.budgets()
    lens, live = list(w.prefill), list(w.prefill)
    out = torch.empty((w.layers, w.batch, w.q_heads, w.head_dim), dtype=c.torch_dtype, device=c.k.device)
    stream = torch.cuda.current_stream()

    def step(t, timing=None):
        nonlocal lens, live
        if timing is not None:
            p.timing = ctypes.pointer(timing)
        else:
            p.timing = None
        ikv.ikv_step(c.shape(), p, c.cache(max(lens)), c.ema, t, qs_dev[t - 1], kn_dev[t - 1], vn_dev[t - 1], out, ws,
                     ws.numel(), stream)
        lens, live = step_lengths(lens, live, budgets, mh)

    W, K = args.warmup, args.steps
    for t in range(1, W + 1):
        step(t)
    torch.cuda.synchronize()
    evs = []
    timings = []
    if want_detail:
        for _ in range(K):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(7)]
            for x in e:
                x.record(stream)  # torch creates the CUDA event on first record; the library re-records it
            evs.append(e)
            tm = ikv.ikv_timing(*[x.cuda_event for x in e])
            timings.append(tm)
    start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    launches0 = ikv.ikv_launch_count()
    start.record(stream)
    for i in range(K):
        step(W + 1 + i, timings[i] if want_detail else None)
    stop.record(stream)
    torch.cuda.synchronize()
    launches = ikv.ikv_launch_count() - launches0
    ms = max_over_ranks(start.elapsed_time(stop), dist, c.k.device)
    res = {"ms": ms, "launches": launches, "lens": lens}
    if want_detail:
        names = ["append", "attend", "combine", "score_ema", "select", "compact"]
        per = {n: [] for n in names}
        for e in evs:
            for j, n in enumerate(names):
                per[n].append(e[j].elapsed_time(e[j + 1]))
        res["kernel_ms"] = {n: sum(v) / len(v) for n, v in per.items()}
    return res


def split_step(c, p, cache, t, q, kn, vn, out, ws, stream, foreign=None):
    """One decode step as a model issues it: ikv_step_begin, then per layer (after the
    caller's own work for that layer, `foreign(l)`, if given) ikv_step_layer, then
    ikv_step_end."""
    from paper_2609_03515_gb300 import ikv

    m = c.utility(p.evict_mode)
    ikv.ikv_step_begin(c.shape(), p, cache, m, t, ws, ws.numel(), stream)
    for l in range(c.layers):
        if foreign is None:
            ikv.ikv_step_layer(c.shape(), p, cache, m, t, l, q[l], kn[l], vn[l], out[l], ws, ws.numel(), stream)
        else:
            ql, kl, vl = foreign(l)
            ikv.ikv_step_layer(c.shape(), p, cache, m, t, l, ql, kl, vl, out[l], ws, ws.numel(), stream)
    ikv.ikv_step_end(c.shape(), p, cache, m, t, ws, ws.numel(), stream)


def run_mode_graph(args, w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, dist, sample_clocks: bool,
                   mh: int = 0, scorer: int = 0, per_layer: str = "", evict: int = 0, agg: int = 0,
                   after_step=None):
    """The same schedule with each steady-state step replayed from a captured CUDA graph.

    After the eager warm-up (decode step 1 evicts ~90% of the prefill, later steps hold
    the budget), one graph per timed step t is captured around ikv_step(t) with that
    step's resident inputs (q, k_new, v_new of step t), so replaying it does exactly what
    the eager call would, with no staging copies; the timed region replays them in order.
    per_layer "split": the step as ikv_step_begin / one ikv_step_layer per layer /
    ikv_step_end; "foreign": the same, with the layer's q, k_new and v_new first copied
    by PyTorch kernels into per-layer buffers (standing in for the projection that a
    model runs before each layer's attention).
    after_step(t, out): called after each warm-up step and each replayed step, once the
    device is idle (parity tests of this exact path); None in a timed run."""
    import torch

    from paper_2609_03515_gb300 import ikv, step_lengths

    reset(c, w, u_dev)
    p = c.params(w.alpha, w.refresh_period, w.score_free, compact_mode, max_holes=mh, scorer=scorer,
                 evict_mode=evict, agg_mode=agg)
    m_state = c.utility(evict)
    budgets = w.budgets()
    assert all(L0 >= B for L0, B in zip(w.prefill, budgets)), "graph replay assumes every sequence at its budget"
    lens, live = list(w.prefill), list(w.prefill)
    dev = c.k.device
    out = torch.empty((w.layers, w.batch, w.q_heads, w.head_dim), dtype=c.torch_dtype, device=dev)
    W, K = args.warmup, args.steps
    ql = torch.empty(qs_dev.shape[2:], dtype=qs_dev.dtype, device=dev)
    kl = torch.empty(kn_dev.shape[2:], dtype=kn_dev.dtype, device=dev)
    vl = torch.empty_like(kl)

    def one(cache, t):
        st = torch.cuda.current_stream()
        if not per_layer:
            ikv.ikv_step(c.shape(), p, cache, m_state, t, qs_dev[t - 1], kn_dev[t - 1], vn_dev[t - 1], out, ws,
                         ws.numel(), st)
            return

        def foreign(l):
            ql.copy_(qs_dev[t - 1, l])
            kl.copy_(kn_dev[t - 1, l])
            vl.copy_(vn_dev[t - 1, l])
            return ql, kl, vl

        split_step(c, p, cache, t, qs_dev[t - 1], kn_dev[t - 1], vn_dev[t - 1], out, ws, st,
                   foreign if per_layer == "foreign" else None)

    for t in range(1, W + 1):
        one(c.cache(max(lens)), t)
        lens, live = step_lengths(lens, live, budgets, mh)
        if after_step is not None:
            torch.cuda.synchronize()
            after_step(t, out)
    torch.cuda.synchronize()
    # the graphs' max_len bounds every later step: the budget plus the dead slots
    # deferred compaction may hold; the warm-up left the workspace's counters zero
    steady = c.cache(min(c.cap - 1, max(max(lens), max(budgets) + mh)))
    p.ws_zeroed = 1
    graphs = []
    n0 = ikv.ikv_launch_count()
    for i in range(K):
        t = W + 1 + i
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            one(steady, t)
        graphs.append((g, ikv.ikv_launch_count() - n0))
        n0 = ikv.ikv_launch_count()
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    clocks = ClockSampler(torch.cuda.current_device()) if sample_clocks else None
    launches = 0
    start.record(stream)
    for i, (g, nl) in enumerate(graphs):
        g.replay()
        launches += nl
        if after_step is not None:
            torch.cuda.synchronize()
            after_step(W + 1 + i, out)
    stop.record(stream)
    torch.cuda.synchronize()
    ms = max_over_ranks(start.elapsed_time(stop), dist, dev)
    res = {"ms": ms, "launches": launches}
    if sample_clocks:
        res["clocks"] = clocks.stop()
    return res


def run_trajectory(w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, mh: int, dist=None):
    """The configuration's whole decode run: decode steps 1 .. w.steps from the prefill,
    step 1 (which scores the whole prefill and evicts most of it) and every deferred
    compaction included.  The steps are launched one by one with programmatic dependent
    launch between the library's kernels (the host stays several steps ahead of the GPU);
    one untimed pass first.  Per-step CUDA graphs measure the same time in a fresh process,
    but after about a thousand graph instantiations in a process the driver runs newly
    captured graphs ~35 us slower each, and a trajectory alone instantiates hundreds.
    Returns the time of all steps."""
    import torch

    from paper_2609_03515_gb300 import ikv, step_lengths

    budgets = w.budgets()
    dev = c.k.device
    out = torch.empty((w.layers, w.batch, w.q_heads, w.head_dim), dtype=c.torch_dtype, device=dev)
    lens, live = list(w.prefill), list(w.prefill)
    bounds = []
    for t in range(1, w.steps + 1):
        bounds.append(max(lens))
        lens, live = step_lengths(lens, live, budgets, mh)
    steady = c.cache(min(c.cap - 1, max(bounds[1:] + [max(budgets) + mh])))
    first = c.cache(bounds[0])
    stream = torch.cuda.current_stream()

    def one_pass(timed: bool):
        reset(c, w, u_dev)
        p = c.params(w.alpha, w.refresh_period, w.score_free, compact_mode, max_holes=mh)
        p.ws_zeroed = 1  # the workspace is zero-filled at creation and every step leaves its counters zero
        start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        if dist and timed:
            dist.barrier()
        torch.cuda.synchronize()
        start.record(stream)
        for t in range(1, w.steps + 1):
            ikv.ikv_step(c.shape(), p, first if t == 1 else steady, c.ema, t, qs_dev[t - 1], kn_dev[t - 1],
                         vn_dev[t - 1], out, ws, ws.numel(), stream)
        stop.record(stream)
        torch.cuda.synchronize()
        return start.elapsed_time(stop)

    one_pass(False)
    ms = one_pass(True)
    assert ikv.ikv_device_status() == 0
    return max_over_ranks(ms, dist, dev)


def sig(x, n: int = 4):
    """x rounded to n significant digits (keeps the JSON line short)."""
    if x is None or x == 0:
        return x
    from math import floor, log10

    return round(x, -int(floor(log10(abs(x)))) + n - 1)


def attention_bytes(w, esz: int) -> int:
    """Algorithmic bytes of one steady-state attention launch over every layer: the K and
    V rows of each sequence's B + 1 cached tokens, plus q."""
    L = [min(x + 1, B + 1) for x, B in zip(w.prefill, w.budgets())]
    return sum(L) * w.layers * w.kv_heads * w.head_dim * 2 * esz + w.layers * w.batch * w.q_heads * w.head_dim * esz


def step_bytes(w, esz: int) -> int:
    """Algorithmic bytes of one steady-state step (refresh): the attention's K/V and q reads,
    the output write, the utilities read and written once, and the new token's K/V rows."""
    L = [min(x + 1, B + 1) for x, B in zip(w.prefill, w.budgets())]
    out = w.layers * w.batch * w.q_heads * w.head_dim * esz
    util = 8 * sum(L)
    append = w.layers * w.batch * w.kv_heads * w.head_dim * 2 * esz
    return attention_bytes(w, esz) + out + util + append


def run_other_config(args, cfg: int, dev, dist, rank: int, compact_mode, mh_arg: int, peak: float, sweep: bool):
    """One more workload, for the per-configuration block: its headline schedule, the same
    inputs under full refresh, the attention and attention + score + EMA roofline from
    eager per-kernel events, and its whole trajectory; with sweep (the Qwen-shaped
    workload) the budget x refresh-period x alpha grid as well.  Fewer timed steps than the
    headline (at most 20 after 3 warm-up steps); everything is freed afterwards."""
    import argparse

    import torch

    import gen
    from paper_2609_03515_gb300 import auto_max_holes

    w = gen.config(cfg)
    w = w.with_(seed=rank_seed(w.seed, rank))
    sub = argparse.Namespace(warmup=3, steps=min(args.steps, 20))
    total = max(w.steps, sub.warmup + sub.steps)
    w = w.with_(steps=total)
    mh = mh_arg if mh_arg >= 0 else auto_max_holes(w.budgets())
    u = w.u_table()
    u_dev = torch.from_numpy(u).to(dev)
    c = setup(w, dev, compact_mode, total)
    ws = c.step_workspace()
    qs_dev, kn_dev, vn_dev = device_inputs(w, u, u_dev, total, dev)
    esz = 2 if w.dtype == gen.BF16 else 4
    K = sub.steps
    eager = run_mode(sub, w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, True, dist, mh)
    head = run_mode_graph(sub, w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, dist, False, mh)
    full_w = w.with_(refresh_period=1, score_free=False)
    sched = schedule_name(w)
    full = head if sched == "full" else run_mode_graph(sub, full_w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode,
                                                        dist, False, mh)
    km = eager["kernel_ms"]
    # the attention + score + EMA time of a refresh step: this schedule's eager score time
    # is an average over its steps, so the full-refresh run's events give it
    kf = km if sched == "full" else run_mode(sub, full_w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, True,
                                             dist, mh)["kernel_ms"]
    ab = attention_bytes(w, esz)
    traj_w = w.with_(steps=gen.config(cfg).steps)
    traj_ms = run_trajectory(traj_w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, mh, dist)
    world = dist.get_world_size() if dist else 1
    res = {"workload": w.name, "schedule": sched,
           "value": sig(job_throughput(w.batch * K, world, head["ms"])),
           "us_per_step": sig(1e3 * head["ms"] / K),
           "attend_frac": sig(ab / (km["attend"] / 1e3) / 1e9 / peak),
           "attend_score_ema_frac": sig((ab + 8 * sum(min(x + 1, B + 1) for x, B in zip(w.prefill, w.budgets())))
                                        / ((kf["attend"] + kf["score_ema"]) / 1e3) / 1e9 / peak),
           "full_value": sig(job_throughput(w.batch * K, world, full["ms"])),
           "speedup_vs_full": sig(full["ms"] / head["ms"]),
           "trajectory": {"steps": traj_w.steps, "value": sig(job_throughput(w.batch * traj_w.steps, world, traj_ms)),
                          "ms": sig(traj_ms)}}
    if sweep:
        grid = {}
        base = None
        for bf in (0.5, 0.25, 0.1):
            for r in (1, 2, 4, 8):
                ww = w.with_(budget_frac=bf, refresh_period=r, score_free=False)
                m = run_mode_graph(sub, ww, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, dist, False,
                                   mh_arg if mh_arg >= 0 else auto_max_holes(ww.budgets()))
                grid[f"b{int(bf * 100)}_r{r}"] = job_throughput(w.batch * K, world, m["ms"])
        alphas = {}
        for al in (0.5, 0.9, 0.99):
            ww = w.with_(budget_frac=0.1, refresh_period=1, score_free=False, alpha=al)
            m = run_mode_graph(sub, ww, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, dist, False, mh)
            alphas[f"a{al}"] = sig(job_throughput(w.batch * K, world, m["ms"]))
        res["sweep"] = {"tok_s": {k: sig(v) for k, v in grid.items()},
                        "lazy_speedup": {k: sig(v / grid[k.split("_")[0] + "_r1"]) for k, v in grid.items()
                                         if not k.endswith("_r1")},
                        "alpha_b10_r1": alphas}
    del c, ws, qs_dev, kn_dev, vn_dev, u_dev
    torch.cuda.empty_cache()
    return res


def trace_ratios(counts):
    """The Appendix's rank-trace measures from one step's overlap counts per utility row,
    {|R & R_prev|, |E & E_prev|, |R & E|, |R|, |E|} (ikv_trace.counts): EMA churn, and on
    steps with a raw top-k its churn, the raw/EMA Jaccard and the raw-top evicted fraction."""
    out = []
    for rr, re_, rx, nr, ne in counts:
        row = {"ema_churn": 1.0 - re_ / ne if ne > 0 else None}
        if nr > 0:
            row["raw_churn"] = 1.0 - rr / nr
            row["jaccard"] = rx / (nr + ne - rx)
            row["raw_top_evicted"] = 1.0 - rx / nr
        out.append(row)
    return out


def run_trace(args, w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, mh: int = 0):
    """Rank-trace diagnostics (raw / EMA top-k churn, raw/EMA Jaccard, raw-top evicted)
    over the timed steps of one schedule, launched eagerly with ikv_params.trace set;
    means over the steps that have them and over the utility rows.  Not timed."""
    import torch

    from paper_2609_03515_gb300 import RankTrace, ikv, step_lengths

    reset(c, w, u_dev)
    tr = RankTrace(c)
    p = c.params(w.alpha, w.refresh_period, w.score_free, compact_mode, max_holes=mh, trace=tr)
    budgets = w.budgets()
    lens, live = list(w.prefill), list(w.prefill)
    out = torch.empty((w.layers, w.batch, w.q_heads, w.head_dim), dtype=c.torch_dtype, device=c.k.device)
    acc = {"raw_churn": [], "ema_churn": [], "jaccard": [], "raw_top_evicted": []}
    W, K = args.warmup, min(args.steps, 50)
    for t in range(1, W + K + 1):
        ikv.ikv_step(c.shape(), p, c.cache(max(lens)), c.ema, t, qs_dev[t - 1], kn_dev[t - 1], vn_dev[t - 1], out, ws,
                     ws.numel(), torch.cuda.current_stream())
        lens, live = step_lengths(lens, live, budgets, mh)
        if t > W:  # churn compares with the previous traced step, so the first timed step has one
            for row in trace_ratios(tr.counts.cpu().tolist()):
                for k, v in row.items():
                    if v is not None and k in acc:
                        acc[k].append(v)
    torch.cuda.synchronize()
    return {k: (sum(v) / len(v) if v else None) for k, v in acc.items()}


def run_e2e(args, w, c, u_dev, ws, compact_mode, qs_h, kn_h, vn_h, dist, mh: int = 0, scorer: int = 0):
    """Same steps through the C ABI, inputs from pinned host memory and the output read back every step.

    Two device buffer sets: the upload of step t+1's inputs and the read-back of step t-1's
    output run while step t computes.  The warm-up launches the steps eagerly with one copy
    stream per direction.  Each timed step then replays a CUDA graph captured for it that
    holds ikv_step(t) and, on a forked branch joined at its end, those two copies (from and
    to fixed pinned host buffers); the first step's upload and the last step's read-back
    are issued around the graphs.  Every step's copies lie inside the timed region."""
    import torch

    from paper_2609_03515_gb300 import ikv, step_lengths

    reset(c, w, u_dev)
    p = c.params(w.alpha, w.refresh_period, w.score_free, compact_mode, max_holes=mh, scorer=scorer)
    budgets = w.budgets()
    lens, live = list(w.prefill), list(w.prefill)
    dev = c.k.device
    q_d = [torch.empty(qs_h.shape[1:], dtype=qs_h.dtype, device=dev) for _ in range(2)]
    kn_d = [torch.empty(kn_h.shape[1:], dtype=kn_h.dtype, device=dev) for _ in range(2)]
    vn_d = [torch.empty(kn_h.shape[1:], dtype=kn_h.dtype, device=dev) for _ in range(2)]
    oshape = (w.layers, w.batch, w.q_heads, w.head_dim)
    out_d = [torch.empty(oshape, dtype=c.torch_dtype, device=dev) for _ in range(2)]
    out_h = [torch.empty(oshape, dtype=c.torch_dtype, pin_memory=True) for _ in range(2)]
    comp = torch.cuda.current_stream()
    up = torch.cuda.Stream(device=dev)    # host -> device uploads
    down = torch.cuda.Stream(device=dev)  # device -> host read-backs (a separate copy engine)
    in_ready = [torch.cuda.Event() for _ in range(2)]
    done = [torch.cuda.Event() for _ in range(2)]
    read = [torch.cuda.Event() for _ in range(2)]

    def upload(t):
        i = t % 2
        with torch.cuda.stream(up):
            q_d[i].copy_(qs_h[t - 1], non_blocking=True)
            kn_d[i].copy_(kn_h[t - 1], non_blocking=True)
            vn_d[i].copy_(vn_h[t - 1], non_blocking=True)
            in_ready[i].record(up)

    def run(t0, n):
        """Eager steps t0 .. t0+n-1; the upload of t0 is issued here, the last read-back is waited for."""
        nonlocal lens, live
        up.wait_stream(comp)
        down.wait_stream(comp)
        upload(t0)
        for t in range(t0, t0 + n):
            i = t % 2
            if t + 1 < t0 + n:
                if t + 1 >= t0 + 2:
                    up.wait_event(done[(t + 1) % 2])   # step t-1 has read the buffers step t+1 reuses
                upload(t + 1)
            comp.wait_event(in_ready[i])
            if t >= t0 + 2:
                comp.wait_event(read[i])             # step t-2's output has been read back
            ikv.ikv_step(c.shape(), p, c.cache(max(lens)), c.ema, t, q_d[i], kn_d[i], vn_d[i], out_d[i], ws,
                         ws.numel(), comp)
            done[i].record(comp)
            with torch.cuda.stream(down):
                down.wait_event(done[i])
                out_h[i].copy_(out_d[i], non_blocking=True)
                read[i].record(down)
            lens, live = step_lengths(lens, live, budgets, mh)
        comp.wait_stream(up)
        comp.wait_stream(down)

    W, K = args.warmup, args.steps
    run(1, W)
    torch.cuda.synchronize()
    steady = c.cache(min(c.cap - 1, max(max(lens), max(budgets) + mh)))
    p.ws_zeroed = 1  # the warm-up left the workspace's counters zero
    T0 = W + 1
    side = torch.cuda.Stream(device=dev)
    step_graphs = []
    for t in range(T0, T0 + K):
        i = t % 2
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            cs = torch.cuda.current_stream()
            side.wait_stream(cs)
            with torch.cuda.stream(side):
                if t + 1 < T0 + K:  # step t+1's inputs into the other buffer set
                    q_d[1 - i].copy_(qs_h[t], non_blocking=True)
                    kn_d[1 - i].copy_(kn_h[t], non_blocking=True)
                    vn_d[1 - i].copy_(vn_h[t], non_blocking=True)
                if t > T0:  # step t-1's output
                    out_h[1 - i].copy_(out_d[1 - i], non_blocking=True)
            ikv.ikv_step(c.shape(), p, steady, c.ema, t, q_d[i], kn_d[i], vn_d[i], out_d[i], ws, ws.numel(), cs)
            cs.wait_stream(side)
        step_graphs.append(g)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record(comp)
    i0, il = T0 % 2, (T0 + K - 1) % 2
    q_d[i0].copy_(qs_h[T0 - 1], non_blocking=True)
    kn_d[i0].copy_(kn_h[T0 - 1], non_blocking=True)
    vn_d[i0].copy_(vn_h[T0 - 1], non_blocking=True)
    for g in step_graphs:
        g.replay()
    out_h[il].copy_(out_d[il], non_blocking=True)
    stop.record(comp)
    torch.cuda.synchronize()
    ms = max_over_ranks(start.elapsed_time(stop), dist, dev)
    h2d = (q_d[0].numel() + kn_d[0].numel() + vn_d[0].numel()) * q_d[0].element_size()
    d2h = out_d[0].numel() * out_d[0].element_size()
    return ms, h2d, d2h


def run_ours(args):
    import numpy as np
    import torch

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    dist = None
    if world > 1:
        import torch.distributed as tdist

        torch.cuda.set_device(local)
        tdist.init_process_group("nccl", device_id=torch.device("cuda", local))
        dist = tdist
    else:
        torch.cuda.set_device(0)

    import gen
    import __graft_entry__

    if rank == 0 or world == 1:
        __graft_entry__.build()
    if dist:
        dist.barrier()
    from paper_2609_03515_gb300 import ikv, step_lengths

    w = gen.config(args.config)
    if args.layers:
        w = w.with_(layers=args.layers, name=f"{w.name}-{args.layers}layers")
    # each rank decodes its own independent sequences (distinct seed per rank)
    w = w.with_(seed=rank_seed(w.seed, rank))
    total_steps = args.warmup + args.steps
    if total_steps > w.steps:
        w = w.with_(steps=total_steps)
    compact_mode = {"short": ikv.IKV_COMPACT_STABLE_SHORT, "stable": ikv.IKV_COMPACT_STABLE,
                    "holefill": ikv.IKV_COMPACT_HOLEFILL}[args.compact]

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        # the oracle on one host thread, then on every host core (one sequence per core)
        n = args.cpu_steps or 8
        smp = OracleSample(w, n + 1)
        smp.step()  # first step outside the sample (allocator warm-up)
        sec = sum(smp.step() for _ in range(n))
        single = {"value": n / sec, "unit": "tokens/s", "cores": 1, "sample": smp.describe(n)}
        del smp
        cpu = oracle_all_cores(w, 1, n)
        cpu["single_thread"] = single

    dev = torch.device("cuda", torch.cuda.current_device())
    u = w.u_table()
    u_dev = torch.from_numpy(u).to(dev)
    # enough resident inputs for the timed steps and for the whole trajectory
    total_steps = max(total_steps, gen.config(args.config).steps)
    w = w.with_(steps=total_steps)
    c = setup(w, dev, compact_mode, total_steps)
    ws = c.step_workspace()
    qs_dev, kn_dev, vn_dev = device_inputs(w, u, u_dev, total_steps, dev)
    T_io = args.warmup + args.steps
    qs_t = qs_dev[:T_io].cpu()

    from paper_2609_03515_gb300 import auto_max_holes

    mh = args.max_holes if args.max_holes >= 0 else auto_max_holes(w.budgets())
    eager = run_mode(args, w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, True, dist, mh)
    full = run_mode_graph(args, w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, dist, True, mh)
    # end to end right after the headline, before the mode comparisons
    qs_pin = qs_t.pin_memory()
    kn_pin = kn_dev[:T_io].cpu().pin_memory()
    vn_pin = vn_dev[:T_io].cpu().pin_memory()
    # five complete end-to-end runs, median reported: host-link bandwidth on the shared
    # machine varies from run to run
    e2e_runs = [run_e2e(args, w, c, u_dev, ws, compact_mode, qs_pin, kn_pin, vn_pin, dist, mh) for _ in range(5)]
    e2e_all = sorted(r[0] for r in e2e_runs)
    e2e_ms, h2d, d2h = e2e_all[2], e2e_runs[0][1], e2e_runs[0][2]

    # the model-integration form: the same headline steps split per layer
    per_layer = {k: run_mode_graph(args, w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, dist, False, mh,
                                   per_layer=k) for k in ("split", "foreign")}
    # the whole decode run of the headline configuration, step 1 and every compaction included
    traj_w = w.with_(steps=gen.config(args.config).steps)
    traj_ms = run_trajectory(traj_w, c, u_dev, qs_dev, kn_dev, vn_dev, ws, compact_mode, mh, dist)
    L = [min(x + 1, B + 1) for x, B in zip(w.prefill, w.budgets())]  # length seen by the timed steps
    att_kernel = ("attend_tc_kernel" if ikv.ikv_attend_path(c.shape(), c.cache(max(L))) == ikv.IKV_PATH_TENSOR_CORE
                  else "attend_f32_kernel" if w.dtype == gen.F32 else "attend_bf16_kernel")

    head_sched = schedule_name(w)
    modes = {}
    mode_kernels = {}
    if not args.no_modes:
        full_w = w.with_(refresh_period=1, score_free=False)
        lazy_w = w.with_(refresh_period=4, score_free=False)
        sf_w = w.with_(refresh_period=1, score_free=True)
        att, vnm, ent = ikv.IKV_SCORE_ATTENTION, ikv.IKV_SCORE_VNORM, ikv.IKV_SCORE_ENTROPY
        stable, layer = ikv.IKV_COMPACT_STABLE, ikv.IKV_EVICT_LAYER
        ema, cum, single_step = ikv.IKV_AGG_EMA, ikv.IKV_AGG_CUMULATIVE, ikv.IKV_AGG_SINGLE_STEP
        variants = (("full", full_w, compact_mode, mh, att, 0, ema),
                    ("lazy4", lazy_w, compact_mode, mh, att, 0, ema),
                    ("score_free", sf_w, compact_mode, mh, att, 0, ema),
                    ("full_vnorm", full_w, compact_mode, mh, vnm, 0, ema),
                    ("full_entropy", full_w, compact_mode, mh, ent, 0, ema),
                    ("full_cumulative", full_w, compact_mode, mh, att, 0, cum),
                    ("full_single_step", full_w, compact_mode, mh, att, 0, single_step),
                    ("full_every_step", full_w, compact_mode, 0, att, 0, ema),
                    ("lazy4_every_step", lazy_w, compact_mode, 0, att, 0, ema),
                    ("score_free_every_step", sf_w, compact_mode, 0, att, 0, ema),
                    ("full_stable_left", full_w, stable, 0, att, 0, ema),
                    ("full_holefill", full_w, ikv.IKV_COMPACT_HOLEFILL, 0, att, 0, ema),
                    ("lazy4_holefill", lazy_w, ikv.IKV_COMPACT_HOLEFILL, 0, att, 0, ema),
                    ("score_free_holefill", sf_w, ikv.IKV_COMPACT_HOLEFILL, 0, att, 0, ema),
                    ("full_layer_evict", full_w, ikv.IKV_COMPACT_HOLEFILL, 0, att, layer, ema),
                    ("lazy4_layer_evict", lazy_w, ikv.IKV_COMPACT_HOLEFILL, 0, att, layer, ema),
                    ("full_layer_evict_stable", full_w, stable, 0, att, layer, ema))
        for name, ww, cm, vmh, sc, ev, ag in variants:
            if name == head_sched and cm == compact_mode and vmh == mh and sc == att and ev == 0 and ag == ema:
                modes[name] = full           # the headline run is this mode
                continue
            modes[name] = run_mode_graph(args, ww, c, u_dev, qs_dev, kn_dev, vn_dev, ws, cm, dist, False, vmh, sc,
                                         evict=ev, agg=ag)
        if args.mode_kernels:
            for name, ww, cm, vmh, sc, ev, ag in variants:
                if ev or ag != ema:
                    continue  # per-kernel events time the step-end EMA eviction path only
                mode_kernels[name] = run_mode(args, ww, c, u_dev, qs_dev, kn_dev, vn_dev, ws, cm, True, dist,
                                              vmh, sc)["kernel_ms"]
    trace = None
    if not args.no_trace:
        # the Appendix's rank-trace table on this workload: full refresh at three alphas
        trace = {f"alpha_{a}": run_trace(args, w.with_(alpha=a, refresh_period=1, score_free=False), c, u_dev, qs_dev,
                                         kn_dev, vn_dev, ws, compact_mode, mh) for a in (0.3, 0.8, 0.9)}
    K = args.steps
    value = job_throughput(w.batch * K, world, full["ms"])
    peak, peak_kind = load_peaks()
    # the other workloads: Lazy4 (ragged batch), Score-Free (64k), and the Qwen-shaped one
    # with its budget x refresh-period x alpha sweep; freed before the next one
    others = {}
    if args.config == 1 and not args.no_configs:
        del c, ws, qs_dev, kn_dev, vn_dev
        torch.cuda.empty_cache()
        for cfg in (2, 3, 4):
            others[str(cfg)] = run_other_config(args, cfg, dev, dist, rank, compact_mode, args.max_holes, peak,
                                                sweep=cfg == 4)
    if rank != 0:
        if dist:
            dist.destroy_process_group()
        return

    esz = 2 if w.dtype == gen.BF16 else 4
    # attention kernel roofline: algorithmic bytes of one launch at the steady-state length
    ab = attention_bytes(w, esz)
    kv_bytes = ab - w.layers * w.batch * w.q_heads * w.head_dim * esz
    att_ms = eager["kernel_ms"]["attend"]
    achieved = ab / (att_ms / 1e3) / 1e9
    traffic = profiled_traffic(att_kernel, w.name)
    # the unit the method's cost is stated in: attention + score + EMA (one launch each per
    # step; eager per-kernel events, so each includes a launch gap), and the whole graphed step
    ase_bytes = ab + 8 * sum(L)
    ase_ms = eager["kernel_ms"]["attend"] + eager["kernel_ms"]["score_ema"]
    st_bytes = step_bytes(w, esz)
    st_ms = full["ms"] / K
    nominal = 8000.0
    l2_note = ("inputs exceed L2 (K/V working set %.0f MB > 129 MB), no flush" % (kv_bytes / 1e6) if kv_bytes > 129e6
               else "K/V working set %.2f MB stays in L2 (launch-bound case), no flush" % (kv_bytes / 1e6))
    line = {
        "metric": METRIC,
        "value": value,
        "unit": "tokens/s",
        "n_gpus": world,
        "steps": K,
        "warmup": args.warmup,
        "ms_per_step": full["ms"] / K,
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "bf16" if w.dtype == gen.BF16 else "f32",
        "data": "synthetic",
        "config": {"workload": w.name, "batch_per_gpu": w.batch, "layers": w.layers, "q_heads": w.q_heads,
                   "kv_heads": w.kv_heads, "head_dim": w.head_dim, "prefill": w.prefill[0] if w.batch == 1 else w.prefill,
                   "budget": w.budgets(), "alpha": w.alpha, "refresh": head_sched, "compaction": args.compact, "max_holes": mh,
                   "timed_steps": f"decode steps {args.warmup + 1}..{args.warmup + K} (steady state; step 1 in warm-up)",
                   "launch": "one CUDA graph per timed step, captured on that step's resident inputs; "
                             "workspace counters kept zero across steps (ikv_params.ws_zeroed)",
                   "l2": l2_note,
                   "parallelism": f"replicas x{world}"},
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                     "traffic": traffic, "kernel": att_kernel, "peak_kind": peak_kind,
                     "bytes_per_launch": ab, "ms_per_launch": att_ms,
                     "attend_score_ema": {"bytes": ase_bytes, "ms": ase_ms,
                                          "frac": ase_bytes / (ase_ms / 1e3) / 1e9 / peak,
                                          "frac_of_nominal_8tbs": ase_bytes / (ase_ms / 1e3) / 1e9 / nominal,
                                          "note": "K/V + q reads and the utilities' read + write over the eager "
                                                  "events of the attention and score kernels (each with its launch gap)"},
                     "step": {"bytes": st_bytes, "ms": st_ms, "frac": st_bytes / (st_ms / 1e3) / 1e9 / peak,
                              "frac_of_nominal_8tbs": st_bytes / (st_ms / 1e3) / 1e9 / nominal,
                              "note": "the whole graphed step: attention, output, utilities, new rows"}},
        "kernel_ms_per_step": eager["kernel_ms"],
        "eager": {"value": job_throughput(w.batch * K, world, eager["ms"]), "ms_per_step": eager["ms"] / K,
                  "note": "same steps launched one by one (per-kernel events above come from this run)"},
        "cpu_baseline": cpu,
        "e2e": {"value": w.batch * K * world / (e2e_ms / 1e3), "unit": "tokens/s", "h2d_bytes_per_step": h2d,
                "d2h_bytes_per_step": d2h, "runs": [w.batch * K * world / (m / 1e3) for m in e2e_all],
                "note": "median of five runs; inputs uploaded from pinned host memory and outputs read back "
                        "every step: each step's CUDA graph holds ikv_step and, on a forked branch, the upload of "
                        "the next step's inputs and the read-back of the previous step's output"},
        "gpu_launches": full["launches"],
        "clocks": full["clocks"],
        "modes": {k: sig(w.batch * K * world / (v["ms"] / 1e3)) for k, v in modes.items()},
    }
    if modes:
        full_v = line["modes"]["full"]
        line["speedup_vs_full"] = {k: sig(v / full_v) for k, v in line["modes"].items() if k != "full"}
        if mode_kernels:
            line["mode_kernel_ms_per_step"] = mode_kernels
        line["modes_note"] = ("full / lazy4 / score_free: refresh every step / every 4th step (Eq. 6) / step 1 "
                              "only, same inputs and compaction as the headline; full_vnorm / full_entropy: the "
                              "VNorm and entropy-weighted scorers under full refresh; full_cumulative / "
                              "full_single_step: the Eq. 3 and Eq. 2 aggregation rules in place of the EMA, full "
                              "refresh; *_every_step: the same "
                              "compaction run on every eviction (max_holes 0); full_stable_left: stable "
                              "compaction that always shifts the suffix left, every step; *_holefill: hole-fill "
                              "compaction every step (same kept sets, survivors not kept in order); "
                              "*_layer_evict: per-layer immediate eviction (each layer keeps its own top-B "
                              "right after its update of a position-indexed state), hole-fill compaction of "
                              "every layer; full_layer_evict_stable: the same with order-preserving compaction")
    if trace is not None:
        line["rank_trace"] = dict({k: {kk: sig(vv) for kk, vv in v.items()} for k, v in trace.items()},
                                  note="full refresh, the headline's inputs and compaction; means over the timed "
                                       "steps and utility rows; raw = the last layer's single-step score, k = the "
                                       "budget (Appendix \"Mechanistic Diagnostics\")")
    line["notes"] = ("per_layer: the headline steps as ikv_step_begin / one ikv_step_layer per layer / ikv_step_end, "
                     "one CUDA graph per step; with_foreign: each layer's q, k_new, v_new first copied by 3 PyTorch "
                     "kernels (not counted in gpu_launches).  trajectory: every decode step of the configuration "
                     "from step 1 (which evicts ~90% of the prefill), deferred compactions included, the steps "
                     "launched one by one with PDL (after one untimed pass).  per_config: the other workloads with "
                     "their headline schedules, at most 20 timed steps after 3 warm-up steps; attend_frac / attend_score_ema_frac of the measured copy peak from "
                     "eager events; speedup_vs_full on the same inputs.  sweep (Qwen-shaped, b=32, 16k): tok/s per "
                     "budget (%) x refresh period r, Lazy speedup over r = 1, alpha at 10% / r = 1.")
    # the last keys: the driver keeps the tail of the line
    line["per_layer"] = {"value": sig(job_throughput(w.batch * K, world, per_layer["split"]["ms"])),
                         "us_per_step": sig(1e3 * per_layer["split"]["ms"] / K),
                         "vs_whole_step": sig(full["ms"] / per_layer["split"]["ms"]),
                         "gpu_launches": per_layer["split"]["launches"],
                         "with_foreign_value": sig(job_throughput(w.batch * K, world, per_layer["foreign"]["ms"]))}
    line["trajectory"] = {"steps": traj_w.steps, "value": sig(job_throughput(w.batch * traj_w.steps, world, traj_ms)),
                          "ms": sig(traj_ms)}
    if others:
        sweep = others["4"].pop("sweep", None)
        line["per_config"] = others
        if sweep:
            line["sweep"] = sweep
    print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()

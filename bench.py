#!/usr/bin/env python
"""Benchmark of the draft + verify hot path (metric: draft+verify sequences/s).

One step = one spec_draft (n heads, full product tree, prune to K) followed by one
spec_verify over base_logits [B, K, n+1, V], on seeded synthetic inputs of the "Llama2-13B-shaped"
configuration (synth.CONFIGS).  Prints ONE JSON line on rank 0.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--config NAME] [--impl ours|reference]

N > 1 (under torchrun): sequences are independent, so every rank runs the full per-GPU
batch with replicated weights and no data-path collective (weak scaling); the reported
value is N * B / max-over-ranks step time.
--impl reference times the CPU oracle (a deliberately plain program) on a bounded sample.
"""
from __future__ import annotations

import argparse
import dataclasses
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "draft+verify sequences/sec"
UNIT = "sequences/s"


# Default run: about 0.6 s of timed steps at the llama2-13b shape, long enough for several clock samples.
DEFAULT_STEPS, DEFAULT_WARMUP = 2000, 50

# DRAM bytes (read + write) per launch as ncu counted them (with the kernels as they are in this tree; None when a kernel
# has changed, until it is captured again)
NCU_TRAFFIC_BYTES = {
    ("llama2-13b", "head_gemm_384_rows"): 270.0e6,
    ("llama2-13b", "verify"): 134.4e6,
}


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return {"hbm_gbs": p["hbm_gbs"], "bf16_tflops": p["bf16_tflops"],
                "bf16_tflops_sustained": p.get("bf16_tflops_sustained", p["bf16_tflops"]), "source": "measured"}
    return {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0, "source": "fallback"}


def kernels_in_graph(graph) -> int:
    """Kernel nodes of a captured graph that was kept."""
    from cuda.bindings import runtime
    raw = runtime.cudaGraph_t(graph.raw_cuda_graph())
    nodes = runtime.cudaGraphGetNodes(raw, runtime.cudaGraphGetNodes(raw)[2])[1]
    return [runtime.cudaGraphNodeGetType(node)[1] for node in nodes].count(runtime.cudaGraphNodeType.cudaGraphNodeTypeKernel)


class ClockSampler:
    """Samples SM clocks and throttle reasons with nvidia-smi while the timed region runs."""
    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu_index = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.gpu_index}", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                 "-lms", "100"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[3:7]):
                if val.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "samples": len(sm), "reasons": sorted(reasons)}


def oracle_weights(sw):
    import oracle
    from paper_2404_19124_b200 import synth
    cfg = sw.cfg
    return oracle.Weights(
        V=cfg.V, d_base=cfg.d_base, d_inner=cfg.d_inner,
        emb=[synth.bf16_bits(t) for t in sw.emb], proj=[synth.bf16_bits(t) for t in sw.proj],
        ln_gamma=[t.detach().cpu().numpy() for t in sw.ln_gamma], ln_beta=[t.detach().cpu().numpy() for t in sw.ln_beta],
        head=[synth.bf16_bits(t) for t in sw.head],
        state_weight=sw.state_weight, emb_weight=sw.emb_weight, ln_eps=sw.ln_eps)


def workload_config(cfg, world: int, n_rot: int):
    """The `config` object of the JSON line: the same keys in the GPU arm and in the reference arm."""
    return {"workload": cfg.name, "B": cfg.B, "K": cfg.K, "n_heads": cfg.n, "topk": list(cfg.topk), "V": cfg.V,
            "d_base": cfg.d_base, "d_inner": cfg.d_inner, "logits_dtype": "bf16",
            "l2": f"weights of more than 1 GB per step exceed L2; verify rotates over {n_rot} distinct logits buffers",
            "parallelism": f"replicas x{world}, sequences independent, no collective"}


def logits_rotation(cfg) -> int:
    """Distinct base_logits buffers a run rotates over (at least 512 MB together, 2 to 8 of them)."""
    logits_bytes = cfg.B * cfg.K * (cfg.n + 1) * cfg.V * 2
    return max(2, min(8, (512 << 20) // logits_bytes + 1))


def time_oracle(cfg, sw, seqs: int, repeats: int):
    """Oracle draft + verify on the first `seqs` sequences of the workload.
    Returns ([(draft seconds, verify seconds)] per repeat, threads used)."""
    import numpy as np
    import oracle
    from paper_2404_19124_b200 import synth
    ow = oracle_weights(sw)
    ctx, tok = synth.make_draft_inputs(cfg, device="cpu", B=seqs)
    ctx_bits, tok_np = synth.bf16_bits(ctx), tok.numpy()
    cand0 = synth.random_cand_tok(cfg, B=seqs)
    logits = synth.bf16_bits(synth.make_base_logits(cfg, cand0, B=seqs))
    times = []
    for _ in range(repeats):
        t0 = time.perf_counter()
        ct, _ = oracle.draft(ow, ctx_bits, tok_np, cfg.topk, cfg.K)
        t1 = time.perf_counter()
        oracle.verify(ct, logits, oracle.BF16)
        times.append((t1 - t0, time.perf_counter() - t1))
    return times, oracle.num_threads()


def run_reference(args, cfg):
    from paper_2404_19124_b200 import synth
    sw = synth.make_weights(cfg, device="cpu")
    # sequences per step: as many of the batch as keep the whole run to about two minutes of CPU time
    probe, _ = time_oracle(cfg, sw, 1, 2)
    seqs = max(1, min(cfg.B, int(120.0 / (min(d + v for d, v in probe) * (args.warmup + args.steps)))))
    times, cores = time_oracle(cfg, sw, seqs, args.warmup + args.steps)
    timed = times[args.warmup:]
    sec = sum(d + v for d, v in timed) / len(timed)
    sec_d = sum(d for d, _ in timed) / len(timed)
    sec_v = sum(v for _, v in timed) / len(timed)
    val = seqs / sec
    sample = f"{seqs} of {cfg.B} sequences of {cfg.name} per step (full tree + verify), plain C oracle, OpenMP"
    out = {
        "impl": "reference", "metric": METRIC, "value": val, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": sec * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
        "config": workload_config(cfg, max(1, args.gpus), logits_rotation(cfg)),
        "cpu_baseline": {"value": val, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample,
                         "draft": seqs / sec_d, "verify": seqs / sec_v},
        "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0,
    }
    print(json.dumps(out), flush=True)


class Workload:
    """One configuration resident in HBM: weights, a handle, draft inputs, rotating logits buffers, workspaces."""

    def __init__(self, cfg, dev, B, synth, torch):
        self.cfg, self.dev, self.B, self.torch = cfg, dev, B, torch
        self.sw = synth.make_weights(cfg, device=dev)
        self.h = B.spec_create(self.sw)
        self.ctx, self.tok = synth.make_draft_inputs(cfg, device=dev)
        n, K, Bn, V = cfg.n, cfg.K, cfg.B, cfg.V
        self.ws = torch.empty(B.spec_draft_workspace_bytes(self.h, Bn, cfg.topk, K), dtype=torch.uint8, device=dev)
        self.cand = torch.empty((Bn, K, n), dtype=torch.int32, device=dev)
        self.logp = torch.empty((Bn, K), dtype=torch.float32, device=dev)
        B.spec_draft(self.h, self.ctx, self.tok, cfg.topk, K, cand_tok=self.cand, cand_logp=self.logp, workspace=self.ws)
        assert B.spec_poll_error(self.ws) == 0
        # base-model logits: rotate over several distinct buffers so verify never re-reads a buffer that could
        # still sit in the 126 MB L2; matches are planted at the tokens the draft proposes
        self.logits_bytes = Bn * K * (n + 1) * V * 2
        self.n_rot = logits_rotation(cfg)
        self.rot = [synth.make_base_logits(dataclasses.replace(cfg, seed=cfg.seed + 100 * i), self.cand, device=dev)
                    for i in range(self.n_rot)]
        self.vws = torch.empty(B.spec_verify_workspace_bytes(Bn, K, n, V, B.SPEC_BF16), dtype=torch.uint8, device=dev)
        self.acc = torch.empty(Bn, dtype=torch.int32, device=dev)
        self.best = torch.empty(Bn, dtype=torch.int32, device=dev)
        self.nxt = torch.empty(Bn, dtype=torch.int32, device=dev)

    def draft(self, i=0):
        c = self.cfg
        self.B.spec_draft(self.h, self.ctx, self.tok, c.topk, c.K, cand_tok=self.cand, cand_logp=self.logp, workspace=self.ws)

    def verify(self, i=0, early=False):
        self.B.spec_verify(self.cand, self.rot[i % self.n_rot], accept_len=self.acc, best_cand=self.best,
                           next_tok=self.nxt, workspace=self.vws, early_exit=early)

    def step(self, i=0):
        self.draft(i)
        self.verify(i)

    def capture(self):
        """n_rot consecutive steps (one per logits buffer) recorded once as a CUDA graph.  Leaves `graph` None
        when stream capture is not available; the steps are then launched call by call."""
        torch, c = self.torch, self.cfg
        self.graph = None
        self.kernels_per_step = 2        # (the least that a draft and a verification can be, if they cannot be counted)
        try:
            cur = torch.cuda.current_stream()
            gs = torch.cuda.Stream()
            gs.wait_stream(cur)
            g = torch.cuda.CUDAGraph(keep_graph=True)
            with torch.cuda.stream(gs):
                # (thread-local capture mode: CUDA calls of other threads, e.g. a process group's watchdog, are
                # none of this capture's business)
                with torch.cuda.graph(g, stream=gs, capture_error_mode="thread_local"):
                    for i in range(self.n_rot):
                        self.B.spec_draft(self.h, self.ctx, self.tok, c.topk, c.K, cand_tok=self.cand, cand_logp=self.logp,
                                          workspace=self.ws, stream=gs)
                        self.B.spec_verify(self.cand, self.rot[i], accept_len=self.acc, best_cand=self.best,
                                           next_tok=self.nxt, workspace=self.vws, stream=gs)
            cur.wait_stream(gs)
            self.kernels_per_step = kernels_in_graph(g) // self.n_rot
            g.instantiate()
            self.graph = g
        except (RuntimeError, ImportError) as e:
            sys.stderr.write(f"CUDA graph capture not available, steps are launched call by call: {e}\n")
        return self.graph is not None

    def run_steps(self, steps: int):
        """Exactly `steps` steps on the current stream: whole replays of the captured graph, the rest call by call."""
        g = getattr(self, "graph", None)
        reps = steps // self.n_rot if g is not None else 0
        for _ in range(reps):
            g.replay()
        for i in range(steps - reps * self.n_rot):
            self.step(i)

    def launch_form(self) -> str:
        if getattr(self, "graph", None) is None:
            return "call by call (spec_draft, spec_verify)"
        return (f"CUDA graph of {self.n_rot} steps (spec_draft + spec_verify captured once, one logits buffer each) "
                f"replayed; steps beyond a whole number of replays call by call")

    def close(self):
        self.graph = None
        self.B.spec_destroy(self.h)
        self.rot = self.sw = self.ws = None
        self.torch.cuda.empty_cache()


def time_steps(torch, W: "Workload", steps: int, warm: int = 5) -> float:
    """Milliseconds per step of W.run_steps(steps), CUDA events on the current stream."""
    stream = torch.cuda.current_stream()
    W.run_steps(warm)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    W.run_steps(steps)
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / steps


def time_loop(torch, fn, iters: int, warm: int = 3) -> float:
    """Milliseconds per call of fn(i), CUDA events on the current stream, after `warm` untimed calls."""
    stream = torch.cuda.current_stream()
    for i in range(warm):
        fn(i)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for i in range(iters):
        fn(i)
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / iters


def head_alone(W: "Workload", level: int, rows: int, iters: int):
    """The head GEMM of `level` with its fused epilogue alone (spec_head_partials), `rows` rows, launched back
    to back: its weights (hundreds of MB) exceed L2, so nothing is re-read from there."""
    torch, B, cfg = W.torch, W.B, W.cfg
    k = cfg.topk[level]
    g = torch.Generator(device=W.dev).manual_seed(5 + level)
    S = (torch.randn(rows, cfg.d_inner, generator=g, device=W.dev) * 0.5).to(torch.bfloat16)
    ws = torch.empty(B.spec_head_workspace_bytes(W.h, rows, k), dtype=torch.uint8, device=W.dev)
    return time_loop(torch, lambda i: B.spec_head_partials(W.h, level, S, k, ws), iters)


def head_roofline(cfg, rows: int, ms: float, peaks, traffic=None):
    """Roofline entry of one head launch: below the ridge the weight stream bounds it, above it the tensor cores."""
    flops = 2.0 * rows * cfg.d_inner * cfg.V
    w_bytes = 2.0 * cfg.V * cfg.d_inner + 2.0 * rows * cfg.d_inner
    ridge = peaks["bf16_tflops"] * 1e12 / (peaks["hbm_gbs"] * 1e9)
    name = f"gemm_tc_kernel (vocabulary head: {rows} x {cfg.d_inner} x {cfg.V})"
    if rows >= ridge:
        ach = flops / (ms * 1e-3) / 1e12
        return {"kernel": name, "bound": "tensor", "achieved": ach, "peak": peaks["bf16_tflops"], "unit": "TFLOP/s",
                "frac": ach / peaks["bf16_tflops"], "traffic": traffic, "peak_source": peaks["source"] + " burst",
                "frac_of_sustained": ach / peaks["bf16_tflops_sustained"], "us": round(ms * 1e3, 2)}
    ach = w_bytes / (ms * 1e-3) / 1e9
    return {"kernel": name, "bound": "hbm", "achieved": ach, "peak": peaks["hbm_gbs"], "unit": "GB/s",
            "frac": ach / peaks["hbm_gbs"], "traffic": traffic, "peak_source": peaks["source"], "us": round(ms * 1e3, 2)}


def verify_roofline(W: "Workload", ms: float, ms_early: float, peaks, traffic=None):
    gbs = W.logits_bytes / (ms * 1e-3) / 1e9
    return {"kernel": "verification: verify_pool_kernel (verify_stream_kernel above 1 GB and for short rows) + verify_accept_kernel",
            "bound": "hbm", "achieved": gbs, "peak": peaks["hbm_gbs"], "unit": "GB/s", "frac": gbs / peaks["hbm_gbs"],
            "peak_source": peaks["source"] + " copy bandwidth", "frac_of_nameplate_8TBs": gbs / 8000.0, "traffic": traffic,
            "us": round(ms * 1e3, 2), "bytes": W.logits_bytes, "early_exit_form_us": round(ms_early * 1e3, 2)}


def workload_entry(W: "Workload", peaks, iters: int, world: int, shard):
    """Step, draft and verify times of one workload and the roofline fractions of its dominant head and of verify."""
    torch, cfg = W.torch, W.cfg
    direct_ms = time_loop(torch, W.step, iters)
    if getattr(W, "graph", None) is None:
        W.capture()
    step_ms = time_steps(torch, W, iters) if W.graph is not None else direct_ms
    draft_ms = time_loop(torch, W.draft, iters)
    verify_ms = time_loop(torch, W.verify, iters)
    early_ms = time_loop(torch, lambda i: W.verify(i, early=True), iters)
    assert W.B.spec_poll_error(W.ws) == 0
    last = cfg.n - 1
    heads = []
    for l in range(cfg.n):
        ms = head_alone(W, l, cfg.nodes(l), max(5, iters // 2))
        heads.append(head_roofline(cfg, cfg.nodes(l), ms, peaks))
    tau = float(W.acc.float().mean().item()) + 1.0
    return {"B": cfg.B, "K": cfg.K, "topk": list(cfg.topk), "V": cfg.V, "d_inner": cfg.d_inner, "steps_timed": iters,
            "step_us": round(step_ms * 1e3, 2), "step_launch": W.launch_form(),
            "step_us_call_by_call": round(direct_ms * 1e3, 2),
            "draft_us": round(draft_ms * 1e3, 2), "verify_us": round(verify_ms * 1e3, 2),
            "verify_early_exit_us": round(early_ms * 1e3, 2),
            "sequences_per_s": shard.whole_job_rate(cfg.B, world, step_ms * 1e-3),
            "dominant_head": heads[last], "heads": [{"rows": cfg.nodes(l), "bound": hd["bound"], "us": hd["us"],
                                                    "frac": round(hd["frac"], 3)} for l, hd in enumerate(heads)],
            "verify_GBs": round(W.logits_bytes / (verify_ms * 1e-3) / 1e9, 1),
            "verify_frac_of_measured_copy": round(W.logits_bytes / (verify_ms * 1e-3) / 1e9 / peaks["hbm_gbs"], 3),
            "synthetic_tokens_per_step": tau}


def run_only(args, cfg, peaks, dev):
    """Single-kernel loops (same launch configuration as inside a step) for ncu captures and sweeps."""
    import torch
    from paper_2404_19124_b200 import binding as B
    from paper_2404_19124_b200 import synth
    stream = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    if args.only in ("head", "head_gemm"):
        if args.vocab:
            cfg = dataclasses.replace(cfg, V=args.vocab)
        rows = args.rows or cfg.nodes(cfg.n - 1)
        k = args.topk or cfg.topk[-1]
        one = dataclasses.replace(cfg, topk=(k,), K=1)
        sw = synth.make_weights(one, device=dev)
        h = B.spec_create(sw)
        if args.block_n:
            B.spec_set_option(h, B.SPEC_OPT_HEAD_BLOCK_N, args.block_n)
        if args.swap_max_rows is not None:
            B.spec_set_option(h, B.SPEC_OPT_HEAD_SWAP_MAX_ROWS, args.swap_max_rows)
        if args.producers:
            B.spec_set_option(h, B.SPEC_OPT_GEMM_PRODUCERS, args.producers)
        if args.pair is not None:
            B.spec_set_option(h, B.SPEC_OPT_HEAD_PAIR, args.pair)
        g = torch.Generator(device=dev).manual_seed(5)
        S = (torch.randn(rows, cfg.d_inner, generator=g, device=dev) * 0.5).to(torch.bfloat16)
        tok = torch.empty((rows, k), dtype=torch.int32, device=dev)
        logp = torch.empty((rows, k), dtype=torch.float32, device=dev)
        ws = torch.empty(B.spec_head_workspace_bytes(h, rows, k), dtype=torch.uint8, device=dev)
        if args.only == "head":
            run = lambda i: B.spec_head_topk(h, 0, S, k, tok=tok, logp=logp, workspace=ws)
        else:
            run = lambda i: B.spec_head_partials(h, 0, S, k, ws)
        flops, nbytes = 2.0 * rows * cfg.d_inner * cfg.V, 2.0 * cfg.V * cfg.d_inner + 2.0 * rows * cfg.d_inner
        what = (f"{'spec_head_topk' if args.only == 'head' else 'spec_head_partials'} rows={rows} d_inner={cfg.d_inner} "
                f"V={cfg.V} topk={k} ({'GEMM + merge kernels' if args.only == 'head' else 'GEMM kernel with its fused epilogue'})")
    else:
        cand = synth.random_cand_tok(cfg, device=dev)
        nbytes = cfg.B * cfg.K * (cfg.n + 1) * cfg.V * 2.0
        n_rot = max(2, min(8, int((512 << 20) // nbytes) + 1))
        rot = [synth.make_base_logits(dataclasses.replace(cfg, seed=cfg.seed + 100 * i), cand, device=dev)
               for i in range(n_rot)]
        vws = torch.empty(B.spec_verify_workspace_bytes(cfg.B, cfg.K, cfg.n, cfg.V, B.SPEC_BF16), dtype=torch.uint8, device=dev)
        outs = [torch.empty(cfg.B, dtype=torch.int32, device=dev) for _ in range(3)]
        run = lambda i: B.spec_verify(cand, rot[i % n_rot], accept_len=outs[0], best_cand=outs[1], next_tok=outs[2], workspace=vws)
        flops = 0.0
        what = f"spec_verify {cfg.name} logits [{cfg.B},{cfg.K},{cfg.n + 1},{cfg.V}] bf16, {n_rot} rotating buffers"
    for i in range(args.warmup):
        run(i)
    torch.cuda.synchronize()
    e0.record(stream)
    for i in range(args.steps):
        run(i)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / args.steps
    print(json.dumps({"only": args.only, "what": what, "us": round(ms * 1e3, 2),
                      "TFLOP/s": round(flops / (ms * 1e-3) / 1e12, 1), "GB/s": round(nbytes / (ms * 1e-3) / 1e9, 1),
                      "frac_bf16_burst": round(flops / (ms * 1e-3) / 1e12 / peaks["bf16_tflops"], 3),
                      "frac_hbm": round(nbytes / (ms * 1e-3) / 1e9 / peaks["hbm_gbs"], 3)}), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=DEFAULT_STEPS)
    ap.add_argument("--warmup", type=int, default=DEFAULT_WARMUP)
    ap.add_argument("--config", default="llama2-13b")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--headline-only", action="store_true", help="skip the `workloads` entries of the other four shapes")
    ap.add_argument("--swap-max-rows", type=int, default=None,
                    help="--only head*: levels of at most this many rows use the weight-stream form (0: never)")
    ap.add_argument("--pair", type=int, default=None, help="--only head*: 1 = CTA pairs for more than 128 rows, 0 = one CTA per tile")
    ap.add_argument("--producers", type=int, default=0, help="--only head*: TMA-issuing threads per CTA (1 or 2)")
    ap.add_argument("--vocab", type=int, default=None, help="--only head*: vocabulary size instead of the workload's")
    ap.add_argument("--topk", type=int, default=None, help="--only head*: branching factor (default: the last level's)")
    ap.add_argument("--only", default=None, choices=["head", "head_gemm", "verify"],
                    help="kernel-level run for profiling: only the vocabulary-head GEMM (+merge) or only verify")
    ap.add_argument("--rows", type=int, default=None, help="--only head: rows of the GEMM (default: last level)")
    ap.add_argument("--block-n", type=int, default=0, help="--only head: force the vocabulary tile width")
    args = ap.parse_args()

    from paper_2404_19124_b200 import synth
    cfg = synth.CONFIGS[args.config]
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))

    if args.impl == "reference":
        if rank == 0:
            if args.steps == DEFAULT_STEPS and args.warmup == DEFAULT_WARMUP:      # defaults are sized for the GPU arm
                args.steps, args.warmup = 3, 1
            run_reference(args, cfg)
        return

    import torch
    from paper_2404_19124_b200 import binding as B
    from paper_2404_19124_b200 import shard

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the draft/verify path has no CPU fallback")
    torch.cuda.set_device(local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))
    if args.warmup < 3:
        args.warmup = 3
    peaks = load_peaks()
    dev = f"cuda:{local_rank}"
    if args.only is not None:
        run_only(args, cfg, peaks, dev)
        return

    # ---------------------------------------------------------------- inputs, resident in HBM
    W = Workload(cfg, dev, B, synth, torch)
    h, n, K, Bn, V = W.h, cfg.n, cfg.K, cfg.B, cfg.V
    ctx, tok, ws, cand, logp, rot, n_rot, vws = W.ctx, W.tok, W.ws, W.cand, W.logp, W.rot, W.n_rot, W.vws
    acc, best, nxt = W.acc, W.best, W.nxt
    logits_bytes = W.logits_bytes
    stream = torch.cuda.current_stream()
    step = W.step

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    def max_over_ranks(x: float) -> float:
        return shard.max_over_ranks(x, dist, dev)

    def timed_region(steps: int):
        """`steps` steps between two events, a barrier and a synchronize on both sides, clocks sampled meanwhile."""
        barrier()
        sampler = ClockSampler(local_rank)
        if rank == 0:
            sampler.start()
            time.sleep(0.25)
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        W.run_steps(steps)
        e1.record(stream)
        barrier()
        ms = max_over_ranks(e0.elapsed_time(e1) / steps)
        return ms, (sampler.stop() if rank == 0 else None)

    # ---------------------------------------------------------------- device-resident timing
    for i in range(args.warmup):
        step(i)
    W.capture()                  # (after the warm-up: every tensor map and attribute the launches need exists)
    launch_form, kernels_per_step = W.launch_form(), W.kernels_per_step
    W.run_steps(n_rot)
    ms_step, clocks = timed_region(args.steps)
    assert B.spec_poll_error(ws) == 0
    tau = float(acc.float().mean().item()) + 1.0
    # Which clock regime was that?  A region of a few milliseconds runs at boost clocks and is over before
    # nvidia-smi has sampled twice; half a second of steps reaches the power-capped clocks.  When the timed
    # region was short a second, long one is measured too and both are reported.
    sustained = None
    region_s = ms_step * 1e-3 * args.steps
    if region_s < 0.5:
        long_steps = int(0.6 / (ms_step * 1e-3)) + 1
        ms_long, clocks_long = timed_region(long_steps)
        sustained = {"steps": long_steps, "ms_per_step": ms_long, "value": shard.whole_job_rate(Bn, world, ms_long * 1e-3),
                     "clocks": clocks_long}
    regime = None
    if rank == 0:
        ck = clocks if sustained is None else sustained["clocks"]
        regime = {"timed_region_s": round(region_s, 4),
                  "kind": "sustained (half a second or more of back-to-back steps)" if region_s >= 0.5
                          else "burst (a timed region of a few milliseconds: boost clocks; see `sustained`)",
                  "sm_mhz_median": clocks["sm_mhz"], "clock_samples": clocks.get("samples"),
                  "sw_power_cap_seen": "sw_power_cap" in (clocks.get("reasons") or []),
                  "sustained_sm_mhz_median": ck["sm_mhz"], "sustained_clock_samples": ck.get("samples"),
                  "sustained_sw_power_cap_seen": "sw_power_cap" in (ck.get("reasons") or [])}

    # ---------------------------------------------------------------- end to end from host buffers
    pin = lambda t: t.cpu().pin_memory()
    h_ctx, h_tok = pin(ctx), pin(tok)
    h_rot = [pin(t) for t in rot[:2]]
    d_logits = torch.empty_like(rot[0])
    d_ctx, d_tok = torch.empty_like(ctx), torch.empty_like(tok)
    h_cand = torch.empty(cand.shape, dtype=cand.dtype).pin_memory()
    h_out = [torch.empty(Bn, dtype=torch.int32).pin_memory() for _ in range(3)]
    h2d = h_ctx.numel() * 2 + h_tok.numel() * 4 + h_rot[0].numel() * 2
    d2h = h_cand.numel() * 4 + 3 * Bn * 4

    copy_stream = torch.cuda.Stream()
    n_groups = min(4, Bn)
    bounds = [Bn * g // n_groups for g in range(n_groups + 1)]
    arrived = [torch.cuda.Event() for _ in range(n_groups)]

    def e2e_step(i):
        # The logits (131 MB at the 13B shape) are most of the step's bytes.  The context state and the token go up
        # first, then the logits follow on a stream of their own, one group of sequences after the other, while
        # the draft runs; each group is verified as soon as it has arrived.
        d_ctx.copy_(h_ctx, non_blocking=True)
        d_tok.copy_(h_tok, non_blocking=True)
        copy_stream.wait_stream(stream)          # (the previous step's verify has read d_logits)
        src = h_rot[i % 2]
        with torch.cuda.stream(copy_stream):
            for g in range(n_groups):
                lo, hi = bounds[g], bounds[g + 1]
                d_logits[lo:hi].copy_(src[lo:hi], non_blocking=True)
                arrived[g].record(copy_stream)
        B.spec_draft(h, d_ctx, d_tok, cfg.topk, K, cand_tok=cand, cand_logp=logp, workspace=ws)
        for g in range(n_groups):
            lo, hi = bounds[g], bounds[g + 1]
            stream.wait_event(arrived[g])
            B.spec_verify(cand[lo:hi], d_logits[lo:hi], accept_len=acc[lo:hi], best_cand=best[lo:hi], next_tok=nxt[lo:hi],
                          workspace=vws)
        h_cand.copy_(cand, non_blocking=True)
        for dst, src in zip(h_out, (acc, best, nxt)):
            dst.copy_(src, non_blocking=True)
        stream.synchronize()      # the caller needs the accepted tokens before the next step

    e2e_steps = max(3, min(args.steps, 50))
    for i in range(3):
        e2e_step(i)
    barrier()
    t0 = time.perf_counter()
    for i in range(e2e_steps):
        e2e_step(i)
    torch.cuda.synchronize()
    e2e_ms = max_over_ranks((time.perf_counter() - t0) * 1e3 / e2e_steps)
    # the grouped form must give what one call over the whole batch gives on the same logits
    e2e_out = [t.clone() for t in h_out]
    W.verify((e2e_steps - 1) % 2)
    torch.cuda.synchronize()
    for got, want in zip(e2e_out, (acc, best, nxt)):
        assert torch.equal(got, want.cpu()), "end-to-end step: grouped verify differs from the whole-batch call"
    del d_logits, h_rot

    # ---------------------------------------------------------------- the same steps launched call by call
    # (the timed region above replays a CUDA graph when capture is available)
    direct_steps = max(3, min(args.steps, 200))
    direct_ms = max_over_ranks(time_loop(torch, step, direct_steps))
    assert B.spec_poll_error(ws) == 0

    # ---------------------------------------------------------------- host time of one spec_draft call
    # CPU clock around the call alone (nothing is waited for): argument checks, the plan, the launches
    torch.cuda.synchronize()
    host_us = []
    for i in range(30):
        t0 = time.perf_counter()
        W.draft(i)
        host_us.append((time.perf_counter() - t0) * 1e6)
        if i % 5 == 4:
            torch.cuda.synchronize()
    host_draft_us = statistics.median(host_us)
    torch.cuda.synchronize()

    # ---------------------------------------------------------------- per-kernel times (CUDA events)
    prof_steps = max(3, min(args.steps, 50))
    B.spec_set_option(h, B.SPEC_OPT_PROFILE, 1)
    sums = None
    for i in range(prof_steps):
        step(i)
        ms = B.spec_profile_read(h)
        sums = ms if sums is None else [a + b for a, b in zip(sums, ms)]
    kern_ms = [s / prof_steps for s in sums]
    B.spec_set_option(h, B.SPEC_OPT_PROFILE, 0)
    draft_ms = time_loop(torch, W.draft, prof_steps)
    verify_ms = time_loop(torch, W.verify, prof_steps)
    verify_early_ms = time_loop(torch, lambda i: W.verify(i, early=True), prof_steps)

    # every level's head alone at its own row count, and the last head at M = B*K rows (GEMM + merge kernels)
    heads = [head_roofline(cfg, cfg.nodes(l), head_alone(W, l, cfg.nodes(l), prof_steps), peaks) for l in range(n)]
    bk_rows = Bn * K
    Sbk = (torch.randn(bk_rows, cfg.d_inner, generator=torch.Generator(device=dev).manual_seed(5), device=dev) * 0.5).to(torch.bfloat16)
    hk = cfg.topk[-1]
    htok = torch.empty((bk_rows, hk), dtype=torch.int32, device=dev)
    hlogp = torch.empty((bk_rows, hk), dtype=torch.float32, device=dev)
    hws = torch.empty(B.spec_head_workspace_bytes(h, bk_rows, hk), dtype=torch.uint8, device=dev)
    bk_ms = time_loop(torch, lambda i: B.spec_head_topk(h, n - 1, Sbk, hk, tok=htok, logp=hlogp, workspace=hws), prof_steps)
    del Sbk, hws

    # the same step with e4m3 copies of the heads attached (used by the levels of up to 128 nodes)
    B.spec_attach_fp8_heads(h)
    ws8 = torch.empty(B.spec_draft_workspace_bytes(h, Bn, cfg.topk, K), dtype=torch.uint8, device=dev)

    def step8(i):
        B.spec_draft(h, ctx, tok, cfg.topk, K, cand_tok=cand, cand_logp=logp, workspace=ws8)
        W.verify(i)

    fp8_step_ms = time_loop(torch, step8, prof_steps)
    assert B.spec_poll_error(ws8) == 0
    B.spec_detach_fp8_heads(h)
    del ws8

    # single-candidate drafts (K = 1, branching 1 everywhere: Sec. 4.2 / Sec. 5) at this workload's widths
    k1 = {}
    one = (1,) * n
    for bk in (1, 16, 64):
        c1 = dataclasses.replace(cfg, topk=one, K=1, B=bk)
        ctx1, tok1 = synth.make_draft_inputs(c1, device=dev)
        ws1 = torch.empty(B.spec_draft_workspace_bytes(h, bk, one, 1), dtype=torch.uint8, device=dev)
        c_out = torch.empty((bk, 1, n), dtype=torch.int32, device=dev)
        l_out = torch.empty((bk, 1), dtype=torch.float32, device=dev)
        ms1 = time_loop(torch, lambda i: B.spec_draft(h, ctx1, tok1, one, 1, cand_tok=c_out, cand_logp=l_out, workspace=ws1),
                        prof_steps)
        assert B.spec_poll_error(ws1) == 0
        w_bytes = sum(2.0 * V * cfg.d_inner + 2.0 * cfg.d_inner * cfg.d_in(l) for l in range(n))
        k1[f"B={bk}"] = {"draft_us": round(ms1 * 1e3, 2), "launches": 2 + 2 * n,
                         "weight_stream_floor_us": round(w_bytes / (peaks["hbm_gbs"] * 1e9) * 1e6, 1),
                         "frac_of_hbm_floor": round(w_bytes / (peaks["hbm_gbs"] * 1e9) / (ms1 * 1e-3), 3)}

    # ---------------------------------------------------------------- vocabulary-parallel heads (N > 1 only)
    # The optional mode for small batches: every rank holds 1/N of each head's vocabulary rows, the per-level
    # lists are all-gathered with NCCL, every rank ends with the same candidates.
    # Whole-draft time with the exchange inside, max over ranks; never part of `value`.
    vocab_parallel = None
    if dist is not None:
        try:
            parts = shard.split_vocab(V, world)
            lo, cnt = parts[rank]
            wsh = dataclasses.replace(W.sw, head=[t[lo:lo + cnt].contiguous() for t in W.sw.head])
            hv = B.spec_create(wsh, vocab_shard=(rank, world, lo))
            wsv = torch.empty(B.spec_draft_workspace_bytes(hv, Bn, cfg.topk, K), dtype=torch.uint8, device=dev)
            cv = torch.empty((Bn, K, n), dtype=torch.int32, device=dev)
            lv = torch.empty((Bn, K), dtype=torch.float32, device=dev)
            vp = lambda i: shard.draft_vocab_parallel(B, hv, ctx, tok, cfg.topk, K, workspace=wsv, cand_tok=cv, cand_logp=lv)
            vp_ms = max_over_ranks(time_loop(torch, vp, max(3, min(args.steps, 50))))
            same = bool(torch.equal(cv, cand))
            vocab_parallel = {"draft_us": round(vp_ms * 1e3, 2), "ranks": world, "unsplit_draft_us": round(draft_ms * 1e3, 2),
                              "same_candidates_as_unsplit_on_rank0": same,
                              "what": "heads split by vocabulary rows over the ranks, NCCL all-gather of the per-level lists included"}
            B.spec_destroy(hv)
        except Exception as e:      # the optional mode must not take the scaling line down with it
            vocab_parallel = {"error": repr(e)[:300]}

    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return

    names = []
    for l in range(n):
        names += [f"proj_gemm[{l}]", f"mix_ln_gelu[{l}]", f"head_gemm[{l}]", f"merge_expand[{l}]"]
    names.append("prune")
    kernels = {nm: round(ms * 1e3, 2) for nm, ms in zip(names, kern_ms)}      # microseconds
    # dominant kernel: the vocabulary-head GEMM of the last (widest) level, alone, back to back
    rows_last = cfg.nodes(n - 1)
    roof = dict(heads[n - 1])
    roof["traffic"] = NCU_TRAFFIC_BYTES.get((cfg.name, f"head_gemm_{rows_last}_rows"))
    roof_verify = verify_roofline(W, verify_ms, verify_early_ms, peaks, NCU_TRAFFIC_BYTES.get((cfg.name, "verify")))
    head_list = {f"head_gemm[{l}]": {"rows": cfg.nodes(l), "bound": hd["bound"], "us": hd["us"], "unit": hd["unit"],
                                     "achieved": round(hd["achieved"], 1), "frac": round(hd["frac"], 3)}
                 for l, hd in enumerate(heads)}

    # ---------------------------------------------------------------- the other workloads (1 GPU only)
    workloads = {cfg.name: {"B": Bn, "K": K, "topk": list(cfg.topk), "V": V, "d_inner": cfg.d_inner, "steps_timed": args.steps,
                            "step_us": round(ms_step * 1e3, 2), "step_launch": launch_form,
                            "step_us_call_by_call": round(direct_ms * 1e3, 2), "draft_us": round(draft_ms * 1e3, 2),
                            "verify_us": round(verify_ms * 1e3, 2), "verify_early_exit_us": round(verify_early_ms * 1e3, 2),
                            "sequences_per_s": shard.whole_job_rate(Bn, world, ms_step * 1e-3), "dominant_head": roof,
                            "heads": [{"rows": cfg.nodes(l), "bound": hd["bound"], "us": hd["us"], "frac": round(hd["frac"], 3)}
                                      for l, hd in enumerate(heads)],
                            "verify_GBs": round(roof_verify["achieved"], 1),
                            "verify_frac_of_measured_copy": round(roof_verify["frac"], 3),
                            "synthetic_tokens_per_step": tau, "host_us_per_spec_draft_call": round(host_draft_us, 1)}}
    cpu = None
    if world == 1:
        sw_cpu = None
        if not args.no_cpu_baseline:
            sw_cpu = synth.SpecWeights(cfg, *[[t.cpu() for t in lst] for lst in (W.sw.emb, W.sw.proj, W.sw.ln_gamma, W.sw.ln_beta, W.sw.head)],
                                       W.sw.state_weight, W.sw.emb_weight, W.sw.ln_eps)
        W.close()
        if not args.headline_only:
            for name, c in synth.CONFIGS.items():
                if name == cfg.name:
                    continue
                Wo = Workload(c, dev, B, synth, torch)
                est = time_loop(torch, Wo.step, 3)
                iters = max(5, min(args.steps, 200, int(150.0 / est) + 1))     # about 0.15 s per timed loop
                entry = workload_entry(Wo, peaks, iters, world, shard)
                torch.cuda.synchronize()
                hu = []
                for i in range(10):
                    t0 = time.perf_counter()
                    Wo.draft(i)
                    hu.append((time.perf_counter() - t0) * 1e6)
                torch.cuda.synchronize()
                entry["host_us_per_spec_draft_call"] = round(statistics.median(hu), 1)
                workloads[name] = entry
                Wo.close()
                del Wo
        if sw_cpu is not None:
            # about 15 s of oracle time: one sequence first to size the sample, then whole passes over as
            # many sequences of the batch as fit
            probe, cores = time_oracle(cfg, sw_cpu, 1, 2)
            seqs = max(1, min(Bn, int(15.0 / min(d + v for d, v in probe))))
            one_pass, cores = time_oracle(cfg, sw_cpu, seqs, 1)
            reps = max(1, min(12, int(round(15.0 / sum(one_pass[0]))) - 1))
            times, cores = time_oracle(cfg, sw_cpu, seqs, reps)
            times = one_pass + times
            t_d, t_v = sum(d for d, _ in times), sum(v for _, v in times)
            cpu = {"value": seqs * len(times) / (t_d + t_v), "unit": UNIT, "cores": cores, "kind": "oracle",
                   "draft": seqs * len(times) / t_d, "verify": seqs * len(times) / t_v,
                   "sample": f"{seqs} of {Bn} sequences of {cfg.name} (full draft tree + verify) x {len(times)} passes, "
                             f"{t_d + t_v:.1f} s of oracle time; `draft` and `verify` are the two parts timed apart, `value` both"}

    out = {
        "metric": METRIC, "value": shard.whole_job_rate(Bn, world, ms_step * 1e-3), "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
        "config": workload_config(cfg, world, n_rot),
        "roofline": roof, "roofline_verify": roof_verify, "head_gemms": head_list,
        "head_gemms_note": "each level's head GEMM with its fused epilogue alone (spec_head_partials), back to back",
        "head_at_BK_rows": {"rows": bk_rows, "us": round(bk_ms * 1e3, 2), "what": "spec_head_topk: head GEMM + merge",
                            "TFLOP/s": round(2.0 * bk_rows * cfg.d_inner * V / (bk_ms * 1e-3) / 1e12, 1),
                            "frac_of_burst": round(2.0 * bk_rows * cfg.d_inner * V / (bk_ms * 1e-3) / 1e12 / peaks["bf16_tflops"], 3)},
        "step_with_e4m3_heads": {"ms_per_step": round(fp8_step_ms, 5), "value": shard.whole_job_rate(Bn, world, fp8_step_ms * 1e-3),
                                 "what": "optional mode: e4m3 head copies on the weight-bound levels, short list re-scored in bf16"},
        "launch": launch_form,
        "call_by_call": {"ms_per_step": round(direct_ms, 5), "steps": direct_steps,
                         "what": "the same steps as separate spec_draft / spec_verify calls on the stream, no graph"},
        "kernel_us": kernels, "kernel_us_note": "separate-kernel form bracketed by events (adds 2-3 us per kernel and takes "
                                                "away the overlap of consecutive kernels); the timed step launches the next "
                                                "level's projection with the head",
        "k1": k1, "k1_note": f"spec_draft with K = 1 and branching 1 at every head, widths of {cfg.name}",
        "workloads": workloads, "regime": regime, "sustained": sustained, "vocab_parallel": vocab_parallel,
        "cpu_baseline": cpu,
        "e2e": {"value": shard.whole_job_rate(Bn, world, e2e_ms * 1e-3), "unit": UNIT, "ms_per_step": e2e_ms,
                "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                "what": "pinned host buffers in, spec_draft + spec_verify call by call, candidates and results back, "
                        "a stream synchronize per step; the logits go up on a second stream in groups of sequences beside the draft, "
                        "each group verified on arrival"},
        "gpu_launches": kernels_per_step * args.steps,
        "clocks": clocks, "synthetic_tokens_per_step": tau,
    }
    print(json.dumps(out), flush=True)
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()

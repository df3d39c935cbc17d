#!/usr/bin/env python
"""Benchmark of the sampled linear backward (VCAS) on B200.

Headline workload: the LLM-sized MLP up-projection (N=8, T=2048, 4096 -> 11008, bf16 inputs, fp32
accumulation) at keep ratios rho = nu = 0.3, with the variance probe (M = 2 Monte-Carlo batches) and the
ratio update run once every F = 100 backward calls.

One STEP = one adaptation period of Alg. 1: 1 probe + 1 ratio update + F sampled backward calls.  The
metric is milliseconds per layer backward = step time / F (probe amortised in).  One call reads 495 MB of
inputs (> the 126 MB L2) and the calls alternate between distinct batches, so every call reads HBM.

Prints ONE JSON line (rank 0).  `--impl reference` times the CPU oracle instead.  The other workloads
(fp32 layer, BERT-base FFN layer with its probe, ViT MLP block, BERT-large stack, the ratio sweep) are
reported under `other_workloads` of the same line.
"""
from __future__ import annotations

import argparse
import json
import os
import re
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

WORKLOAD = "llm_mlp_up"
RHO = NU = 0.3
F_CALLS = 100
PROBE_M = 2
PROBE_ROWS = 128       # rows of the parameter gradient the probe samples (App. D), of the layer's 11008
N_BATCHES = 2
METRIC = "sampled linear-bwd ms/layer"
SLAB = 1024            # d_out columns of the layer that one oracle sample computes (CPU baseline)
SWEEP = (1.0, 0.7, 0.5, 0.3, 0.1)


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        d = json.load(open(path))
        return dict(hbm=d["hbm_gbs"], tc_burst=d["bf16_tflops"], tc_sustained=d["bf16_tflops_sustained"],
                    source="measured")
    return dict(hbm=6650.0, tc_burst=1590.0, tc_sustained=1400.0, source="fallback")


def ncu_traffic(kernel: str, workload: str):
    """DRAM bytes per launch of `kernel` on `workload` from the ncu capture summarised in
    profiles/dram_traffic.md, or None when there is no capture or the kernel's source file has changed
    since it was taken (the table stores the file's SHA-256)."""
    import hashlib
    path = os.path.join(ROOT, "profiles", "dram_traffic.md")
    if not os.path.exists(path):
        return None
    for line in open(path):
        f = [x.strip().strip("`") for x in line.strip().strip("|").split("|")]
        if len(f) >= 5 and f[0] == kernel and f[1] == workload:
            src = os.path.join(ROOT, "paper_2402_17227_b200", "csrc", f[3])
            if not os.path.exists(src):
                return None
            sha = hashlib.sha256(open(src, "rb").read()).hexdigest()
            return float(f[2]) if sha == f[4] else None
    return None


class ClockSampler:
    """Samples nvidia-smi clocks and throttle reasons every 20 ms.  It is started before the warm-up (nvidia-smi
    takes a while to deliver its first sample); stop(t0, t1) keeps the samples whose time stamps lie inside
    the timed region [t0, t1] (host wall clock)."""
    Q = ("timestamp,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index, self.proc, self.lines, self.thread = index, None, [], None

    def start(self):
        import threading
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "20"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True, bufsize=1)
        except OSError:
            self.proc = None
            return

        def pump():
            for line in self.proc.stdout:
                self.lines.append(line)
        self.thread = threading.Thread(target=pump, daemon=True)
        self.thread.start()

    def wait_ready(self, timeout=8.0):
        """Blocks until nvidia-smi has delivered its first sample (it can take seconds on a busy host)."""
        t_end = time.time() + timeout
        while self.proc is not None and not self.lines and time.time() < t_end:
            time.sleep(0.02)

    def stop(self, t0=None, t1=None):
        import datetime
        if self.proc is None:
            return dict(sm_mhz=None, sm_max_mhz=None, reasons=["nvidia-smi unavailable"])
        time.sleep(0.05)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        if self.thread is not None:
            self.thread.join(timeout=2)
        out = "".join(self.lines)
        sm, mx, reasons, seen = [], [], set(), 0
        for line in out.strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            seen += 1
            if t0 is not None and t1 is not None:
                try:
                    ts = datetime.datetime.strptime(f[0], "%Y/%m/%d %H:%M:%S.%f").timestamp()
                except ValueError:
                    continue
                if ts < t0 or ts > t1 + 0.02:
                    continue
            try:
                sm.append(float(f[1])); mx.append(float(f[2]))
            except ValueError:
                continue
            for name, v in zip(("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"), f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        return dict(sm_mhz=statistics.median(sm) if sm else None, sm_max_mhz=max(mx) if mx else None,
                    reasons=sorted(reasons), samples=len(sm), samples_outside_timed_region=seen - len(sm))


# ------------------------------------------------------------------------------------ CPU oracle
def oracle_slab_call(case, rho, nu, batch=0, seed=0, slab=SLAB):
    """One sampled backward by the CPU oracle of the layer restricted to its first `slab` output features
    (all N*T rows, all d_in; dY[:, :slab], W[:slab]).  Returns (seconds, scale) where scale = d_out / slab is
    the factor by which the layer's two products are larger than the sample's."""
    import numpy as np
    from oracle import vcas_oracle as o
    from paper_2402_17227_b200 import inputs
    slab = min(slab, case.d_out)
    X, dY, W = inputs.make_layer(case, batch=batch, d_out=slab)
    to64 = lambda t: t.float().numpy().astype(np.float64)
    X, dY, W = to64(X), to64(dY), to64(W)
    t0 = time.perf_counter()
    o.linear_bwd(X, dY, W, case.N, case.T, float(np.float32(rho)), float(np.float32(nu)), seed)
    return time.perf_counter() - t0, case.d_out / slab


def blas_threads() -> int:
    try:
        from threadpoolctl import threadpool_info
        n = [p.get("num_threads", 1) for p in threadpool_info() if p.get("user_api") == "blas"]
        return max(n) if n else (os.cpu_count() or 1)
    except Exception:
        return os.cpu_count() or 1


def cpu_baseline(case, rho, nu, reps):
    ts = []
    scale = 1.0
    for k in range(reps):
        t, scale = oracle_slab_call(case, rho, nu, batch=k % N_BATCHES, seed=k)
        ts.append(t)
    ms = 1e3 * scale * sum(ts) / len(ts)
    return {"value": ms, "unit": "ms", "cores": blas_threads(), "kind": "oracle",
            "sample": f"{reps} oracle calls (numpy float64, BLAS threads = cores) on a slab of {min(SLAB, case.d_out)} of the "
                      f"layer's {case.d_out} output features with all rows; time scaled by {scale:.2f} (extrapolated)"}


def run_reference(args):
    """The oracle as it stands, on the host cores: each step is one bounded sample of the workload."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import numpy  # noqa: F401  (loads BLAS so that the thread count can be read)
    from paper_2402_17227_b200 import inputs
    case = inputs.CASES[WORKLOAD]
    for w in range(min(args.warmup, 1)):
        oracle_slab_call(case, RHO, NU, batch=w % N_BATCHES, seed=w)
    ts, scale = [], 1.0
    for k in range(args.steps):
        t, scale = oracle_slab_call(case, RHO, NU, batch=k % N_BATCHES, seed=1000 + k)
        ts.append(t)
    ms = 1e3 * scale * sum(ts) / len(ts)
    cores = blas_threads()
    line = {
        "impl": "reference", "metric": METRIC, "value": ms, "unit": "ms", "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * sum(ts) / len(ts), "higher_is_better": False, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": workload_config(case, 1, "one sampled backward by the CPU oracle of a slab of "
                                  f"{SLAB} of the layer's {case.d_out} output features; value = time x {scale:.2f}"),
        "cpu_baseline": {"value": ms, "unit": "ms", "cores": cores, "kind": "oracle",
                         "sample": f"{args.steps} slab calls, one per step ({SLAB} of {case.d_out} output features, "
                                   f"all rows), time scaled by {scale:.2f} (extrapolated)"},
        "e2e": {"value": ms, "unit": "ms", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0,
    }
    print(json.dumps(line))


def workload_config(case, world, step):
    return {"workload": WORKLOAD, "N": case.N, "T": case.T, "d_in": case.d_in, "d_out": case.d_out,
            "rho": RHO, "nu": NU, "step": step,
            "l2": "each call reads 495 MB of inputs (> 126 MB L2); calls alternate between distinct batches",
            "parallelism": f"{world} data-parallel replica(s), no exchange"}


# ---------------------------------------------------------------------------------- GPU helpers
class Timer:
    def __init__(self, torch, dist, dist_util, dev, world):
        self.torch, self.dist, self.du, self.dev, self.world = torch, dist, dist_util, dev, world

    def barrier(self):
        if self.world > 1:
            self.dist.barrier()
        self.torch.cuda.synchronize()

    def __call__(self, fn, reps):
        """Milliseconds of `reps` runs of fn (CUDA events on the current stream), max over ranks."""
        torch = self.torch
        self.barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            fn()
        e1.record()
        self.barrier()
        return self.du.max_over_ranks(e0.elapsed_time(e1), self.dev)


def stage_profile(torch, layer, calls_sampled, calls_dense):
    """Per-stage milliseconds per call from CUDA events at the stage boundaries (kernels serialised on one
    stream).  The calls are enqueued behind a spinning kernel so that their launches are queued when the
    GPU reaches them and the events bracket GPU time, not the host's launch cost."""
    layer.set_profiling(True)
    torch.cuda.synchronize()
    torch.cuda._sleep(4_000_000)
    n_s = calls_sampled()
    ms_s, _ = layer.stage_times()
    torch.cuda._sleep(4_000_000)
    n_d = calls_dense()
    ms_d, _ = layer.stage_times()
    layer.set_profiling(False)
    per = [m / max(1, n_s) for m in ms_s[:5]] + [ms_d[5] / max(1, n_d), ms_d[6] / max(1, n_d)]
    return per


def point_report(case, rho, nu, kA, kW, t_s, t_d, per, pk):
    """One (rho, nu) point in the layout of the report: kept rows, times, achieved rates and fractions."""
    R, d_in, d_out = case.R, case.d_in, case.d_out
    b = 4 if str(case.dtype).endswith("float32") else 2
    score_bytes = R * d_out * b                 # the first pass reads every row of dY once (X: kept rows only, later)
    flops_ratio = 2.0 * R / max(1.0, kA + kW)
    rate = lambda work, ms: (work / ms / 1e9) if ms and ms > 0 else None
    out = {
        "rho": rho, "nu": nu, "kept_A": kA, "kept_W": kW,
        "sampled_ms": t_s, "dense_ms": t_d, "speedup_vs_dense": t_d / t_s if t_s else None,
        "flops_reduction_ratio": flops_ratio,
        "speedup_over_flops_ratio": (t_d / t_s / flops_ratio) if t_s else None,
    }
    if per is not None:
        gbs = score_bytes / per[0] / 1e6 if per[0] else None
        out.update({
            "rownorm": {"ms": per[0], "GBs": gbs, "frac_of_hbm_peak": gbs / pk["hbm"] if gbs else None},
            "sampler_ms": per[1],
            "dx": {"ms": per[2], "TFLOPs": rate(2.0 * kA * d_in * d_out, per[2]),
                   "frac_of_bf16_peak": (rate(2.0 * kA * d_in * d_out, per[2]) or 0) / pk["tc_burst"]},
            "pack_ms": per[3],
            "dw": {"ms": per[4], "TFLOPs": rate(2.0 * kW * d_in * d_out, per[4]),
                   "frac_of_bf16_peak": (rate(2.0 * kW * d_in * d_out, per[4]) or 0) / pk["tc_burst"]},
            "dense_dx_TFLOPs": rate(2.0 * R * d_in * d_out, per[5]),
            "dense_dw_TFLOPs": rate(2.0 * R * d_in * d_out, per[6]),
        })
    return out


def measure_layer(case, vb, inputs, torch, dev, pk, ratios, seeds, profile=True, tensors=None, layer=None,
                  graph=False):
    """Sampled and dense backward of one layer at several (rho, nu): per call and per stage.  graph: the timed
    calls are replayed from a CUDA graph (for layers so small that the host's launch cost would bound them)."""
    N, T, d_in, d_out, R = case.N, case.T, case.d_in, case.d_out, case.R
    if tensors is None:
        tensors = [t.to(dev) for t in inputs.make_layer(case)]
    X, dY, W = tensors
    own = layer is None
    if own:
        layer = vb.Layer(N, T, d_in, d_out, case.dtype)
    dX = torch.empty(R, d_in, dtype=case.dtype, device=dev)
    dW = torch.empty(d_out, d_in, dtype=torch.float32, device=dev)
    out = {"N": N, "T": T, "d_in": d_in, "d_out": d_out, "seeds_per_point": len(seeds),
           "workspace_bytes": layer.workspace_bytes(), "points": []}
    n = len(seeds)

    def time_calls(fn):
        """ms per call of fn(seed) over the seeds (eager launches, or one CUDA graph of all of them replayed)."""
        for sd in seeds[:3]:
            fn(sd)
        torch.cuda.synchronize()
        run = lambda: [fn(sd) for sd in seeds]
        if graph:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                run()
            run = g.replay
            run()
        torch.cuda.synchronize()
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        run()
        e[1].record()
        torch.cuda.synchronize()
        return e[0].elapsed_time(e[1]) / n
    t_d = time_calls(lambda sd: layer.dense_bwd(X, dY, W, dX=dX, dW=dW))
    for rho, nu in ratios:
        t_s = time_calls(lambda sd: layer.linear_bwd_plain(X, dY, W, rho, nu, sd, dX, dW))
        per = None
        if profile:
            def cs():
                for sd in seeds:
                    layer.linear_bwd_plain(X, dY, W, rho, nu, sd, dX, dW)
                return n

            def cd():
                for _ in range(4):
                    layer.dense_bwd(X, dY, W, dX=dX, dW=dW)
                return 4
            per = stage_profile(torch, layer, cs, cd)
        kA = kW = 0.0
        for sd in seeds:
            smp = layer.score(X, dY, rho, nu, sd)
            kA += smp.cntA * T / n
            kW += smp.cntW / n
        out["points"].append(point_report(case, rho, nu, kA, kW, t_s, t_d, per, pk))
    assert layer.device_status() == 0, "device-side wait timed out"
    if own:
        layer.close()
    return out


def measure_bert_base_with_probe(vb, inputs, torch, dev, pk):
    """BERT-base FFN up-projection (rho = .3, nu = .4) with the variance probe (M = 4) every 100 calls: ms per
    layer backward with the probe amortised in, and the sampled / dense call alone (CUDA-graph replays)."""
    case = inputs.CASES["bert_base_ffn_up"]
    F, M, NB = 100, 4, 8
    cfg = vb.default_config()
    cfg.F, cfg.M = F, M
    layer = vb.Layer(case.N, case.T, case.d_in, case.d_out, case.dtype, vb.GEMM_AUTO, cfg)
    host = [inputs.make_layer(case, batch=b) for b in range(NB)]
    W = host[0][2].to(dev)
    Xs, dYs = [h[0].to(dev) for h in host], [h[1].to(dev) for h in host]
    dX = torch.empty(case.R, case.d_in, dtype=case.dtype, device=dev)
    dW = torch.empty(case.d_out, case.d_in, dtype=torch.float32, device=dev)
    probe_out = torch.zeros(5, dtype=torch.float32, device=dev)
    k = [0]

    def calls():
        for _ in range(F):
            b = k[0] % NB
            layer.linear_bwd_plain(Xs[b], dYs[b], W, case.rho, case.nu, k[0], dX, dW)
            k[0] += 1

    def dense():
        for _ in range(F):
            b = k[0] % NB
            layer.dense_bwd(Xs[b], dYs[b], W, dX=dX, dW=dW)
            k[0] += 1
    calls(); dense()
    torch.cuda.synchronize()
    g_calls, g_dense = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g_calls):
        calls()
    with torch.cuda.graph(g_dense):
        dense()

    def period():
        layer.variance_probe(Xs[:M], dYs[:M], W, case.rho, case.nu, 1.0, 7777 + k[0], out=probe_out)
        v = probe_out.cpu().numpy()
        vb.update_ratios(1.0, [1.0], [1.0], [v[0]], [v[1]], [v[2]], [v[3]], [v[4]], cfg)
        g_calls.replay()

    def ms_of(fn, reps):
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            fn()
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / reps
    for _ in range(3):
        period()
    t_period = ms_of(period, 10)
    t_calls = ms_of(g_calls.replay, 10)
    t_dense = ms_of(g_dense.replay, 10)
    pt = measure_layer(case, vb, inputs, torch, dev, pk, [(case.rho, case.nu)], list(range(16)),
                       tensors=(Xs[0], dYs[0], W), layer=layer, graph=True)
    pt.update({"ms_per_layer_with_probe_every_100_calls": t_period / F, "sampled_call_ms_graph_replay": t_calls / F,
               "dense_call_ms_graph_replay": t_dense / F, "probe_M": M,
               "speedup_vs_dense_graph_replay": t_dense / t_calls})
    layer.close()
    return pt


def measure_vit_block(vb, inputs, torch, dev, pk):
    """ViT-base MLP block (N=64, T=197, 768 -> 3072 -> 768): backward through fc2 with the GELU Jacobian fused
    into its dX epilogue, then fc1 on the library's own output through the chain entry point: fc1 takes fc2's
    kept-data list and the row norms its epilogue produced, so dZ1 is not read again for scoring.  The dense block
    is the exact backward of both linears with the same GELU Jacobian in fc2's epilogue."""
    from paper_2402_17227_b200.stack import LinearStack, StackLayer
    fc2, fc1 = inputs.CASES["vit_base_mlp_fc2"], inputs.CASES["vit_base_mlp_fc1"]
    N, T, hidden, d = fc2.N, fc2.T, fc2.d_in, fc2.d_out
    R = N * T
    H = inputs.make_preactivation(fc2, width=hidden).to(dev)
    A = torch.nn.functional.gelu(H.float()).to(torch.bfloat16)
    _, dZ2, W2 = [t.to(dev) for t in inputs.make_layer(fc2)]
    X1, _, W1 = [t.to(dev) for t in inputs.make_layer(fc1)]
    layers = [StackLayer("fc2", hidden, d, W2, [A], [dZ2], H=[H]),
              StackLayer("fc1", d, hidden, W1, [X1], [None], chained=True)]
    stack = LinearStack(layers, N, T, skip_dropped_rows=False, overlap_layers=True)
    rho, nu = [fc2.rho, fc2.rho], [fc2.nu, fc2.nu]
    seeds = list(range(20))
    for sd in seeds[:3]:
        stack.backward(rho, nu, seed=sd)
        stack.dense_backward()
    torch.cuda.synchronize()
    e = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    e[0].record()
    for sd in seeds:
        stack.backward(rho, nu, seed=sd)
    e[1].record()
    for _ in seeds:
        stack.dense_backward()
    e[2].record()
    torch.cuda.synchronize()
    kept = []
    for sd in seeds:
        stack.backward(rho, nu, seed=sd)
        s2, s1 = layers[0].handle.last_sampling(), layers[1].handle.last_sampling()
        kept.append((s2.cntA * T, s2.cntW, s1.cntA * T, s1.cntW))
    kA2, kW2, kA1, kW1 = [sum(k[i] for k in kept) / len(kept) for i in range(4)]
    t_s, t_d = e[0].elapsed_time(e[1]) / len(seeds), e[1].elapsed_time(e[2]) / len(seeds)
    ratio = 4.0 * R / max(1.0, kA2 + kW2 + kA1 + kW1)
    assert stack.device_status() == 0
    stack.close()
    return {"N": N, "T": T, "d": d, "hidden": hidden, "rho": fc2.rho, "nu": fc2.nu, "seeds": len(seeds),
            "sampled_block_ms": t_s, "dense_block_ms": t_d, "speedup_vs_dense": t_d / t_s,
            "kept_rows": {"fc2_A": kA2, "fc2_W": kW2, "fc1_A": kA1, "fc1_W": kW1},
            "flops_reduction_ratio": ratio, "speedup_over_flops_ratio": t_d / t_s / ratio,
            "dense_tflops": 8.0 * R * d * hidden / t_d / 1e9,
            "note": "fc1 is chained to fc2 (kept-data list and row norms handed down); dense block: exact products "
                    "of both linears with the GELU Jacobian in fc2's epilogue"}


def measure_bert_large_stack(vb, inputs, torch, dev, steps=200, F=50, M=2):
    """The 96 linears of a 24-block BERT-large-shaped stack (N=32, T=512, d=1024: QKV 1024->3072, attention output
    1024->1024, FFN 1024->4096->1024 with the GELU Jacobian fused), backward from the top layer down with the
    chain entry point: every layer receives the list of data the layer above kept, the FFN pair hands its row
    norms down from the dX epilogue.  Keep ratios start at rho_l = 0.8 (top) ... 0.2 (bottom), nu = 0.3; every F
    steps Alg. 1 probes every layer (M batches) and updates (s, rho_l, nu_l); the passes of a period are replayed from
    a CUDA graph.  QKV and the attention output have
    no attention between them here, so each linear has its own synthetic incoming gradient; all blocks share one
    pool of activations and gradients per shape (two variants), with their own random weights."""
    import numpy as np
    from paper_2402_17227_b200.stack import LinearStack, StackLayer
    N, T, d, ffn, qkv, blocks = 32, 512, 1024, 4096, 3072, 24
    bf = torch.bfloat16
    cfg = vb.default_config()
    cfg.F, cfg.M = F, M
    cfg.rho_min, cfg.nu_min = 1.0 / N, 1e-3
    specs = [("ffn_down", ffn, d, True, False), ("ffn_up", d, ffn, False, True), ("attn_out", d, d, False, False),
             ("qkv", d, qkv, False, False)]
    pool = {}
    for k, (name, d_in, d_out, gelu, chained) in enumerate(specs):
        c = inputs.LayerCase(name, N, T, d_in, d_out, bf, 1.0, 0.5, 0.5, 0.3, data_seed=4000 + k)
        batches = [inputs.make_layer(c, batch=b, device=dev) for b in range(M)]
        Xs, H = [b[0] for b in batches], None
        if gelu:
            H = [inputs.make_preactivation(c, batch=b, width=d_in, device=dev) for b in range(M)]
            Xs = [torch.nn.functional.gelu(h.float()).to(bf) for h in H]
        pool[name] = (Xs, [b[1] for b in batches], H)
    gw = torch.Generator(dev).manual_seed(99)
    layers = []
    for blk in range(blocks - 1, -1, -1):
        for name, d_in, d_out, gelu, chained in specs:
            W = (torch.randn(d_out, d_in, generator=gw, device=dev, dtype=torch.float32) * 0.02).to(bf)
            Xs, dYs, H = pool[name]
            layers.append(StackLayer(f"b{blk}.{name}", d_in, d_out, W, Xs, dYs, H=H, chained=chained))
    # every consumer takes the kept-data list; a layer's dW branch runs beside the layers below it
    stack = LinearStack(layers, N, T, config=cfg, skip_dropped_rows=True, overlap_layers=True)
    for hd in stack.handles.values():
        hd.set_probe_subsample(128, 0)          # App. D: the probe's variances on a sample of the parameter rows
    L = len(layers)
    # Alg. 1's state in layer order (index 0 = lowest layer); the stack runs in backward order (top first)
    state = dict(s=0.75, rho=list(np.linspace(0.2, 0.8, L)), nu=[0.3] * L)
    traj = []

    def adapt(t):
        V = stack.probe(state["rho"][::-1], state["nu"][::-1], state["s"], seed=31 * t).cpu().numpy()[::-1]
        s, rho, nu = vb.update_ratios(state["s"], state["rho"], state["nu"], V[:, 0], V[:, 1], V[:, 2], V[:, 3],
                                      V[:, 4], cfg)
        state.update(s=s, rho=rho, nu=nu)
        traj.append({"t": t, "s": s, "rho_bottom": rho[0], "rho_top": rho[-1], "nu_min": min(nu), "nu_max": max(nu)})

    PASSES = 5          # passes (with their own seeds and batch variants) captured into one CUDA graph

    def capture(t0):
        # The ratios only change when Alg. 1 adapts them, so the passes of a period are captured once into a CUDA
        # graph (the library neither synchronises nor allocates) and replayed: the host's launch cost of 96 calls
        # of about eight kernels each would otherwise bound the step.
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for k in range(PASSES):
                stack.backward(state["rho"][::-1], state["nu"][::-1], seed=t0 + k, variant=t0 + k)
        return g

    def run_period(t0, n):
        adapt(t0)
        g = capture(t0)
        for _ in range(n // PASSES):
            g.replay()
        return g
    for t in range(3):                          # warm-up at the initial ratios
        stack.backward(state["rho"][::-1], state["nu"][::-1], seed=t, variant=t)
    stack.dense_backward()
    torch.cuda.synchronize()
    e = [torch.cuda.Event(enable_timing=True) for _ in range(6)]
    e[0].record()
    g_last = None
    for t0 in range(0, steps, F):
        g_last = run_period(t0, F)
    e[1].record()
    torch.cuda.synchronize()
    ms_step = e[0].elapsed_time(e[1]) / steps
    # at the final ratios: sampled passes alone (graph replay and eager launches), dense passes (graph replay)
    g_dense = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g_dense):
        for k in range(PASSES):
            stack.dense_backward(variant=k)
    torch.cuda.synchronize()
    reps = 4
    e[1].record()
    for _ in range(reps):
        g_last.replay()
    e[2].record()
    for _ in range(reps):
        g_dense.replay()
    e[3].record()
    for t in range(PASSES):
        stack.backward(state["rho"][::-1], state["nu"][::-1], seed=10_000 + t, variant=t)
    e[4].record()
    torch.cuda.synchronize()
    ms_sampled = e[1].elapsed_time(e[2]) / (reps * PASSES)
    ms_dense = e[2].elapsed_time(e[3]) / (reps * PASSES)
    ms_sampled_eager = e[3].elapsed_time(e[4]) / PASSES
    ev, kept = [], []

    def hook(i, lay, after):
        x = torch.cuda.Event(enable_timing=True)
        x.record()
        ev.append(x)
        if after:
            smp = lay.handle.last_sampling()
            kept.append((lay.name.split(".")[1], smp.cntA * T, smp.cntW, lay.d_in * lay.d_out))
    by_type, dense_by_type = {}, {}
    for rep in range(3):
        ev.clear()
        stack.backward(state["rho"][::-1], state["nu"][::-1], seed=20_000 + rep, variant=rep, hook=hook)
        torch.cuda.synchronize()
        for i, lay in enumerate(layers):
            k = lay.name.split(".")[1]
            by_type[k] = by_type.get(k, 0.0) + ev[2 * i].elapsed_time(ev[2 * i + 1]) / 3
    ev2 = []

    def hook2(i, lay, after):
        x = torch.cuda.Event(enable_timing=True)
        x.record()
        ev2.append(x)
    stack.dense_backward(hook=hook2)
    torch.cuda.synchronize()
    for i, lay in enumerate(layers):
        k = lay.name.split(".")[1]
        dense_by_type[k] = dense_by_type.get(k, 0.0) + ev2[2 * i].elapsed_time(ev2[2 * i + 1])
    flops_dense = sum(2.0 * 2.0 * N * T * lay.d_in * lay.d_out for lay in layers)
    flops_sampled = sum(2.0 * (a + w) * dd for _, a, w, dd in kept) / 3
    out = {
        "N": N, "T": T, "d": d, "blocks": blocks, "linears": L, "steps": steps, "F": F, "M": M,
        "ms_per_step_with_probes": ms_step, "ms_per_step_sampled_at_final_ratios": ms_sampled,
        "ms_per_step_sampled_eager_launches": ms_sampled_eager,
        "ms_per_step_dense": ms_dense, "speedup_vs_dense": ms_dense / ms_sampled,
        "speedup_vs_dense_with_probes": ms_dense / ms_step,
        "flops_reduction_ratio": flops_dense / max(1.0, flops_sampled),
        "speedup_over_flops_ratio": (ms_dense / ms_sampled) / (flops_dense / max(1.0, flops_sampled)),
        "dense_tflops": flops_dense / ms_dense / 1e9,
        "ms_per_step_by_layer_type_sampled": by_type, "ms_per_step_by_layer_type_dense": dense_by_type,
        "kept_rows_mean_by_type": {k: {"kept_A": float(np.mean([a for n_, a, w, _ in kept if n_ == k])),
                                       "kept_W": float(np.mean([w for n_, a, w, _ in kept if n_ == k]))}
                                   for k in by_type},
        "initial": {"s": 0.75, "rho_top": 0.8, "rho_bottom": 0.2, "nu": 0.3},
        "trajectory": traj, "final": {"s": state["s"], "rho": [round(float(x), 4) for x in state["rho"]],
                                      "nu": [round(float(x), 4) for x in state["nu"]]},
        "workspace_bytes": stack.workspace_bytes(), "handles": len(stack.handles), "probe_sampled_rows": 128,
    }
    assert stack.device_status() == 0
    stack.close()
    return out


def kernel_run(args):
    """A small run for profilers: `--kernel-run WORKLOAD` makes 2 warm-up + `--calls` sampled backward calls and as
    many dense ones of one workload at (--rho, --nu), inputs drawn on the device, and prints one JSON line."""
    import torch
    from paper_2402_17227_b200 import binding as vb
    from paper_2402_17227_b200 import build as vbuild
    from paper_2402_17227_b200 import inputs
    vbuild.build()
    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    case = inputs.CASES[args.kernel_run]
    X, dY, W = inputs.make_layer(case, device=dev)
    layer = vb.Layer(case.N, case.T, case.d_in, case.d_out, case.dtype)
    dX = torch.empty(case.R, case.d_in, dtype=case.dtype, device=dev)
    dW = torch.empty(case.d_out, case.d_in, dtype=torch.float32, device=dev)
    for k in range(2 + args.calls):
        layer.linear_bwd_plain(X, dY, W, args.rho, args.nu, k, dX, dW)
    torch.cuda.synchronize()
    l0 = layer.launch_count()
    for k in range(args.calls):
        layer.dense_bwd(X, dY, W, dX=dX, dW=dW)
    torch.cuda.synchronize()
    smp = layer.last_sampling()
    print(json.dumps({"workload": case.name, "rho": args.rho, "nu": args.nu, "calls": args.calls,
                      "kept_A": smp.cntA * case.T, "kept_W": smp.cntW, "launches_sampled": l0,
                      "status": layer.device_status()}))
    layer.close()


def shortened(v):
    """The same report in fewer characters, so that the one line it goes into stays within 12 KB: numbers to four digits, lists
    of like records as a table, long lists of numbers by their ends."""
    if isinstance(v, float):
        return float(f"{v:.4g}")
    if isinstance(v, dict):
        return {k: shortened(x) for k, x in v.items()}
    if isinstance(v, list) and len(v) > 2 and all(isinstance(x, dict) for x in v):
        def flat(d, prefix=""):
            return {k2: x2 for k, x in d.items() for k2, x2 in (flat(x, prefix + k + ".") if isinstance(x, dict) else
                                                                {prefix + k: x}).items()}
        rows = [flat(shortened(x)) for x in v]
        if all(list(r) == list(rows[0]) for r in rows):
            return {"columns": list(rows[0]), "rows": [list(r.values()) for r in rows]}
    if isinstance(v, list) and len(v) > 16 and all(isinstance(x, (int, float)) for x in v):
        return {"first": shortened(v[0]), "last": shortened(v[-1]), "min": shortened(min(v)), "max": shortened(max(v)), "count": len(v)}
    if isinstance(v, (list, tuple)):
        return [shortened(x) for x in v]
    return v


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="vcas", choices=["vcas", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extra", action="store_true", help="skip the workloads reported under other_workloads")
    ap.add_argument("--sweep", default="grid", choices=["grid", "diag"],
                    help="ratio sweep on the headline layer: the 5 x 5 grid of (rho, nu), or its diagonal only")
    ap.add_argument("--kernel-run", default=None, metavar="WORKLOAD",
                    help="profiling aid: a few sampled and dense calls of one workload, nothing else")
    ap.add_argument("--rho", type=float, default=RHO)
    ap.add_argument("--nu", type=float, default=NU)
    ap.add_argument("--calls", type=int, default=2)
    args = ap.parse_args()
    if args.kernel_run is not None:
        return kernel_run(args)
    if args.impl == "reference":
        return run_reference(args)
    args.warmup = max(args.warmup, 3)

    import torch
    import torch.distributed as dist

    from paper_2402_17227_b200 import binding as vb
    from paper_2402_17227_b200 import build as vbuild
    from paper_2402_17227_b200 import dist_util
    from paper_2402_17227_b200 import inputs

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)
    if rank == 0:
        vbuild.build()
    if world > 1:
        dist.barrier()
    vb.lib()
    pk = peaks()
    timed = Timer(torch, dist, dist_util, dev, world)

    case = inputs.CASES[WORKLOAD]
    N, T, d_in, d_out, R = case.N, case.T, case.d_in, case.d_out, case.R
    cfg = vb.default_config()
    cfg.F, cfg.M = F_CALLS, PROBE_M
    layer = vb.Layer(N, T, d_in, d_out, case.dtype, vb.GEMM_AUTO, cfg)

    # rank r draws its own batches (data-parallel replicas: per-replica sampling, no exchange here)
    host = [inputs.make_layer(case, batch=b) for b in dist_util.rank_batches(rank, N_BATCHES)]
    W = host[0][2].to(dev)
    Xs = [h[0].to(dev) for h in host]
    dYs = [h[1].to(dev) for h in host]
    dX = torch.empty(R, d_in, dtype=case.dtype, device=dev)
    dW = torch.empty(d_out, d_in, dtype=torch.float32, device=dev)
    probe_out = torch.zeros(5, dtype=torch.float32, device=dev)
    state = dict(s=1.0, rho=[1.0], nu=[1.0])
    call_no = [0]

    def calls_only():
        for _ in range(F_CALLS):
            b = call_no[0] % N_BATCHES
            layer.linear_bwd_plain(Xs[b], dYs[b], W, RHO, NU, call_no[0], dX, dW)
            call_no[0] += 1

    def dense_only():
        for _ in range(F_CALLS):
            b = call_no[0] % N_BATCHES
            layer.dense_bwd(Xs[b], dYs[b], W, dX=dX, dW=dW)
            call_no[0] += 1

    # The F backward calls of a period are captured once into a CUDA graph (the library neither
    # synchronises nor allocates, so its calls can be captured) and replayed every step: a training
    # loop would capture its step the same way, and replay removes the host's launch cost.
    calls_only(); dense_only()
    torch.cuda.synchronize()
    l_before = layer.launch_count()
    graph_calls = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph_calls):
        calls_only()
    launches_per_period = layer.launch_count() - l_before
    graph_dense = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph_dense):
        dense_only()
    probe_launches = [0]

    # the probe on all rows of the parameter gradient and on a sample of them (App. D); the steps use the sample
    def probe_ms():
        for _ in range(2):
            layer.variance_probe(Xs[:PROBE_M], dYs[:PROBE_M], W, RHO, NU, 1.0, 1, out=probe_out)
        return timed(lambda: layer.variance_probe(Xs[:PROBE_M], dYs[:PROBE_M], W, RHO, NU, 1.0, 1, out=probe_out), 3) / 3
    probe_full_ms = probe_ms()
    layer.set_probe_subsample(PROBE_ROWS, 0)
    probe_sub_ms = probe_ms()

    def step():
        # Alg. 1: every F calls probe the variances on M batches and update (s, rho_l, nu_l) ...
        l0 = layer.launch_count()
        layer.variance_probe(Xs[:PROBE_M], dYs[:PROBE_M], W, RHO, NU, state["s"], 7777 + call_no[0], out=probe_out)
        probe_launches[0] = layer.launch_count() - l0
        v = probe_out.cpu().numpy()
        s_new, rho_new, nu_new = vb.update_ratios(state["s"], state["rho"], state["nu"], [v[0]], [v[1]], [v[2]],
                                                  [v[3]], [v[4]], cfg)
        state.update(s=s_new, rho=rho_new, nu=nu_new)
        # ... then F sampled backward calls (at the workload's fixed ratios, so that every step does the same work)
        graph_calls.replay()

    clocks = ClockSampler(local)
    if rank == 0:
        clocks.start()
    for _ in range(args.warmup):
        step()
    if rank == 0:
        clocks.wait_ready()       # nvidia-smi is delivering samples from here on
    wall0 = time.time()
    total_ms = timed(step, args.steps)
    wall1 = time.time()
    launches = args.steps * (launches_per_period + probe_launches[0])
    clock_info = clocks.stop(wall0, wall1) if rank == 0 else None
    ms_per_step = total_ms / args.steps
    value = dist_util.ms_per_layer(ms_per_step, F_CALLS, world)      # whole-job: all ranks' calls per unit time

    # -- the same period without the probe, the dense backward (graph replays), and per-stage times
    reps = 3
    ms_sampled = timed(graph_calls.replay, reps) / (reps * F_CALLS)
    ms_dense = timed(graph_dense.replay, reps) / (reps * F_CALLS)
    prof_seeds = [99000 + k for k in range(40)]

    def prof_sampled():
        for k, sd in enumerate(prof_seeds):
            layer.linear_bwd_plain(Xs[k % N_BATCHES], dYs[k % N_BATCHES], W, RHO, NU, sd, dX, dW)
        return len(prof_seeds)

    def prof_dense():
        for k in range(8):
            layer.dense_bwd(Xs[k % N_BATCHES], dYs[k % N_BATCHES], W, dX=dX, dW=dW)
        return 8
    per = stage_profile(torch, layer, prof_sampled, prof_dense)
    kept_A = kept_W = 0.0
    for k, sd in enumerate(prof_seeds):      # realised kept rows of those calls (the FLOPs the products did)
        smp = layer.score(Xs[k % N_BATCHES], dYs[k % N_BATCHES], RHO, NU, sd)
        kept_A += smp.cntA * T / len(prof_seeds)
        kept_W += smp.cntW / len(prof_seeds)
    assert layer.device_status() == 0, "device-side wait timed out"

    # -- data-parallel replicas (App. C): the sum of the replicas' dW, issued after every call and overlapped with
    # the calls that follow, waited for at the end of the period (eager launches; the headline's calls are graph replays)
    ms_ddp = None
    if world > 1:
        red = dist_util.GradReducer()
        dWs = [torch.empty_like(dW) for _ in range(4)]

        def ddp_period():
            for k in range(F_CALLS):
                b = k % N_BATCHES
                if len(red.works) >= 4:
                    red.works.pop(0).wait()     # the buffer about to be rewritten has been reduced
                layer.linear_bwd_plain(Xs[b], dYs[b], W, RHO, NU, 777000 + k, dX, dWs[k % 4])
                red.reduce_async(dWs[k % 4])
            red.wait()
        ddp_period()
        ms_ddp = timed(ddp_period, 2) / (2 * F_CALLS * world)

    # -- end to end through the C ABI from pinned host buffers (H2D of X, dY; D2H of dX, dW every call)
    pin = [(h[0].pin_memory(), h[1].pin_memory()) for h in host[:2]]
    hX, hdY = torch.empty_like(Xs[0]), torch.empty_like(dYs[0])
    out_dX = torch.empty(R, d_in, dtype=case.dtype).pin_memory()
    out_dW = torch.empty(d_out, d_in, dtype=torch.float32).pin_memory()

    def e2e_calls(n):
        for k in range(n):
            hX.copy_(pin[k % 2][0], non_blocking=True)
            hdY.copy_(pin[k % 2][1], non_blocking=True)
            layer.linear_bwd_plain(hX, hdY, W, RHO, NU, 424242 + k, dX, dW)
            out_dX.copy_(dX, non_blocking=True)
            out_dW.copy_(dW, non_blocking=True)
        torch.cuda.synchronize()

    e2e_calls(2)
    n_e2e = 6
    e2e_serial_ms = timed(lambda: e2e_calls(n_e2e), 1) / (n_e2e * world)

    # The same calls as a user would pipeline them: inputs and outputs double-buffered on the device, the copy
    # of call k + 1's inputs and of call k - 1's outputs on their own streams beside call k's kernels (PCIe is
    # full duplex).  Every call still copies all of its inputs in and all of its outputs out.
    cur = torch.cuda.current_stream()
    s_in, s_out = torch.cuda.Stream(), torch.cuda.Stream()
    dXs2 = [dX, torch.empty_like(dX)]
    dWs2 = [dW, torch.empty_like(dW)]
    inX = [hX, torch.empty_like(hX)]
    indY = [hdY, torch.empty_like(hdY)]

    def e2e_pipelined(n):
        ev_in = [torch.cuda.Event() for _ in range(n)]
        ev_done = [torch.cuda.Event() for _ in range(n)]
        ev_out = [torch.cuda.Event() for _ in range(n)]
        for k in range(n):
            b = k % 2
            with torch.cuda.stream(s_in):
                if k >= 2:
                    s_in.wait_event(ev_done[k - 2])      # the call that read this input buffer has finished
                inX[b].copy_(pin[b][0], non_blocking=True)
                indY[b].copy_(pin[b][1], non_blocking=True)
                ev_in[k].record(s_in)
            cur.wait_event(ev_in[k])
            if k >= 2:
                cur.wait_event(ev_out[k - 2])            # this output buffer has been copied out
            layer.linear_bwd_plain(inX[b], indY[b], W, RHO, NU, 434343 + k, dXs2[b], dWs2[b])
            ev_done[k].record(cur)
            with torch.cuda.stream(s_out):
                s_out.wait_event(ev_done[k])
                out_dX.copy_(dXs2[b], non_blocking=True)
                out_dW.copy_(dWs2[b], non_blocking=True)
                ev_out[k].record(s_out)
        torch.cuda.synchronize()

    e2e_pipelined(2)
    n_pipe = 8
    e2e_ms = timed(lambda: e2e_pipelined(n_pipe), 1) / (n_pipe * world)
    h2d = Xs[0].numel() * 2 + dYs[0].numel() * 2
    d2h = dX.numel() * 2 + dW.numel() * 4
    del pin, hX, hdY, out_dX, out_dW, inX, indY, dXs2, dWs2

    extra = None
    if world == 1 and not args.no_extra:
        sweep_seeds = list(range(20))
        grid = [(r, n) for r in SWEEP for n in SWEEP if args.sweep == "grid" or r == n]
        extra = {
            # the 5 x 5 grid of keep ratios on the headline layer, 20 seeds per point
            "llm_mlp_up_ratio_sweep": measure_layer(case, vb, inputs, torch, dev, pk, grid, sweep_seeds,
                                                    tensors=(Xs[0], dYs[0], W), layer=layer),
        }
        del Xs, dYs, host
        torch.cuda.empty_cache()
        extra["fp32_small"] = measure_layer(inputs.CASES["fp32_small"], vb, inputs, torch, dev, pk, [(0.5, 0.5)],
                                            list(range(50)), graph=True)
        extra["bert_base_ffn_up"] = measure_bert_base_with_probe(vb, inputs, torch, dev, pk)
        extra["vit_base_mlp_block"] = measure_vit_block(vb, inputs, torch, dev, pk)
        torch.cuda.empty_cache()
        extra["bert_large_stack"] = measure_bert_large_stack(vb, inputs, torch, dev)
        torch.cuda.empty_cache()
        # a BERT-large FFN linear at the keep ratios of a top, a middle and a bottom layer
        extra["bert_large_ffn_up"] = measure_layer(inputs.CASES["bert_large_ffn_up"], vb, inputs, torch, dev, pk,
                                                   [(0.8, 0.3), (0.5, 0.3), (0.2, 0.3)], list(range(20)))
        torch.cuda.empty_cache()
        # twice the rows of any other workload (N = 16, T = 2048: 32768 rows, more SampleW scores than fit one
        # CTA's registers or a quarter of its shared memory)
        long_case = inputs.LayerCase("long_seq_ffn_up", 16, 2048, 1024, 4096, torch.bfloat16, 1.0, 0.5, 0.5, 0.3)
        extra["long_seq_ffn_up"] = measure_layer(long_case, vb, inputs, torch, dev, pk, [(0.5, 0.3), (0.3, 0.3)],
                                                 list(range(10)))

    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return

    names = ["rownorm_kernel", "sampler_kernel", "umma_dx_kernel", "pack_kernel", "umma_dw_kernel"]
    bytes_score = R * d_out * 2                                   # the scoring pass reads every row of dY once
    flops_dx = 2.0 * kept_A * d_in * d_out
    flops_dw = 2.0 * kept_W * d_in * d_out
    stages = {
        "rownorm_kernel": dict(ms=per[0], bound="hbm", achieved=bytes_score / per[0] / 1e6 if per[0] else None),
        "sampler_kernel": dict(ms=per[1], bound="latency"),
        "umma_dx_kernel": dict(ms=per[2], bound="tensor", achieved=flops_dx / per[2] / 1e9 if per[2] else None),
        "pack_kernel": dict(ms=per[3], bound="hbm"),
        "umma_dw_kernel": dict(ms=per[4], bound="tensor", achieved=flops_dw / per[4] / 1e9 if per[4] else None),
    }
    # The stage times come from 40 calls back to back behind a timed region of seconds: the GPU sits at its power
    # cap (see `clocks`), so tensor-bound stages are held against the sustained bf16 peak, not the burst one.
    for k, v in stages.items():
        if v.get("achieved"):
            v["frac"] = v["achieved"] / (pk["hbm"] if v["bound"] == "hbm" else pk["tc_sustained"])
            if v["bound"] == "tensor":
                v["frac_of_burst_peak"] = v["achieved"] / pk["tc_burst"]
    dom = max(range(5), key=lambda i: per[i])
    dname = names[dom]
    if stages[dname]["bound"] == "tensor":
        roof = dict(bound="tensor", kernel=dname, achieved=stages[dname]["achieved"], peak=pk["tc_sustained"],
                    unit="TFLOP/s", traffic=ncu_traffic(dname, WORKLOAD),
                    peak_source=pk["source"] + " bf16 sustained (kernel timed inside a long, power-capped run)",
                    frac_of_burst_peak=stages[dname]["achieved"] / pk["tc_burst"])
    else:
        if dname != "rownorm_kernel":   # the small latency-bound stages are reported under the scoring pass
            dname = "rownorm_kernel"
        roof = dict(bound="hbm", kernel=dname, achieved=stages[dname]["achieved"], peak=pk["hbm"], unit="GB/s",
                    traffic=ncu_traffic(dname, WORKLOAD), peak_source=pk["source"] + " copy bandwidth")
    roof["frac"] = roof["achieved"] / roof["peak"] if roof["achieved"] else None
    roof["kernel_ms"] = stages[dname]["ms"]

    flops_ratio = 2.0 * R / max(1, kept_A + kept_W)
    line = {
        "metric": METRIC, "value": value, "unit": "ms", "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_per_step, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
        "dtype": "bf16", "data": "synthetic",
        "config": workload_config(case, world, f"1 variance probe (M={PROBE_M}) + 1 ratio update + {F_CALLS} sampled "
                                  "backward calls (the calls replayed from one CUDA graph)"),
        "clocks": clock_info,
        "e2e": {"value": e2e_ms, "unit": "ms", "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                "serial_value": e2e_serial_ms,
                "note": "one vcas_linear_bwd per step with X, dY copied from pinned host memory and dX, dW copied back "
                        "to pinned host memory; value: the copies of neighbouring steps run on their own streams "
                        "beside the kernels (double-buffered); serial_value: copy in, compute, copy out one after "
                        "the other"},
        "gpu_launches": int(launches),
        "roofline": roof,
        "stages": stages,
        "sampled_ms_per_layer": ms_sampled, "dense_ms_per_layer": ms_dense,
        "ms_per_layer_with_dw_allreduce_overlapped": ms_ddp,
        "dense_stages_ms": {"umma_dx_kernel": per[5], "umma_dw_kernel": per[6]},
        "speedup_vs_dense": ms_dense / ms_sampled if ms_sampled else None,
        "flops_reduction_ratio": flops_ratio,
        "speedup_over_flops_ratio": (ms_dense / ms_sampled) / flops_ratio if ms_sampled else None,
        "dense_tflops": 4.0 * R * d_in * d_out / ms_dense / 1e9,
        "kept_rows": {"kept_A": kept_A, "kept_W": kept_W, "R": R, "note": "mean over the 40 profiled calls"},
        "workspace_bytes": layer.workspace_bytes(),
        "probe": {"M": PROBE_M, "ms_all_parameter_rows": probe_full_ms, "ms_sampled_rows": probe_sub_ms,
                  "sampled_rows": PROBE_ROWS, "of_rows": d_out, "used_in_steps": "sampled rows"},
        "adaptation_state": state,
        "other_workloads": extra,
    }
    if not args.no_cpu_baseline and world == 1:
        line["cpu_baseline"] = cpu_baseline(case, RHO, NU, reps=3)
    for key in ("stages", "other_workloads", "roofline", "adaptation_state"):
        line[key] = shortened(line[key])
    print(json.dumps(line, separators=(",", ":")))
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()

"""Benchmark: depth-staggered scaled-Fibonacci sparse attention on GB300.

Default workload (one "step" = the whole hot path over one batch): 16 layers
of forward + backward, B=16, H=8, T=1024, D=64, W=8, Fibonacci base K=15,
learned schedule alpha_l = 0.5 + sigmoid(theta_l) with theta_l ~ N(0, 0.5),
bf16 I/O with fp32 accumulation, distinct per-layer buffers (1.07 GB of
inputs per step, larger than L2).  Metric: query-heads per second (B*H*T per
layer per fwd+bwd), with the achieved HBM bandwidth of the dominant kernel
against the measured GB300 copy bandwidth.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gb300|reference]

Under torchrun each rank runs its own copy of the workload on its own GPU
(weak scaling, replicas only: the path has no exchange step); rank 0 prints
one JSON line.  ``--impl reference`` times the fp64 CPU oracle on a bounded
sample of the same workload (the paper ships no code to run).
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402
import torch  # noqa: E402

METRIC = "queries/s and achieved HBM GB/s (% of GB300 roofline), fwd+bwd, T=1024"
UNIT = "query-heads/s"
B, H, T, D, W, L, K = 16, 8, 1024, 64, 8, 16, 15
SEED = 3                      # learned-alpha backward workload
ESIZE = 2                     # bf16
ROW_BYTES = D * ESIZE


def max_over_ranks(x: float, device=None) -> float:
    """Slowest rank's time: all-reduce MAX over the process group (NCCL on
    GPUs, gloo on CPU); the identity when not distributed."""
    dist = torch.distributed
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(x)
    on_gpu = dist.get_backend() == "nccl"
    t = torch.tensor([float(x)], dtype=torch.float64, device=device if on_gpu else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(world: int, steps: int, ms_max: float) -> float:
    """Whole-job query-heads per second: every rank processes its own copy of
    the per-rank workload (weak scaling), timed by the slowest rank."""
    return world * steps * L * B * H * T / (ms_max / 1e3)


def workload_config():
    return {"workload": "fwd+bwd, 16 layers, learned alpha (theta_l ~ N(0,0.5)), Fibonacci K=15",
            "B": B, "H": H, "Hkv": H, "T": T, "D": D, "W": W, "layers": L, "K": K, "seed": SEED,
            "io": "bf16, fp32 accumulate; each layer's RoPE-rotated keys kept from its forward for its backward",
            "l2": "inputs larger than L2: distinct per-layer buffers, 1.07 GB of inputs per step"}


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as fh:
            p = json.load(fh)
        return float(p["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


# ------------------------------------------------------------------ clocks --

class ClockSampler:
    """nvidia-smi clock/throttle sampling during the timed region."""
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []
        self.t0 = self.t1 = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append((time.time(), line.strip()))

    def mark(self, which):
        setattr(self, which, time.time())

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = []
        for ts, line in self.lines:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            rows.append((ts, parts))
        inside = [r for ts, r in rows if self.t0 and self.t1 and self.t0 - 0.15 <= ts <= self.t1 + 0.15] or \
            [r for _, r in rows]
        if not inside:
            return None

        def num(x):
            try:
                return float(x)
            except ValueError:
                return None

        sm = [num(r[1]) for r in inside if num(r[1]) is not None]
        mx = [num(r[2]) for r in inside if num(r[2]) is not None]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in inside for i in range(4) if r[5 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(inside)}


# ------------------------------------------------------------ GPU workload --

class Workload:
    def __init__(self, device, seed_base=SEED, layers=L):
        import paper_2606_28560_gb300 as fa
        from paper_2606_28560_gb300 import inputs
        self.fa = fa
        self.dev = device
        self.L = layers
        theta = inputs.theta_learned(L, seed=SEED)
        self.alphas = [float(a) for a in fa.alpha_schedule("learned", L, theta=theta)]
        self.f = fa.base("fib", K)
        shp = (B, H, T, D)
        bf = torch.bfloat16
        self.q, self.k, self.v, self.g = [], [], [], []
        for l in range(layers):
            s = inputs.layer_seed(seed_base, l)
            ts = [torch.empty(shp, dtype=bf, device=device) for _ in range(4)]
            for j, t in enumerate(ts):
                inputs.device_normal_(t, s * 10 + j)
            self.q.append(ts[0]); self.k.append(ts[1]); self.v.append(ts[2]); self.g.append(ts[3])
        self.out = [torch.empty(shp, dtype=bf, device=device) for _ in range(layers)]
        # rotated keys of each layer, written by its forward and read by its backward
        self.rk = [torch.empty(shp, dtype=torch.float16, device=device) for _ in range(layers)]
        # forward residuals of each layer (rotated q, p per slot, rung score
        # differences), read by its backward instead of recomputing the scores
        self.res = [torch.empty(fa.residual_bytes(B, H, T, W, K, bf), dtype=torch.uint8, device=device)
                    for _ in range(layers)]
        self.use_res = True
        self.lse = [torch.empty((B, H, T), dtype=torch.float32, device=device) for _ in range(layers)]
        self.dq = [torch.empty(shp, dtype=bf, device=device) for _ in range(layers)]
        self.dk = [torch.empty(shp, dtype=bf, device=device) for _ in range(layers)]
        self.dv = [torch.empty(shp, dtype=bf, device=device) for _ in range(layers)]
        self.dth = torch.zeros((layers, 4), dtype=torch.float32, device=device)
        self.dd = torch.zeros((layers, 32), dtype=torch.float32, device=device)
        self.ws_f = torch.empty(fa.fwd_workspace_bytes(B, H, T, W, K, bf), dtype=torch.uint8, device=device)
        self.ws_b = torch.empty(fa.bwd_workspace_bytes(B, H, T, W, K, bf), dtype=torch.uint8, device=device)

    def _res(self, l):
        return self.res[l] if self.use_res else None

    def step(self):
        fa = self.fa
        for l in range(self.L):
            fa.fwd(self.q[l], self.k[l], self.v[l], self.alphas[l], self.f, W, out=self.out[l], lse=self.lse[l],
                   workspace=self.ws_f, rotated_k=self.rk[l], residuals=self._res(l))
        for l in reversed(range(self.L)):
            fa.bwd(self.q[l], self.k[l], self.v[l], self.lse[l], self.g[l], self.alphas[l], self.f, W,
                   out=self.out[l], dq=self.dq[l], dk=self.dk[l], dv=self.dv[l], dtheta=self.dth[l],
                   dd=self.dd[l], workspace=self.ws_b, rotated_k=self.rk[l], residuals=self._res(l))

    def step_fixed(self, rung_grads: bool):
        """The same step at alpha = 1 in every layer (integer rung distances);
        without rung_grads the backward skips dL/dtheta (a fixed schedule)."""
        fa = self.fa
        for l in range(self.L):
            fa.fwd(self.q[l], self.k[l], self.v[l], 1.0, self.f, W, out=self.out[l], lse=self.lse[l],
                   workspace=self.ws_f, rotated_k=self.rk[l], residuals=self._res(l))
        for l in reversed(range(self.L)):
            fa.bwd(self.q[l], self.k[l], self.v[l], self.lse[l], self.g[l], 1.0, self.f, W,
                   out=self.out[l], dq=self.dq[l], dk=self.dk[l], dv=self.dv[l],
                   dtheta=self.dth[l] if rung_grads else None, dd=self.dd[l] if rung_grads else None,
                   workspace=self.ws_b, rotated_k=self.rk[l], rung_grads=rung_grads, residuals=self._res(l))

    def step_static(self, alphas, round_offsets: bool):
        """The same step under a static schedule (no dL/dtheta): rung
        distances interpolated, or rounded to integers (the paper's
        integer-offset variants)."""
        fa = self.fa
        for l in range(self.L):
            fa.fwd(self.q[l], self.k[l], self.v[l], float(alphas[l]), self.f, W, out=self.out[l], lse=self.lse[l],
                   workspace=self.ws_f, rotated_k=self.rk[l], residuals=self._res(l), round_offsets=round_offsets)
        for l in reversed(range(self.L)):
            fa.bwd(self.q[l], self.k[l], self.v[l], self.lse[l], self.g[l], float(alphas[l]), self.f, W,
                   out=self.out[l], dq=self.dq[l], dk=self.dk[l], dv=self.dv[l], workspace=self.ws_b,
                   rotated_k=self.rk[l], rung_grads=False, residuals=self._res(l), round_offsets=round_offsets)

    def fwd_only(self, W_):
        fa = self.fa
        for l in range(self.L):
            fa.fwd(self.q[l], self.k[l], self.v[l], self.alphas[l], self.f, W_, out=self.out[l], lse=self.lse[l],
                   workspace=self.ws_f, rotated_k=self.rk[l])


def method_bytes():
    """Bytes the method itself must move per launch of each kernel (the
    compulsory traffic of the attention, bf16 rows of 128 B, fp32 lse): the
    forward reads Q, K (rotated), V and writes O and lse; the query pass reads
    q, k, v, dO, O and lse and writes dQ; the key pass reads q and dO and
    writes dK and dV.  The RoPE prologue moves no method bytes of its own (its
    key read is the forward's K, counted there)."""
    n = B * H * T
    rows = n * ROW_BYTES
    return {"fwd": 4 * rows + 4 * n, "rope_k": 0,
            "bwd_query_mma": 6 * rows + 4 * n,
            "bwd_key_mma": 4 * rows}


def overhead_bytes():
    """Traffic the design adds on top of the method bytes, per launch: the
    rotated keys written by the prologue and read in place of K; the forward
    residuals (rotated q as bf16 rows, the unnormalised weight of each of the S
    slots, the rung score differences, 1 / row sum) written by the forward and
    read by the backward; dS per slot written by the query pass and, with the
    weights, read by the key pass."""
    n = B * H * T
    S = W + 1 + K
    rows = n * ROW_BYTES
    return {"rope_k": 2 * rows,
            "fwd": rows + 4 * n * S + 4 * n * K + 4 * n,
            "bwd_query_mma": 4 * n * S + 4 * n * K + 4 * n + 4 * n * S,
            "bwd_key_mma": 2 * 4 * n * S + 4 * n}


def step_method_bytes():
    """Per step (16 layers of forward and backward): each tensor once, 512 B
    forward (Q, K, V, O) and 1024 B backward (Q, K, V, O, dO read; dQ, dK, dV
    written) per query-head."""
    return L * B * H * T * (4 + 8) * ROW_BYTES


# DRAM traffic (dram__bytes_read.sum + dram__bytes_write.sum) of one launch,
# from an `ncu --set full` capture of `bench.py --ncu-case bwd` (B=32, the same
# H, T, D, W); every launch reads and writes each of its tensors once, so the
# bytes scale with B.  The counters belong to the sources hashed here (code
# lines only: comments and blank lines are left out): once the code of a file
# of the kernel changes, the figure is reported as null until the next capture.
NCU_TRAFFIC = {
    "bwd_query_mma": {"bytes_at_b32": 165826304 + 34677504,
                      "sources": ("bwd_mma.cu", "mma_common.cuh", "fwd_mma.cuh", "fibattn_internal.cuh"),
                      "sha256": "7a6eb2f7d4feb3df5fe17da5c123412960a0f981820708d5c6c8d90417a9135f"},
    "bwd_key_mma": {"bytes_at_b32": 104474112 + 36588544,
                    "sources": ("bwd_key_mma.cu", "mma_common.cuh", "fwd_mma.cuh", "fibattn_internal.cuh"),
                    "sha256": "4ff4e27482277785ddef47bd09570cc27c9726b314342d7705918d65cdc68e90"},
    "fwd": {"bytes_at_b32": 100786432 + 57735424,
            "sources": ("fwd_mma.cu", "mma_common.cuh", "fwd_mma.cuh", "fibattn_internal.cuh"),
            "sha256": "f5e65c2459e7c5aefee87e45327bf46bd1462355ff93fb85501562b94d5cc0c5"},
}


def sources_sha256(names) -> str:
    """sha256 over the code lines of the named kernel sources (// and /* */
    comments, trailing blanks and empty lines removed; the sources hold no
    string literal with a comment marker)."""
    import hashlib
    import re
    h = hashlib.sha256()
    for n in names:
        with open(os.path.join(ROOT, "paper_2606_28560_gb300", "csrc", n), encoding="utf-8") as fh:
            text = re.sub(r"/\*.*?\*/", "", fh.read(), flags=re.S)
        for line in text.splitlines():
            line = line.split("//", 1)[0].rstrip()
            if line:
                h.update(line.encode() + b"\n")
    return h.hexdigest()


def ncu_traffic(kernel: str):
    """Per-launch DRAM bytes of `kernel` at the bench's B, or None."""
    e = NCU_TRAFFIC.get(kernel)
    if e is None or sources_sha256(e["sources"]) != e["sha256"]:
        return None
    return round(e["bytes_at_b32"] * B / 32)


def capture(fn, device, profile=True):
    """Capture fn() (library launches on torch's current stream) into a CUDA
    graph.  With profile, the library's per-kernel events become event nodes of
    the graph and time every replay; they also sit between the kernels, where
    they keep a kernel from starting during its predecessor's last wave, so the
    headline time comes from a graph captured without them."""
    from paper_2606_28560_gb300.binding import profile_enable
    side = torch.cuda.Stream(device)
    side.wait_stream(torch.cuda.current_stream(device))
    with torch.cuda.stream(side):
        fn()
    torch.cuda.current_stream(device).wait_stream(side)
    torch.cuda.synchronize(device)
    profile_enable(profile)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fn()
    return g


def run_gpu(args, rank, world, device):
    from paper_2606_28560_gb300.binding import profile_enable, profile_summary

    dist = world > 1
    wl = Workload(device)
    stream = torch.cuda.current_stream(device)
    for _ in range(args.warmup):                 # eager warm-up (module load, attributes)
        wl.step()
    torch.cuda.synchronize(device)

    # one step = 16 layers fwd + bwd, captured once (no profiling nodes)
    graph = capture(wl.step, device, profile=False)
    for _ in range(args.warmup):
        graph.replay()
    torch.cuda.synchronize(device)

    def barrier():
        if dist:
            torch.distributed.barrier()

    clocks = ClockSampler(int(os.environ.get("LOCAL_RANK", "0")) if dist else device.index or 0)
    if rank == 0:
        clocks.start()
        time.sleep(0.3)
    barrier()
    torch.cuda.synchronize(device)
    clocks.mark("t0")
    # an event between replays: the whole region and each step's time
    evs = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps + 1)]
    evs[0].record(stream)
    for i in range(args.steps):
        graph.replay()
        evs[i + 1].record(stream)
    torch.cuda.synchronize(device)
    clocks.mark("t1")
    barrier()
    ms = evs[0].elapsed_time(evs[-1])
    step_ms = sorted(evs[i].elapsed_time(evs[i + 1]) for i in range(args.steps))
    clk = clocks.stop() if rank == 0 else None
    # per-kernel device times: the same step captured with the library's event
    # nodes, replayed after the timed region
    gprof = capture(wl.step, device, profile=True)
    for _ in range(max(3, args.warmup)):
        gprof.replay()
    torch.cuda.synchronize(device)
    prof = profile_summary()                     # per kernel: the last replay
    profile_enable(False)
    del gprof
    launches_per_step = sum(v[1] for v in prof.values())

    ms_max = max_over_ranks(ms, device)
    value = job_throughput(world, args.steps, ms_max)

    # roofline of the dominant kernel (largest share of device time), on the
    # method's bytes; the design's extra traffic is reported beside it
    hbm, peak_kind = peaks()
    algo = method_bytes()
    over = overhead_bytes()
    tot = sum(v[0] for v in prof.values()) or 1.0
    dom = max(prof.items(), key=lambda kv: kv[1][0])[0] if prof else "fwd"
    dms, dcnt = prof.get(dom, (0.0, 1))
    avg_s = dms / max(dcnt, 1) / 1e3
    achieved = algo.get(dom, 0) / avg_s / 1e9 if avg_s > 0 else 0.0

    def per_launch_s(v):
        return v[0] / max(v[1], 1) / 1e3

    kernels = {k: {"ms_per_step": round(v[0], 4), "launches_per_step": v[1], "share": round(v[0] / tot, 4),
                   "us_per_launch": round(v[0] / max(v[1], 1) * 1e3, 2),
                   "method_bytes_per_launch": algo.get(k, 0), "overhead_bytes_per_launch": over.get(k, 0),
                   "method_GBps": round(algo.get(k, 0) / per_launch_s(v) / 1e9, 1) if v[0] > 0 else None,
                   "method_frac_of_hbm": round(algo.get(k, 0) / per_launch_s(v) / 1e9 / hbm, 4) if v[0] > 0 else None,
                   "with_overhead_GBps": round((algo.get(k, 0) + over.get(k, 0)) / per_launch_s(v) / 1e9, 1)
                   if v[0] > 0 else None}
               for k, v in prof.items()}

    # forward only at the same shape (W sweep): layer time from a graph without
    # profiling nodes, the forward kernel's time from a profiled capture
    fwd_sweep = {}
    for W_ in (6, 8, 10, 12):
        wl.fwd_only(W_)
        torch.cuda.synchronize(device)
        gf = capture(lambda: wl.fwd_only(W_), device, profile=False)
        for _ in range(2):
            gf.replay()
        a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        reps = max(3, args.steps // 4)
        a0.record(stream)
        for _ in range(reps):
            gf.replay()
        a1.record(stream)
        torch.cuda.synchronize(device)
        layer_us = a0.elapsed_time(a1) / (reps * L) * 1e3
        del gf
        gp = capture(lambda: wl.fwd_only(W_), device, profile=True)
        for _ in range(2):
            gp.replay()
        torch.cuda.synchronize(device)
        p = profile_summary()
        profile_enable(False)
        del gp
        fms, fcnt = p.get("fwd", (0.0, 1))
        us = fms / max(fcnt, 1) * 1e3
        cbytes = 4 * B * H * T * ROW_BYTES
        fwd_sweep[f"W{W_}"] = {"fwd_kernel_us": round(us, 2), "layer_us_incl_rope": round(layer_us, 2),
                               "compulsory_GBps": round(cbytes / (layer_us * 1e-6) / 1e9, 1),
                               "frac_of_hbm": round(cbytes / (layer_us * 1e-6) / 1e9 / hbm, 4),
                               "fwd_kernel_frac_of_hbm": round(cbytes / (us * 1e-6) / 1e9 / hbm, 4)}

    # the integer path: alpha = 1 in every layer, with and without dL/dtheta
    integer = {}
    for name, rg in (("alpha1_with_dtheta", True), ("alpha1_no_dtheta", False)):
        gi = capture(lambda: wl.step_fixed(rg), device, profile=False)
        for _ in range(2):
            gi.replay()
        a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        reps = max(3, args.steps // 3)
        a0.record(stream)
        for _ in range(reps):
            gi.replay()
        a1.record(stream)
        torch.cuda.synchronize(device)
        integer[name] = {"ms_per_step": round(a0.elapsed_time(a1) / reps, 4)}
        del gi
    lin = wl.fa.alpha_schedule("linear", L)
    for name, rnd in (("linear_rounded_no_dtheta", True), ("linear_interpolated_no_dtheta", False)):
        gi = capture(lambda: wl.step_static(lin, rnd), device, profile=False)
        for _ in range(2):
            gi.replay()
        a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        reps = max(3, args.steps // 3)
        a0.record(stream)
        for _ in range(reps):
            gi.replay()
        a1.record(stream)
        torch.cuda.synchronize(device)
        integer[name] = {"ms_per_step": round(a0.elapsed_time(a1) / reps, 4)}
        del gi
    integer["linear_interpolated_over_rounded"] = round(integer["linear_interpolated_no_dtheta"]["ms_per_step"] /
                                                        integer["linear_rounded_no_dtheta"]["ms_per_step"], 3)
    integer["learned_alpha_ms_per_step"] = round(ms_max / args.steps, 4)
    integer["interpolated_over_integer"] = round(integer["learned_alpha_ms_per_step"] /
                                                 integer["alpha1_with_dtheta"]["ms_per_step"], 3)

    # the same step with a backward that recomputes the scores (no residuals)
    wl.use_res = False
    gr = capture(wl.step, device, profile=False)
    for _ in range(2):
        gr.replay()
    a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    reps = max(3, args.steps // 3)
    a0.record(stream)
    for _ in range(reps):
        gr.replay()
    a1.record(stream)
    torch.cuda.synchronize(device)
    wl.use_res = True
    del gr
    recompute = {"ms_per_step": round(a0.elapsed_time(a1) / reps, 4),
                 "residuals_ms_per_step": round(ms_max / args.steps, 4)}
    recompute["residuals_speedup"] = round(recompute["ms_per_step"] / recompute["residuals_ms_per_step"], 3)

    gqa = run_gqa_forward(wl, device, args, stream)
    configs = run_configs(device, args, stream)
    e2e = run_e2e(args, wl, device, dist)
    stack = run_autograd_stack(device)
    return dict(value=value, ms=ms_max, clk=clk, dom=dom, achieved=achieved, hbm=hbm, peak_kind=peak_kind,
                algo=algo, over=over, kernels=kernels, fwd_sweep=fwd_sweep, e2e=e2e, launches=launches_per_step * args.steps,
                stack=stack, integer=integer, gqa=gqa, configs=configs, recompute=recompute,
                median_ms=step_ms[len(step_ms) // 2], min_ms=step_ms[0], max_ms=step_ms[-1])


def run_gqa_forward(wl, device, args, stream):
    """The 16 layers at the paper's head split (H = 8 query heads, Hkv = 2 kv
    heads), same B, T, W and schedule as the step, graphed: the forward alone
    (groups of 4 query heads share each CTA's staged keys and values) and the
    whole forward + backward step with residuals."""
    import paper_2606_28560_gb300 as fa
    from paper_2606_28560_gb300 import inputs
    Hkv = 2
    kv = []
    for l in range(L):
        k = torch.empty((B, Hkv, T, D), dtype=torch.bfloat16, device=device)
        v = torch.empty((B, Hkv, T, D), dtype=torch.bfloat16, device=device)
        inputs.device_normal_(k, 5000 + 2 * l)
        inputs.device_normal_(v, 5001 + 2 * l)
        kv.append({"k": k, "v": v, "rk": torch.empty((B, Hkv, T, D), dtype=torch.float16, device=device),
                   "dk": torch.empty_like(k), "dv": torch.empty_like(v),
                   "res": fa.residuals_like(wl.q[l], W, K)})
    ws_f = torch.empty(fa.fwd_workspace_bytes(B, H, T, W, K, torch.bfloat16, Hkv=Hkv), dtype=torch.uint8,
                       device=device)
    ws_b = torch.empty(fa.bwd_workspace_bytes(B, H, T, W, K, torch.bfloat16, Hkv=Hkv), dtype=torch.uint8,
                       device=device)

    def fwd_all(res=False):
        for l in range(L):
            c = kv[l]
            fa.fwd(wl.q[l], c["k"], c["v"], wl.alphas[l], wl.f, W, out=wl.out[l], lse=wl.lse[l], workspace=ws_f,
                   rotated_k=c["rk"], residuals=c["res"] if res else None)

    def step():
        fwd_all(True)
        for l in reversed(range(L)):
            c = kv[l]
            fa.bwd(wl.q[l], c["k"], c["v"], wl.lse[l], wl.g[l], wl.alphas[l], wl.f, W, out=wl.out[l],
                   dq=wl.dq[l], dk=c["dk"], dv=c["dv"], dtheta=wl.dth[l], dd=wl.dd[l], workspace=ws_b,
                   rotated_k=c["rk"], residuals=c["res"])

    out = {"B": B, "H": H, "Hkv": Hkv, "T": T, "W": W}
    for name, fn in (("fwd", fwd_all), ("fwd_bwd", step)):
        fn()
        torch.cuda.synchronize(device)
        g = capture(fn, device, profile=False)
        for _ in range(2):
            g.replay()
        a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        reps = max(3, args.steps // 3)
        a0.record(stream)
        for _ in range(reps):
            g.replay()
        a1.record(stream)
        torch.cuda.synchronize(device)
        ms = a0.elapsed_time(a1) / reps
        del g
        if name == "fwd":
            out["layer_us_incl_rope"] = round(ms / L * 1e3, 2)
            out["query_heads_per_s"] = round(B * H * T * L / (ms * 1e-3), 1)
        else:
            out["fwd_bwd_ms_per_step"] = round(ms, 4)
            out["fwd_bwd_query_heads_per_s"] = round(B * H * T * L / (ms * 1e-3), 1)
    del kv
    return out


def run_configs(device, args, stream):
    """The long-sequence workloads, 16 layers of distinct buffers, graphed
    (RoPE of k included): T = 4096 extrapolation (B4 H8 W10, coprime
    stagger), forward alone; T = 16384 stress (B2 H8 W12, linear stagger),
    forward alone and forward + backward with residuals, for the Fibonacci
    (K = 15) and the power-of-2 (K = 10) base."""
    import paper_2606_28560_gb300 as fa
    from paper_2606_28560_gb300 import inputs
    hbm = peaks()[0]
    out = {}
    cases = (("T4096_B4_W10_coprime_fib", 4, 4096, 10, "coprime", "fib", 15, False),
             ("T16384_B2_W12_linear_fib", 2, 16384, 12, "linear", "fib", 15, True),
             ("T16384_B2_W12_linear_pow2", 2, 16384, 12, "linear", "pow2", 10, True))
    for name, Bc, Tc, Wc, sched, base, Kc, bwd in cases:
        alphas = [float(a) for a in fa.alpha_schedule(sched, L)]
        f = fa.base(base, Kc)
        shp = (Bc, H, Tc, D)
        bf = torch.bfloat16
        lay = []
        for l in range(L):
            ts = [torch.empty(shp, dtype=bf, device=device) for _ in range(4)]
            for j, t in enumerate(ts):
                inputs.device_normal_(t, 7000 + 10 * l + j)
            lay.append({"q": ts[0], "k": ts[1], "v": ts[2], "g": ts[3], "o": torch.empty_like(ts[0]),
                        "lse": torch.empty((Bc, H, Tc), dtype=torch.float32, device=device),
                        "rk": torch.empty(shp, dtype=torch.float16, device=device),
                        "res": fa.residuals_like(ts[0], Wc, Kc) if bwd else None,
                        "dq": torch.empty_like(ts[0]), "dk": torch.empty_like(ts[0]), "dv": torch.empty_like(ts[0])})
        ws_f = torch.empty(fa.fwd_workspace_bytes(Bc, H, Tc, Wc, Kc, bf), dtype=torch.uint8, device=device)
        ws_b = torch.empty(fa.bwd_workspace_bytes(Bc, H, Tc, Wc, Kc, bf), dtype=torch.uint8, device=device)
        dth = torch.zeros((L, 4), dtype=torch.float32, device=device)

        def fwd_all(res=False):
            for l, c in enumerate(lay):
                fa.fwd(c["q"], c["k"], c["v"], alphas[l], f, Wc, out=c["o"], lse=c["lse"], workspace=ws_f,
                       rotated_k=c["rk"], residuals=c["res"] if res else None)

        def step():
            fwd_all(True)
            for l in reversed(range(L)):
                c = lay[l]
                fa.bwd(c["q"], c["k"], c["v"], c["lse"], c["g"], alphas[l], f, Wc, out=c["o"], dq=c["dq"],
                       dk=c["dk"], dv=c["dv"], dtheta=dth[l], workspace=ws_b, rotated_k=c["rk"],
                       residuals=c["res"])

        r = {"B": Bc, "H": H, "T": Tc, "W": Wc, "K": Kc, "schedule": sched, "base": base}
        for what, fn in (("fwd", fwd_all), ("fwd_bwd", step)) if bwd else (("fwd", fwd_all),):
            fn()
            torch.cuda.synchronize(device)
            g = capture(fn, device, profile=False)
            g.replay()
            a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            reps = 3
            a0.record(stream)
            for _ in range(reps):
                g.replay()
            a1.record(stream)
            torch.cuda.synchronize(device)
            ms = a0.elapsed_time(a1) / reps
            del g
            qh = Bc * H * Tc * L
            if what == "fwd":
                r["fwd_layer_us_incl_rope"] = round(ms / L * 1e3, 2)
                r["fwd_query_heads_per_s"] = round(qh / (ms * 1e-3), 1)
                r["fwd_frac_of_hbm"] = round(qh * 4 * ROW_BYTES / (ms * 1e-3) / 1e9 / hbm, 4)
            else:
                r["fwd_bwd_ms_per_step"] = round(ms, 4)
                r["fwd_bwd_query_heads_per_s"] = round(qh / (ms * 1e-3), 1)
                r["step_frac_of_hbm"] = round(qh * 12 * ROW_BYTES / (ms * 1e-3) / 1e9 / hbm, 4)
        out[name] = r
        del lay, ws_f, ws_b
        torch.cuda.empty_cache()
    return out


def run_autograd_stack(device, warm=2, reps=3):
    """A 16-layer attention stack (q = k = v = the previous output, no
    projections) through the torch.autograd wrapper, forward and backward of
    L = sum(out), per alpha schedule, at T = 1024 (B16) and T = 4096 (B4):
    eager steps, Python and autograd included."""
    import paper_2606_28560_gb300 as fa
    from paper_2606_28560_gb300 import inputs
    f = fa.base("fib", K)
    res = {}
    for Bs, Ts in ((16, 1024), (4, 4096)):
        x = torch.empty((Bs, H, Ts, D), dtype=torch.bfloat16, device=device)
        inputs.device_normal_(x, 77)
        x.requires_grad_(True)
        for kind in ("fixed", "linear", "coprime", "learned"):
            th = inputs.theta_learned(L, seed=SEED) if kind == "learned" else None
            alphas = fa.alpha_schedule(kind, L, theta=th)
            layers = [fa.FibAttention(W=W, offsets=f, theta=fa.theta_of_alpha(float(a)),
                                      learned=(kind == "learned")).to(device) for a in alphas]

            def step():
                out = fa.attention_stack(x, layers)
                out.float().sum().backward()
                x.grad = None

            for _ in range(warm):
                step()
            torch.cuda.synchronize(device)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(reps):
                step()
            e1.record()
            torch.cuda.synchronize(device)
            ms = e0.elapsed_time(e1) / reps
            res[f"T{Ts}_B{Bs}_{kind}"] = {"ms_per_step": round(ms, 3),
                                          "query_heads_per_s": round(Bs * H * Ts * L / (ms * 1e-3), 1)}
        del x
    return res


def run_e2e(args, wl, device, dist):
    """Same step through the public API with host buffers: every step copies
    its inputs (q, k, v, dout of all layers) from pinned host memory and reads
    the results (out, dq, dk, dv, dtheta of all layers) back to pinned host
    memory, inside the timed region.  The copies run on two copy streams and
    overlap the compute: a layer's forward waits only for its own q, k, v,
    its backward for its own dout, and each result goes back as soon as the
    layer that produced it is done.  The device inputs are double-buffered by
    step, as a prefetching loader would: step s + 1's inputs stream in while
    step s's gradients stream out, so both directions of the link stay busy.
    Every buffer is reused only after the work that last read or wrote it
    (per-layer events)."""
    fa = wl.fa
    n_in = 4 * L
    host_in = [torch.empty((B, H, T, D), dtype=torch.bfloat16, pin_memory=True) for _ in range(n_in)]
    for i, h in enumerate(host_in):
        src = (wl.q, wl.k, wl.v, wl.g)[i % 4][i // 4]
        h.copy_(src)
    host_out = [torch.empty((B, H, T, D), dtype=torch.bfloat16, pin_memory=True) for _ in range(4 * L)]
    host_th = torch.empty((L, 4), dtype=torch.float32, pin_memory=True)
    # input sets by step parity: the workload's own buffers and a second copy
    sets = [(wl.q, wl.k, wl.v, wl.g),
            tuple([torch.empty_like(x) for x in t] for t in (wl.q, wl.k, wl.v, wl.g))]
    # compute on a stream of its own: work on the legacy default stream would
    # serialise with the copy streams
    comp, s_in, s_out = torch.cuda.Stream(device), torch.cuda.Stream(device), torch.cuda.Stream(device)
    ev_in = [[torch.cuda.Event() for _ in range(L)] for _ in range(2)]    # q, k, v of layer l on the device
    ev_g = [[torch.cuda.Event() for _ in range(L)] for _ in range(2)]     # dout of layer l on the device
    ev_b = [[torch.cuda.Event() for _ in range(L)] for _ in range(2)]     # backward of layer l done (set free)
    ev_f = [torch.cuda.Event() for _ in range(L)]            # forward of layer l done
    ev_bo = [torch.cuda.Event() for _ in range(L)]           # backward of layer l done (outputs ready)
    ev_oc = [torch.cuda.Event() for _ in range(L)]           # out of layer l read back
    ev_gc = [torch.cuda.Event() for _ in range(L)]           # dq, dk, dv of layer l read back
    ev_th = torch.cuda.Event()                               # dtheta read back
    steps = max(2, min(args.steps, 20))
    state = {"step": 0}

    def one():
        p = state["step"] % 2
        state["step"] += 1
        q, k, v, g = sets[p]
        with torch.cuda.stream(s_in):
            for l in range(L):
                s_in.wait_event(ev_b[p][l])      # the step before last is done with this set
                for j, dst in enumerate((q, k, v)):
                    dst[l].copy_(host_in[4 * l + j], non_blocking=True)
                ev_in[p][l].record(s_in)
            for l in reversed(range(L)):
                g[l].copy_(host_in[4 * l + 3], non_blocking=True)
                ev_g[p][l].record(s_in)
        for l in range(L):
            comp.wait_event(ev_in[p][l])
            comp.wait_event(ev_oc[l])            # the previous step's out of this layer is on the host
            fa.fwd(q[l], k[l], v[l], wl.alphas[l], wl.f, W, out=wl.out[l], lse=wl.lse[l],
                   workspace=wl.ws_f, rotated_k=wl.rk[l], residuals=wl.res[l], stream=comp)
            ev_f[l].record(comp)
            s_out.wait_event(ev_f[l])
            with torch.cuda.stream(s_out):
                host_out[4 * l].copy_(wl.out[l], non_blocking=True)
                ev_oc[l].record(s_out)
        comp.wait_event(ev_th)                   # the previous step's dtheta is on the host
        for l in reversed(range(L)):
            comp.wait_event(ev_g[p][l])
            comp.wait_event(ev_gc[l])            # the previous step's gradients of this layer are on the host
            fa.bwd(q[l], k[l], v[l], wl.lse[l], g[l], wl.alphas[l], wl.f, W, out=wl.out[l],
                   dq=wl.dq[l], dk=wl.dk[l], dv=wl.dv[l], dtheta=wl.dth[l], dd=wl.dd[l], workspace=wl.ws_b,
                   rotated_k=wl.rk[l], residuals=wl.res[l], stream=comp)
            ev_b[p][l].record(comp)
            ev_bo[l].record(comp)
            s_out.wait_event(ev_bo[l])
            with torch.cuda.stream(s_out):
                for j, src in enumerate((wl.dq, wl.dk, wl.dv)):
                    host_out[4 * l + 1 + j].copy_(src[l], non_blocking=True)
                ev_gc[l].record(s_out)
        with torch.cuda.stream(s_out):
            host_th.copy_(wl.dth, non_blocking=True)
            ev_th.record(s_out)

    with torch.cuda.stream(comp):
        one()
        one()
        torch.cuda.synchronize(device)
        if dist:
            torch.distributed.barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(comp)
        s_in.wait_stream(comp)                   # the first timed copies start after e0
        s_out.wait_stream(comp)
        # per step: when its last result (dtheta) is on the host
        done = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
        for i in range(steps):
            one()
            done[i].record(s_out)
        comp.wait_stream(s_out)                  # the last step ends when its results are on the host
        comp.wait_stream(s_in)
        e1.record(comp)
        torch.cuda.synchronize(device)
    ms = max_over_ranks(e0.elapsed_time(e1), device)
    gaps = sorted(done[i].elapsed_time(done[i + 1]) for i in range(steps - 1))
    world = torch.distributed.get_world_size() if dist else 1
    value = job_throughput(world, steps, ms)
    bi = n_in * B * H * T * ROW_BYTES
    bo = 4 * L * B * H * T * ROW_BYTES + L * 4 * 4
    ok = all(torch.equal(host_out[4 * l + 1].to(device), wl.dq[l]) for l in (0, L - 1))
    return {"value": value, "unit": UNIT, "h2d_bytes_per_step": bi, "d2h_bytes_per_step": bo,
            "ms_per_step": round(ms / steps, 4), "results_on_host_match": ok,
            "step_gap_ms": {"min": round(gaps[0], 4), "median": round(gaps[len(gaps) // 2], 4),
                            "max": round(gaps[-1], 4)},
            "copies": "two copy streams overlapping the compute; device inputs double-buffered by step "
                      "(the next step's inputs stream in while this step's gradients stream out); per-layer events"}


# ------------------------------------------------------------- CPU oracle --

def oracle_sample(seconds_target=10.0, nthreads=None):
    """Time the fp64 oracle (as it stands) on a bounded sample of the
    workload: fwd + bwd of whole layers (B=16, H=8, T=1024 each), layer after
    layer, until about ``seconds_target`` of wall time has been spent."""
    import oracle as O
    from paper_2606_28560_gb300 import inputs
    nthreads = nthreads or (os.cpu_count() or 1)
    theta = inputs.theta_learned(L, seed=SEED)
    alphas = O.alpha_schedule("learned", L, theta=theta)
    f = O.fib_base(K)
    done_q, spent, layers = 0, 0.0, 0
    while spent < seconds_target and layers < L:
        s = inputs.layer_seed(SEED, layers)
        q, k, v = inputs.qkv(B, H, T, seed=s, dtype=torch.bfloat16)
        g = inputs.dout(B, H, T, seed=s, dtype=torch.bfloat16)
        q, k, v, g = (x.double().numpy() for x in (q, k, v, g))
        d = O.offsets_fp32(float(np.float32(alphas[layers])), f)
        t0 = time.perf_counter()
        O.forward(q, k, v, W, d, nthreads=nthreads)
        O.backward(q, k, v, g, W, d, nthreads=nthreads)
        spent += time.perf_counter() - t0
        done_q += B * H * T
        layers += 1
    return {"value": done_q / spent, "unit": UNIT, "cores": nthreads, "kind": "oracle",
            "sample": f"{layers} full layer(s) fwd+bwd (B=16 H=8 T=1024 each, {done_q} query-heads), "
                      f"fp64 C oracle, {spent:.1f} s wall on {nthreads} threads"}


def cpu_model() -> str:
    """The host CPU's model line (lscpu, else /proc/cpuinfo, else the machine type)."""
    import platform
    import subprocess
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.lower().startswith("model name"):
                return line.split(":", 1)[1].strip()
    except (OSError, subprocess.SubprocessError):
        pass
    try:
        with open("/proc/cpuinfo") as fh:
            for line in fh:
                if line.lower().startswith("model name"):
                    return line.split(":", 1)[1].strip()
    except OSError:
        pass
    return platform.machine()


def oracle_per_config():
    """The fp64 oracle, as it stands, on one full layer of each measured
    configuration, single-threaded and on all host cores: config 2 forward
    (B16 H8 T1024 W8, linear schedule, layer 7), config 3 forward (B4 H8 T4096
    W10, coprime schedule, layer 1), config 4 forward + backward (B16 H8 T1024
    W8, learned schedule, layer 0).  Seconds per layer and query-heads/s."""
    import oracle as O
    from paper_2606_28560_gb300 import inputs
    nall = os.cpu_count() or 1
    f = O.fib_base(K)
    cases = [("config2_fwd_W8", 16, 1024, 8, float(O.alpha_schedule("linear", L)[7]), False, 1),
             ("config3_fwd_W10", 4, 4096, 10, float(O.alpha_schedule("coprime", L, stride=7)[1]), False, 2),
             ("config4_fwd_bwd_W8", 16, 1024, 8,
              float(O.alpha_schedule("learned", L, theta=inputs.theta_learned(L, seed=SEED))[0]), True, SEED)]
    out = {"cpu_model": cpu_model(), "host_threads": nall}
    for name, Bc, Tc, Wc, alpha, bwd, seed in cases:
        q, k, v = inputs.qkv(Bc, H, Tc, seed=seed, dtype=torch.bfloat16)
        g = inputs.dout(Bc, H, Tc, seed=seed + 100, dtype=torch.bfloat16)
        q, k, v, g = (x.double().numpy() for x in (q, k, v, g))
        d = O.offsets_fp32(float(np.float32(alpha)), f)
        O.forward(q, k, v, Wc, d, nthreads=nall)          # untimed: first-touch of the oracle's buffers
        row = {}
        for nt in sorted({1, nall}):
            t0 = time.perf_counter()
            O.forward(q, k, v, Wc, d, nthreads=nt)
            if bwd:
                O.backward(q, k, v, g, Wc, d, nthreads=nt)
            dt = time.perf_counter() - t0
            row[f"threads_{nt}"] = {"s_per_layer": round(dt, 3), "query_heads_per_s": round(Bc * H * Tc / dt, 1)}
        out[name] = row
    return out


def run_reference(args, rank, world):
    """Reference arm: the fp64 CPU oracle, timed as it stands on the host
    cores; each step is a bounded sample (one layer fwd+bwd or part of one)."""
    if rank != 0:
        return
    nthreads = os.cpu_count() or 1
    per_step = []
    budget = max(1.0, 60.0 / max(args.steps + args.warmup, 1))
    for i in range(args.warmup + args.steps):
        r = oracle_sample(seconds_target=budget, nthreads=nthreads)
        if i >= args.warmup:
            per_step.append(r["value"])
    value = statistics.median(per_step)
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic N(0,1), seeded",
            "config": workload_config(),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": nthreads, "kind": "oracle",
                             "sample": r["sample"] + " (per step)"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ------------------------------------------------------------- ncu cases --

def ncu_case(which: str):
    """A small fixed case for ncu captures of one kernel: B=32 H=8 T=1024 W=8,
    two layers of distinct buffers (Q, K, V, O of one layer = 134 MB, larger
    than L2), one forward (and backward) per layer after one warm-up pass, the
    path the bench times: the forward keeps its rotated keys and residuals,
    the backward reads them (per layer and pass: RoPE of k, forward, query
    pass, key pass).  `fwd_plain`: the forward alone without residuals (the
    forward-only workload, alpha 0.9 in both layers).  `fp32`: forward and
    backward with fp32 I/O (the row-gather kernels), B=16, alpha 0.9 (the same
    bytes a layer)."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_28560_gb300 as fa
    from paper_2606_28560_gb300 import inputs
    dev = torch.device("cuda", 0)
    fp32 = which == "fp32"
    Bc, layers = 16 if fp32 else 32, 2
    dtype = torch.float32 if fp32 else torch.bfloat16
    f = fa.base("fib", K)
    bufs = []
    for l in range(layers):
        ts = [torch.empty((Bc, H, T, D), dtype=dtype, device=dev) for _ in range(4)]
        for j, t in enumerate(ts):
            inputs.device_normal_(t, 1000 + 10 * l + j)
        bufs.append(ts + [None if fp32 else fa.residuals_like(ts[0], W, K), fa.rotated_k_like(ts[1])])
    for rep in range(2):
        for l, (q, k, v, g, res, rk) in enumerate(bufs):
            if which == "fwd_plain":
                fa.fwd(q, k, v, 0.9, f, W, rotated_k=rk)
                continue
            alpha = 0.9 if fp32 else 0.8 + 0.1 * l
            out, lse = fa.fwd(q, k, v, alpha, f, W, residuals=res, rotated_k=rk)
            if which != "fwd":
                fa.bwd(q, k, v, lse, g, alpha, f, W, out=out, residuals=res, rotated_k=rk)
    torch.cuda.synchronize(dev)
    print(f"ncu case {which} done")


# -------------------------------------------------------------------- main --

def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--ncu-case", choices=["fwd", "fwd_plain", "bwd", "fp32"], default=None,
                    help="run a small fixed case for an ncu capture and exit")
    args = ap.parse_args()
    if args.ncu_case:
        ncu_case(args.ncu_case)
        return

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))

    if args.impl == "reference":
        run_reference(args, rank, world)
        return

    import __graft_entry__
    __graft_entry__.build()
    device = torch.device("cuda", local)
    torch.cuda.set_device(device)
    if world > 1:
        torch.distributed.init_process_group("nccl", device_id=device)
    if args.warmup < 3:
        args.warmup = 3
    r = run_gpu(args, rank, world, device)
    if rank == 0:
        cpu = None
        cpu_configs = None
        if not args.no_cpu_baseline and world == 1:
            cpu = oracle_sample(seconds_target=10.0)
            cpu_configs = oracle_per_config()
        line = {
            "metric": METRIC, "value": r["value"], "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": r["ms"] / args.steps,
            "step_ms": {"median": round(r["median_ms"], 4), "min": round(r["min_ms"], 4),
                        "max": round(r["max_ms"], 4), "median_per_layer_us": round(r["median_ms"] / L * 1e3, 2)},
            "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic N(0,1), seeded",
            "config": workload_config(),
            "timing": "CUDA graph of one step (16 layers fwd+bwd, programmatic dependent launches) replayed; "
                      "per-kernel times from a second capture of the step with event nodes around each kernel",
            "roofline": {"bound": "hbm", "kernel": r["dom"], "achieved": round(r["achieved"], 1),
                         "peak": r["hbm"], "unit": "GB/s", "frac": round(r["achieved"] / r["hbm"], 4),
                         "traffic": ncu_traffic(r["dom"]), "peak_source": r["peak_kind"],
                         "algorithmic_bytes_per_launch": r["algo"].get(r["dom"]),
                         "overhead_bytes_per_launch": r["over"].get(r["dom"]),
                         "step": {"method_bytes": step_method_bytes(),
                                  "achieved": round(step_method_bytes() / (r["ms"] / args.steps / 1e3) / 1e9, 1),
                                  "frac": round(step_method_bytes() / (r["ms"] / args.steps / 1e3) / 1e9 / r["hbm"],
                                                4)}},
            "kernels": r["kernels"],
            "forward_only_B16H8T1024": r["fwd_sweep"],
            "autograd_stack_16_layers": r["stack"],
            "integer_vs_interpolated_16_layers": r["integer"],
            "backward_recomputing_scores_16_layers": r["recompute"],
            "forward_gqa_16_layers": r["gqa"],
            "long_sequence_16_layers": r["configs"],
            "cpu_baseline": cpu,
            "cpu_oracle_per_config": cpu_configs,
            "e2e": r["e2e"],
            "gpu_launches": r["launches"],
            "clocks": r["clk"],
        }
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()

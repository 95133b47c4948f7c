"""Benchmark of the HeteroFold transfer hot path on GB300.

A step is one pass of the whole path over one batch: alignment CSR
(hf_align_build), plan metadata (hf_plan_create), the fused map
(hf_transfer).  Default workload: the 32K-receiver-token Llama-3.1-8B-shaped
-> Ministral-shaped transfer (Token Alignment + three-layer neighbourhood,
bf16 caches and maps, fp32 accumulation).

Prints one JSON line (rank 0).  --impl reference times the fp64 CPU oracle
on a bounded sample of the same workload instead.
"""

from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "transferred receiver-KV tokens/sec and µs per 32K transfer; % of roofline"
UNIT = "receiver tokens/s"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="llama_to_ministral_32k")
    ap.add_argument("--e2e-steps", type=int, default=7)
    ap.add_argument("--e2e-groups", type=int, default=0,
                    help="receiver-layer groups of hf_transfer_host (0: library default)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=15.0)
    ap.add_argument("--round-built-operands", action="store_true",
                    help="computed operand rows rounded once to bf16 (no value + residual pair)")
    ap.add_argument("--graph", action="store_true",
                    help="replay the step as CUDA graphs (alignment + plan, transfer) recorded "
                         "once before the timed steps")
    ap.add_argument("--pool-before-map", action="store_true",
                    help="overlap mean pooling before the map (pooled operand rows per distinct "
                         "row) instead of pooling the mapped sender rows")
    return ap.parse_args()


# Workload name suffixes that switch the alignment or layer rule of a base
# workload: "_overlap" (overlap mean pooling), "_interp" (two-layer
# interpolation); e.g. llama_to_ministral_32k_overlap_interp.
MODE_SUFFIXES = {"_overlap": {"align_mode": "overlap_mean"}, "_interp": {"layer_mode": "interp"}}


def workload(name):
    from paper_2609_32259_gb300 import workloads as W
    mods = {}
    stripped = True
    while stripped:
        stripped = False
        for suf, kw in MODE_SUFFIXES.items():
            if name.endswith(suf):
                name = name[: -len(suf)]
                mods.update(kw)
                stripped = True
    table = {
        "llama_to_ministral_32k": lambda: W.llama_to_ministral(32768),
        "llama_to_qwen25_4k": lambda: W.llama_to_qwen25(4096),
        "qwen25_to_llama_batched_paged": W.qwen25_to_llama_batched,
        "qwen25_to_llama_kv_ridge_4k": lambda: W.qwen25_to_llama_kv_ridge(4096),
        "tiny": W.tiny,
    }
    w = None
    for prefix, make in (("ministral_to_llama_", W.ministral_to_llama),
                         ("llama_to_ministral_", W.llama_to_ministral),
                         ("llama_to_qwen25_", W.llama_to_qwen25),
                         ("qwen25_to_llama_kv_ridge_", W.qwen25_to_llama_kv_ridge)):
        if name.startswith(prefix) and name[len(prefix):].isdigit():
            w = make(int(name[len(prefix):]))
    if w is None:
        w = table[name]()
    if mods:
        tag = "".join(f"_{mods[k]}" for k in ("align_mode", "layer_mode") if k in mods)
        w = w.with_(name=w.name + tag, **mods)
    return w


def aggregate(times_ms, T_r_per_rank, world):
    """Max over ranks of each time (ms); whole-job throughput = all ranks'
    receiver tokens / the slowest rank's step time."""
    times = list(times_ms)
    if world > 1:
        import torch
        import torch.distributed as dist
        dev = torch.device("cuda", torch.cuda.current_device()) if (
            dist.get_backend() == "nccl") else torch.device("cpu")
        t = torch.tensor(times, dtype=torch.float64, device=dev)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        times = [float(x) for x in t.cpu()]
    value = world * T_r_per_rank / (times[0] * 1e-3)
    return value, times


def peaks():
    """(HBM GB/s, bf16 TFLOP/s burst, bf16 TFLOP/s sustained, source)."""
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return (float(p["hbm_gbs"]), float(p["bf16_tflops"]),
                float(p.get("bf16_tflops_sustained", p["bf16_tflops"])), "measured")
    return 6800.0, 1900.0, 1700.0, "fallback"


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------
class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.proc = None
        self.gpu = gpu_index

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.QUERY}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except (FileNotFoundError, OSError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, mx, pw, reasons = [], [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            try:
                pw.append(float(f[3]))
            except ValueError:
                pass
            for n, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_min_mhz": min(sm), "sm_max_mhz": max(mx),
                "power_w_median": statistics.median(pw) if pw else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def kernel_sources_sha256():
    """Hash of the transfer kernel's sources (invalidates stored counters)."""
    import hashlib
    h = hashlib.sha256()
    for name in ("hf_transfer.cu", "hf_device.cuh"):
        with open(os.path.join(ROOT, "paper_2609_32259_gb300", "csrc", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()


# ---------------------------------------------------------------------------
# algorithmic work of one transfer
# ---------------------------------------------------------------------------
def algorithmic_work(w, tok, U, n_distinct_cols):
    """FLOPs and bytes a transfer cannot avoid.

    FLOP: 2 * (2 L_r) * min(U, S) * K * d_r, U = distinct alignment rows
    (rows with identical inputs share one map output before RoPE), S = the
    sender tokens the alignment references: the map is linear, so the
    pooling can come before it (U rows) or after it (S rows), whichever is
    fewer.
    Bytes: the receiver cache written once; every referenced sender row read
    once per sender layer (the three-layer neighbourhoods of these depth
    pairs touch every sender layer); the maps and biases read once; the CSR
    and per-row metadata."""
    e = 2 if w.dtype == "bf16" else 4
    flops = 2.0 * 2 * w.L_r * min(U, n_distinct_cols) * w.K * w.d_r
    T_r = tok.T_r
    # sender layers the layer table reads (all of them for Eq. 1 and the
    # interpolation on these depth pairs; the selected ones for an explicit table)
    n_layers = (len({t for seg_l in w.seg_layer for seg in seg_l for t in seg})
                if w.layer_mode == "explicit" else w.L_s)
    bytes_ = (2 * w.L_r * T_r * w.d_r * e            # receiver cache
              + n_layers * 2 * n_distinct_cols * w.d_s * e  # sender rows
              + 2 * w.L_r * w.K * w.d_r * e          # maps
              + 2 * w.L_r * w.d_r * 4                # bias
              + T_r * 4 * 6)                         # CSR + run / position / row metadata
    return flops, float(bytes_)


# ---------------------------------------------------------------------------
# the oracle on host cores (cpu_baseline and --impl reference)
# ---------------------------------------------------------------------------
class OracleSample:
    """A contiguous block of receiver rows of the workload, all layers and
    roles, with everything the oracle needs already in host memory."""

    def __init__(self, w, tok, sender, Wm, b, r, n_rows, start=None):
        import numpy as np
        from oracle import heterofold_oracle as O
        self.O = O
        csr = O.alignment_csr(w.align_mode, tok.s_tok_ptr, tok.r_tok_ptr, tok.s_end, tok.r_end)
        T = tok.T_r
        n_rows = max(1, min(n_rows, T))
        j0 = (T - n_rows) // 2 if start is None else start
        rows = np.arange(j0, j0 + n_rows)
        e0, e1 = int(csr.row_ptr[j0]), int(csr.row_ptr[j0 + n_rows])
        cols = csr.col[e0:e1]
        c_lo, c_hi = int(cols.min()), int(cols.max()) + 1
        self.csr = O.CSR(csr.row_ptr[j0:j0 + n_rows + 1] - e0, cols - c_lo, csr.w[e0:e1])
        self.sender = sender[:, :, c_lo:c_hi].float().cpu().numpy()
        self.A = Wm.float().cpu().numpy().transpose(0, 1, 3, 2)
        self.b = b.cpu().numpy()
        self.r = r
        if w.layer_mode == "explicit":
            self.segs = O.explicit_segments(w.seg_layer, np.asarray(w.seg_w, np.float32))
        else:
            self.segs = O.layer_segments(w.layer_mode, w.L_s, w.L_r)
        self.pos = O.receiver_positions(tok.r_tok_ptr)[j0:j0 + n_rows]
        self.inv = O.rope_inv_freq(w.theta_r, w.D_r)
        self.w = w
        self.n_rows = n_rows

    def run(self):
        w = self.w
        if w.kv_ridge:  # the per-head maps of the KV Ridge apply
            sel = [[t[0] for t in seg] for seg in w.seg_layer]
            Wh = [[[self.A[l][c][:, h * w.D_r:(h + 1) * w.D_r] for h in range(w.H_r)]
                   for c in range(2)] for l in range(w.L_r)]
            bh = self.b.reshape(w.L_r, 2, w.H_r, w.D_r)
            return self.O.kv_ridge_transfer(self.sender, self.csr, sel, Wh, bh, H_r=w.H_r,
                                            D_r=w.D_r, pos=self.pos, inv_freq_r=self.inv)
        return self.O.transfer(self.sender, self.csr, self.segs, self.A, self.b, self.r,
                               H_r=w.H_r, D_r=w.D_r, pos=self.pos, inv_freq_r=self.inv)


def _pool_after_map(w, pool_before_map=False):
    """Overlap mean pooling applied to the mapped sender rows (the library's
    choice unless the caller asks otherwise or the pooled row itself is
    needed: key norm, sender keys rotated back per position)."""
    return (w.align_mode == "overlap_mean" and not pool_before_map and not w.knorm
            and not w.sender_k_rotated)


def launches_per_step(w, pool_before_map=False):
    """Kernel launches of one hf_align_build + hf_plan_create + hf_transfer on
    texts past 32,768 tokens or 64 requests (step_launches: any text):
    alignment (TA: sender check, match, max-scan; same-index: one kernel;
    overlap: sender check, count, scan, fill), plan (init, layer table,
    rows, scan, runs; sender positions or span rows; window key scan and
    windows when the pooling follows the map), one transfer kernel."""
    align = {"ta": 3, "same_index": 1, "overlap_mean": 4}[w.align_mode]
    plan = (5 + (1 if (w.sender_k_rotated or w.span_gap) else 0)
            + (2 if _pool_after_map(w, pool_before_map) else 0))
    return align + plan + 1


def step_launches(w, tok, pool_before_map=False, round_built=False, captured=False):
    """Kernel launches of one hf_align_build + hf_plan_create + hf_transfer: up
    to 32,768 tokens a side and 64 requests the alignment and the plan are one
    launch each; bf16 operand rows that are computed are made before each
    transfer launch, outside of captures, for as many receiver layers as 512 MB
    hold: by one pass, or two where rotated keys and computed values differ."""
    n = launches_per_step(w, pool_before_map)
    if max(tok.T_r, tok.T_s) <= 32768 and w.n_req <= 64:
        n = 3
    if (w.dtype == "bf16" and not captured and not _copied_operands(w, pool_before_map)
            and _made_rows_pay(w, tok, pool_before_map, round_built)):
        one_role = _copied_operands(w.with_(sender_k_rotated=False), pool_before_map) and \
            w.align_mode != "overlap_mean"
        rows = tok.T_s if _pool_after_map(w, pool_before_map) else tok.T_r
        layer = (1 if one_role else 2) * max(rows, 1) * w.K * (2 if round_built else 4)
        if layer <= 4 << 29:
            passes = 2 if w.sender_k_rotated and not one_role else 1
            n += (passes + 1) * -(-w.L_r // min(w.L_r, max(1, (1 << 29) // layer))) - 1
    return n


def _made_rows_pay(w, tok, pool_before_map, round_built):
    """The library's rule for computed rows (made_rows_pay of hf_plan.cu)."""
    passes = w.d_r // (512 if w.d_r % 512 == 0 else 256 if w.d_r % 256 == 0 else 128)
    if w.sender_k_rotated or passes > 2:
        return True
    after = _pool_after_map(w, pool_before_map)
    rows = (tok.T_s if after else min(tok.T_s, tok.T_r) if w.align_mode == "same_index"
            else tok.T_r * 28 // 100 if w.align_mode == "ta" else tok.T_r)
    staged = (after or w.align_mode != "overlap_mean") and not round_built
    small = rows * w.K <= (5000000 if w.align_mode == "ta" else 16000000)
    if passes == 2:
        return small or not staged
    tiles = 2 * w.L_r * -(-rows // 256)
    rounds = -(-tiles // 76)
    return small if not staged else 2 * tiles <= 76 or (
        w.K <= 1024 and rounds <= 3 and 4 * tiles <= 3 * 76 * rounds)


def _copied_operands(w, pool_before_map=False):
    """Every map input row is a copy of one sender row: one-entry alignment
    rows (or sender rows whose maps are pooled afterwards), segments of one
    sender layer of weight 1, keys without RoPE."""
    if w.layer_mode == "interp" or w.sender_k_rotated:
        return False
    if w.align_mode == "overlap_mean" and not _pool_after_map(w, pool_before_map):
        return False
    if w.layer_mode == "explicit":
        return all(len(terms) == 1 and float(terms[0]) == 1.0
                   for layer in w.seg_w for terms in layer)
    return True


def blas_threads():
    for k in ("OPENBLAS_NUM_THREADS", "OMP_NUM_THREADS", "MKL_NUM_THREADS"):
        v = os.environ.get(k)
        if v and v.isdigit():
            return int(v)
    return os.cpu_count() or 1


def sized_oracle_sample(w, tok, sender, Wm, b, r, seconds):
    """Calibrates the sample size so one oracle pass takes ~`seconds`."""
    probe = OracleSample(w, tok, sender, Wm, b, r, 32)
    t0 = time.perf_counter()
    probe.run()
    dt = max(time.perf_counter() - t0, 1e-3)
    n = int(32 * seconds / dt)
    n = max(32, min(n, tok.T_r))
    return OracleSample(w, tok, sender, Wm, b, r, n)


# ---------------------------------------------------------------------------
def run_reference(args):
    """--impl reference: the fp64 oracle on the host cores, one bounded
    sample of the workload per step."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    import torch
    from paper_2609_32259_gb300 import workloads as W
    w = workload(args.workload)
    tok = W.tokens(w)
    dev = torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")
    sender = W.sender_kv(w, W.sender_cache_rows(w, tok), dev)
    Wm, b, r = W.maps(w, dev)
    per_step = max(1.0, min(8.0, 150.0 / max(1, args.steps + args.warmup)))
    samp = sized_oracle_sample(w, tok, sender, Wm, b, r, per_step)
    for _ in range(args.warmup):
        samp.run()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        samp.run()
    dt = (time.perf_counter() - t0) / max(1, args.steps)
    value = samp.n_rows / dt
    sample = (f"{samp.n_rows} contiguous receiver rows x {w.L_r} layers x K/V of "
              f"{w.name} per step (dense fp64 numpy, oracle as written)")
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": dt * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": w.name, "T_r": tok.T_r, "T_s": tok.T_s,
                   "mode": f"{w.align_mode}+{w.layer_mode}"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": blas_threads(),
                         "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def run_ours(args):
    import numpy as np
    import torch
    import torch.distributed as dist

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    if not torch.cuda.is_available():
        print(json.dumps({"error": "no CUDA device"}))
        return 1
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    import __graft_entry__ as g
    if rank == 0:
        g.build()
    if world > 1:
        dist.barrier()
    from paper_2609_32259_gb300 import pipeline, workloads as W

    w = workload(args.workload)
    tok = W.tokens(w)
    sender = W.sender_kv(w, W.sender_cache_rows(w, tok), dev)
    Wm, b, r = W.maps(w, dev)
    paged = W.paged_layout(w, tok) if w.paged else None
    job = pipeline.job_from_workload(w, tok, sender, Wm, b, r, paged=paged, device=dev,
                                     round_built_operands=args.round_built_operands,
                                     pool_before_map=args.pool_before_map)
    stream = torch.cuda.current_stream(dev)

    for _ in range(max(3, args.warmup)):
        job.step(stream)
    torch.cuda.synchronize()
    status = job.device_status()
    U = job.distinct_rows()
    _, col, _ = job.csr()
    n_cols = int(np.unique(col).size)

    # timed region: K whole steps, plus the transfer kernel alone per step.
    # A working set below 512 MB could stay in the 129 MB L2 from one step to
    # the next, so such workloads write a 256 MB buffer between steps, outside
    # the timed events of each step.
    working_set = (sender.numel() * sender.element_size() + Wm.numel() * Wm.element_size()
                   + job.receiver.numel() * job.receiver.element_size())
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev) if working_set < (512 << 20) else None
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    st = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.3)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    if args.graph:
        job.capture()
        job.replay()
        torch.cuda.synchronize()
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    t_start.record(stream)
    for i in range(args.steps):
        if flush is not None:
            flush.fill_(i & 0xff)
        st[i][0].record(stream)
        if args.graph:
            job.replay(prep=True, xfer=False)
        else:
            job.align(stream)
            job.make_plan(stream)
        ev[i][0].record(stream)
        if args.graph:
            job.replay(prep=False, xfer=True)
        else:
            job.transfer(stream)
        ev[i][1].record(stream)
        st[i][1].record(stream)
    t_end.record(stream)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clk = clocks.stop()
    step_ms = (t_start.elapsed_time(t_end) / args.steps if flush is None
               else statistics.mean(a.elapsed_time(bb) for a, bb in st))
    kern_all = [a.elapsed_time(bb) for a, bb in ev]
    kern_ms = statistics.mean(kern_all)
    # spread of the kernel time over the run (a power cap shows as later
    # steps slower than the first ones)
    q = sorted(kern_all)
    kern_spread = {"p10": q[len(q) // 10], "p50": q[len(q) // 2], "p90": q[(9 * len(q)) // 10],
                   "first_tenth_mean": statistics.mean(kern_all[:max(1, len(q) // 10)]),
                   "last_tenth_mean": statistics.mean(kern_all[-max(1, len(q) // 10):])}
    value, (step_ms, kern_ms) = aggregate([step_ms, kern_ms], tok.T_r, world)

    # end to end through the API with host buffers
    e2e = None
    if not args.no_e2e:
        h_sender = torch.empty(sender.shape, dtype=sender.dtype, pin_memory=True)
        h_sender.copy_(sender)
        h_recv = torch.empty(job.receiver.shape, dtype=job.receiver.dtype, pin_memory=True)
        h_s_end = torch.as_tensor(tok.s_end).pin_memory()
        h_r_end = torch.as_tensor(tok.r_end).pin_memory()
        n_e2e = max(1, args.e2e_steps)
        torch.cuda.synchronize()
        marks = [torch.cuda.Event(enable_timing=True) for _ in range(n_e2e + 1)]
        for it in range(n_e2e + 1):  # first pass warms up
            if it >= 1:
                marks[it - 1].record(stream)
            job.s_end.copy_(h_s_end, non_blocking=True)
            job.r_end.copy_(h_r_end, non_blocking=True)
            job.align(stream)
            job.make_plan(stream)
            # hf_transfer_host: sender copied in, receiver copied out, by
            # receiver-layer groups overlapped with the computation
            job.transfer_host(h_sender, h_recv, args.e2e_groups, stream)
        marks[n_e2e].record(stream)
        torch.cuda.synchronize()
        # per-step times; the host link of these shared machines shows
        # occasional 2-5x slow steps, so the median step is reported
        per_step = [marks[i].elapsed_time(marks[i + 1]) for i in range(n_e2e)]
        e2e_mean = statistics.mean(per_step)
        e2e_ms = statistics.median(per_step)
        e2e_value, (e2e_ms, e2e_mean) = aggregate([e2e_ms, e2e_mean], tok.T_r, world)
        # the same steps with the receiver cache left in device memory (the
        # receiver model reads it there); the status word is read back
        for it in range(n_e2e + 1):
            if it >= 1:
                marks[it - 1].record(stream)
            job.s_end.copy_(h_s_end, non_blocking=True)
            job.r_end.copy_(h_r_end, non_blocking=True)
            job.align(stream)
            job.make_plan(stream)
            job.transfer_host(h_sender, None, args.e2e_groups, stream)
            job.device_status(stream)
        marks[n_e2e].record(stream)
        torch.cuda.synchronize()
        resident_ms = statistics.median(marks[i].elapsed_time(marks[i + 1]) for i in range(n_e2e))
        _, (resident_ms,) = aggregate([resident_ms], tok.T_r, world)
        # hf_transfer_host reads only the referenced sender rows when every
        # alignment row is one sender token (here: Token Alignment, Eq. 1)
        one_token_rows = (w.align_mode in ("ta", "same_index") and w.layer_mode == "paper3"
                          and not w.sender_k_rotated)
        sender_bytes = (w.L_s * 2 * U * w.d_s * sender.element_size() if one_token_rows
                        else sender.numel() * sender.element_size())
        h2d = sender_bytes + h_s_end.numel() * 4 + h_r_end.numel() * 4
        d2h = job.receiver.numel() * job.receiver.element_size()
        e2e = {"value": e2e_value, "unit": UNIT, "ms_per_step": e2e_ms,
               "ms_per_step_mean": e2e_mean, "steps": n_e2e, "statistic": "median step",
               "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h),
               "api": "hf_align_build + hf_plan_create + hf_transfer_host (pinned host caches)",
               "sender_read": "referenced rows only" if one_token_rows else "whole layers",
               "receiver_in_device_memory": {
                   "value": tok.T_r * world / (resident_ms * 1e-3), "ms_per_step": resident_ms,
                   "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": 4}}
        del h_sender, h_recv

    hbm_gbs, tflops, tflops_sust, src = peaks()
    flops, bytes_ = algorithmic_work(w, tok, U, n_cols)
    t_k = kern_ms * 1e-3
    t_tensor = flops / (tflops * 1e12)
    t_hbm = bytes_ / (hbm_gbs * 1e9)
    if t_tensor >= t_hbm:
        roof = {"bound": "tensor", "achieved": flops / t_k / 1e12, "peak": tflops,
                "unit": "TFLOP/s", "frac": (flops / t_k / 1e12) / tflops}
    else:
        roof = {"bound": "hbm", "achieved": bytes_ / t_k / 1e9, "peak": hbm_gbs,
                "unit": "GB/s", "frac": (bytes_ / t_k / 1e9) / hbm_gbs}
    # the same contraction over every receiver row (no sharing between rows
    # with identical alignment rows): the plain 2 * 2L_r * T_r * K * d_r
    # count; its "fraction" can exceed 1 because the kernel does not do it
    flops_dense = 2.0 * 2 * w.L_r * tok.T_r * w.K * w.d_r
    roof.update({"traffic": None, "peak_source": src, "kernel": "transfer_kernel",
                 "flop_dense_rows": flops_dense,
                 "tensor_dense_equivalent_tflops": flops_dense / t_k / 1e12,
                 "dense_equivalent_frac": (flops_dense / t_k / 1e12) / tflops,
                 "dense_note": ("FLOP of the map over all T_r receiver rows, as if each row "
                                "were contracted; the kernel contracts the distinct rows only"),
                 "frac_of_sustained_peak": (flops / t_k / 1e12) / tflops_sust,
                 "kernel_ms": kern_ms, "kernel_ms_spread": kern_spread,
                 "flop_alg": flops, "bytes_alg": bytes_,
                 "hbm_achieved_gbs": bytes_ / t_k / 1e9,
                 "tensor_achieved_tflops": flops / t_k / 1e12,
                 "roofline_ms": max(t_tensor, t_hbm) * 1e3})
    # DRAM bytes of one transfer-kernel launch from an ncu capture
    # (profiles/transfer_traffic.json), used only while the kernel sources
    # are the ones the capture was taken with
    traffic_file = os.path.join(ROOT, "profiles", "transfer_traffic.json")
    if os.path.exists(traffic_file):
        with open(traffic_file) as f:
            tr = json.load(f).get(w.name)
        if tr and tr.get("kernel_sha256") == kernel_sources_sha256():
            roof["traffic"] = tr["bytes"]
            roof["traffic_source"] = tr["source"]

    cpu = None
    if rank == 0 and not args.no_cpu_baseline:
        samp = sized_oracle_sample(w, tok, sender, Wm, b, r, args.cpu_seconds)
        t0 = time.perf_counter()
        samp.run()
        dt = time.perf_counter() - t0
        cpu = {"value": samp.n_rows / dt, "unit": UNIT, "cores": blas_threads(),
               "kind": "oracle", "seconds": dt,
               "sample": (f"{samp.n_rows} contiguous receiver rows x {w.L_r} layers x K/V "
                          f"of {w.name} (dense fp64 numpy oracle as written)")}

    launches = step_launches(w, tok, args.pool_before_map, args.round_built_operands,
                             captured=args.graph)
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": step_ms,
        "us_per_transfer": step_ms * 1e3, "us_per_transfer_kernel": kern_ms * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": w.dtype, "data": "synthetic",
        "config": {"workload": w.name, "T_r": tok.T_r, "T_s": tok.T_s,
                   "distinct_rows": U, "sender": f"{w.L_s}x{w.H_s}x{w.D_s}",
                   "receiver": f"{w.L_r}x{w.H_r}x{w.D_r}",
                   "mode": f"{w.align_mode}+{w.layer_mode}",
                   "pooling": ("after the map (mapped sender rows pooled in the epilogue)"
                               if _pool_after_map(w, args.pool_before_map) else
                               "before the map" if w.align_mode == "overlap_mean" else None),
                   "operands": ("copied sender rows" if _copied_operands(w, args.pool_before_map)
                                else "computed rows rounded once to bf16"
                                if args.round_built_operands or w.dtype != "bf16"
                                else "computed rows as bf16 value + residual"),
                   "l2": ("inputs larger than L2 (no flush)" if flush is None else
                          "256 MB L2 flush write between steps (outside the timed events)"),
                   "launch": ("CUDA graph replay (align + plan, transfer)" if args.graph
                              else "stream launches"),
                   "parallelism": "replicas" if world > 1 else "single"},
        "roofline": roof, "cpu_baseline": cpu, "e2e": e2e, "clocks": clk,
        "gpu_launches": launches * args.steps, "device_status": status,
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    job.close()
    if world > 1:
        dist.destroy_process_group()
    return 0


def run_batch(args):
    """A three-agent message round: six directions (every family pair), each
    a message span after a context, transferred by one hf_transfer_batch
    call per step; the same directions one hf_transfer after another are
    timed beside it."""
    import numpy as np
    import torch
    if not torch.cuda.is_available():
        print(json.dumps({"error": "no CUDA device"}))
        return 1
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    import __graft_entry__ as g
    g.build()
    from paper_2609_32259_gb300 import binding as B, pipeline, workloads as W
    ws = W.message_round()
    jobs, works = [], []
    for w in ws:
        tok = W.tokens(w)
        sender = W.sender_kv(w, W.sender_cache_rows(w, tok), dev)
        Wm, b, r = W.maps(w, dev)
        jobs.append(pipeline.job_from_workload(w, tok, sender, Wm, b, r, device=dev))
        works.append((w, tok))
    stream = torch.cuda.current_stream(dev)

    def prepare():
        for j in jobs:
            j.align(stream)
            j.make_plan(stream)

    def batch():
        B.transfer_batch([j.plan for j in jobs], [j.sender for j in jobs],
                         [j.receiver for j in jobs], stream)

    def sequential():
        for j in jobs:
            j.transfer(stream)

    for _ in range(max(3, args.warmup)):
        prepare()
        batch()
        sequential()
    torch.cuda.synchronize()
    if args.graph:  # the six alignments + plans, and the one batched transfer, as graphs
        g_prep, g_batch = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(g_prep):
            for j in jobs:
                j.align(torch.cuda.current_stream())
                j.make_plan(torch.cuda.current_stream())
        with torch.cuda.graph(g_batch):
            B.transfer_batch([j.plan for j in jobs], [j.sender for j in jobs],
                             [j.receiver for j in jobs], torch.cuda.current_stream())
        prepare = g_prep.replay
        batch = g_batch.replay
        prepare()
        batch()
        torch.cuda.synchronize()
    status = max(j.device_status() for j in jobs)
    flops = bytes_ = 0.0
    T_total = 0
    for (w, tok), j in zip(works, jobs):
        _, col, _ = j.csr()
        f, by = algorithmic_work(w, tok, j.distinct_rows(), int(np.unique(col).size))
        flops += f
        bytes_ += by
        T_total += tok.T_r
    res = {}
    clocks = ClockSampler(0)
    clocks.start()
    time.sleep(0.3)
    for name, fn in (("batch", batch), ("sequential", sequential)):
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
              for _ in range(args.steps)]
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        t0.record(stream)
        for i in range(args.steps):
            prepare()
            ev[i][0].record(stream)
            fn()
            ev[i][1].record(stream)
        t1.record(stream)
        torch.cuda.synchronize()
        res[name] = (t0.elapsed_time(t1) / args.steps,
                     statistics.mean(a.elapsed_time(bb) for a, bb in ev))
    clk = clocks.stop()
    step_ms, kern_ms = res["batch"]
    hbm_gbs, tflops, tflops_sust, src = peaks()
    t_k = kern_ms * 1e-3
    if flops / (tflops * 1e12) >= bytes_ / (hbm_gbs * 1e9):
        roof = {"bound": "tensor", "achieved": flops / t_k / 1e12, "peak": tflops,
                "unit": "TFLOP/s", "frac": flops / t_k / 1e12 / tflops}
    else:
        roof = {"bound": "hbm", "achieved": bytes_ / t_k / 1e9, "peak": hbm_gbs,
                "unit": "GB/s", "frac": bytes_ / t_k / 1e9 / hbm_gbs}
    roof.update({"traffic": None, "peak_source": src, "kernel": "transfer_kernel x6",
                 "kernel_ms": kern_ms, "flop_alg": flops, "bytes_alg": bytes_})
    line = {
        "metric": METRIC, "value": T_total / (step_ms * 1e-3), "unit": UNIT, "n_gpus": 1,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": step_ms,
        "us_per_transfer_kernel": kern_ms * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
        "config": {"workload": "message_round_6x160", "directions": [w.name for w in ws],
                   "T_r_total": T_total, "context_tokens": ws[0].span_gap,
                   "sequential_kernel_ms": res["sequential"][1],
                   "sequential_step_ms": res["sequential"][0],
                   "l2": "maps (1.2 GB) larger than L2 (no flush)",
                   "launch": ("CUDA graph replay (align + plan of the six directions, batched "
                              "transfer)" if args.graph else "stream launches"),
                   "parallelism": "single"},
        "roofline": roof, "cpu_baseline": None, "e2e": None, "clocks": clk,
        "gpu_launches": (sum(step_launches(w, tok) - 1 for w, tok in works) + 1) * args.steps,
        "device_status": status,
    }
    print(json.dumps(line), flush=True)
    for j in jobs:
        j.close()
    return 0


def run_fold(args):
    """hf_fold (Eq. 9) over every map of the 32K Llama->Ministral-shaped
    direction (80 maps of 1,024 x 3,072, rank 16), folded in place."""
    import torch
    if not torch.cuda.is_available():
        print(json.dumps({"error": "no CUDA device"}))
        return 1
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    import __graft_entry__ as g
    g.build()
    from paper_2609_32259_gb300 import binding as B, workloads as W
    w = W.llama_to_ministral(32768)
    Wm, b, _ = W.maps(w, dev)
    n_maps, rank = 2 * w.L_r, 16
    gen = torch.Generator(device=dev).manual_seed(11)
    Bm = torch.randn((n_maps, w.d_r, rank), generator=gen, device=dev) * 0.02
    Gm = torch.randn((n_maps, rank, w.d_r), generator=gen, device=dev) * 0.02
    Wf = Wm.view(n_maps, w.d_r, w.K)
    bf = b.view(n_maps, w.d_r)
    stream = torch.cuda.current_stream(dev)
    for _ in range(max(3, args.warmup)):
        B.fold("bf16", Wf, bf, Bm, Gm, Wf, bf, stream)
    torch.cuda.synchronize()
    clocks = ClockSampler(0)
    clocks.start()
    time.sleep(0.3)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        B.fold("bf16", Wf, bf, Bm, Gm, Wf, bf, stream)
    e1.record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    ms = e0.elapsed_time(e1) / args.steps
    # read W and write W_final once; the factors and biases are small.  The 4 *
    # rank FLOP per element (T = B^T W, then G^T T) are three and six bf16
    # products on the warp-level tensor instructions and take less than the bytes.
    bytes_ = 2.0 * Wf.numel() * 2 + (Bm.numel() + Gm.numel() + 2 * bf.numel()) * 4
    flops = 4.0 * rank * Wf.numel()
    hbm_gbs, _, _, src = peaks()
    hbm_ach = bytes_ / (ms * 1e-3) / 1e9
    line = {"metric": "maps folded per second (Eq. 9)", "value": n_maps / (ms * 1e-3),
            "unit": "maps/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "bf16", "data": "synthetic",
            "config": {"workload": "fold_llama8b_to_ministral_maps", "n_maps": n_maps,
                       "d_R": w.d_r, "K": w.K, "rank": rank,
                       "l2": "inputs larger than L2 (no flush)", "parallelism": "single"},
            "roofline": {"bound": "hbm", "achieved": hbm_ach, "peak": hbm_gbs, "unit": "GB/s",
                         "frac": hbm_ach / hbm_gbs, "traffic": None, "peak_source": src,
                         "kernel": "fold_mma_kernel + fold_b_kernel", "flop_alg": flops,
                         "bytes_alg": bytes_},
            "cpu_baseline": None, "e2e": None, "clocks": clk, "gpu_launches": 2 * args.steps}
    print(json.dumps(line), flush=True)
    return 0


def run_recolor(args):
    """hf_recolor_fit (Eq. 3-5) for one map of the 32K Llama->Ministral-shaped
    direction: 32,768 weighted sample pairs, d_S = 3 x 1,024, d_R = 1,024."""
    import torch
    if not torch.cuda.is_available():
        print(json.dumps({"error": "no CUDA device"}))
        return 1
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    import __graft_entry__ as g
    g.build()
    from paper_2609_32259_gb300 import binding as B
    N, d_s, d_r = 32768, 3072, 1024
    gen = torch.Generator(device=dev).manual_seed(12)
    X = (torch.randn((N, d_s), generator=gen, device=dev)
         @ (torch.randn((d_s, d_s), generator=gen, device=dev) / d_s ** 0.5)).to(torch.bfloat16)
    A_true = torch.randn((d_s, d_r), generator=gen, device=dev) / d_s ** 0.5
    Y = (X.float() @ A_true + 0.5 * torch.randn((N, d_r), generator=gen, device=dev)).to(torch.bfloat16)
    w = torch.rand((N,), generator=gen, device=dev) + 0.5
    ws = torch.empty(B.recolor_workspace_size(N, d_s, d_r), dtype=torch.uint8, device=dev)
    W_out = torch.empty((d_r, d_s), dtype=torch.bfloat16, device=dev)
    b_out = torch.empty((d_r,), dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)
    B.recolor_fit("bf16", X, Y, w, W_out, b_out, ws, reg=1e-3, stream=stream)  # warm-up
    torch.cuda.synchronize()
    clocks = ClockSampler(0)
    clocks.start()
    time.sleep(0.3)
    steps = max(1, min(args.steps, 5))
    t0 = time.perf_counter()
    for _ in range(steps):
        _, its = B.recolor_fit("bf16", X, Y, w, W_out, b_out, ws, reg=1e-3, stream=stream,
                               return_iters=True)
    torch.cuda.synchronize()
    ms = (time.perf_counter() - t0) * 1e3 / steps
    clk = clocks.stop()
    # products performed: moments (upper triangle); the covariances' factors and
    # their inverses (2 d^3 / 3 each); two per polar iteration; the whitening of
    # Sigma_ZY and the two products of A
    flops = (1.0 * N * (d_s + d_r) ** 2
             + 2.0 / 3.0 * (d_s ** 3 + d_r ** 3)
             + 4.0 * its[2] * d_s * d_r * d_r
             + 2 * (2.0 * d_s * d_s * d_r + 2.0 * d_s * d_r * d_r))
    sm_mhz = clk.get("sm_mhz") or 2070.0
    alu_peak = 152 * 128 * 2 * sm_mhz * 1e6 / 1e12
    # the products run on the bf16 tensor cores with each fp32 operand split
    # into three bf16 parts and the six largest of the nine partial products
    # kept: six bf16 products per fp32 product
    emu_peak = peaks()[1] / 6.0
    achieved = flops / (ms * 1e-3) / 1e12
    line = {"metric": "Recolor maps fitted per second (Eq. 3-5)", "value": 1e3 / ms,
            "unit": "maps/s", "n_gpus": 1, "steps": steps, "warmup": 1, "ms_per_step": ms,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": "recolor_fit_32768x3072x1024", "N": N, "d_S": d_s, "d_R": d_r,
                       "reg": 1e-3, "l2": "inputs larger than L2 (no flush)",
                       "parallelism": "single", "timing": "host clock around synchronous calls"},
            "roofline": {"bound": "tensor", "achieved": achieved, "peak": emu_peak,
                         "unit": "TFLOP/s", "frac": achieved / emu_peak, "traffic": None,
                         "peak_source": "measured bf16 tensor peak / 6 (fp32 products as six "
                                        "bf16 products)",
                         "kernel": "gemm_kernel (+ operand split, reduce and elementwise passes)",
                         "frac_of_fp32_alu_peak": achieved / alu_peak,
                         "flop_alg": flops, "iterations": its},
            "cpu_baseline": None, "e2e": None, "clocks": clk, "gpu_launches": None}
    print(json.dumps(line), flush=True)
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "message_round":
        return run_batch(args)
    if args.workload == "fold":
        return run_fold(args)
    if args.workload == "recolor":
        return run_recolor(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())

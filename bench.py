"""Benchmark: hybrid SpMM on the power-law graph workload (one JSON line on stdout).

Workload (default): RMAT(.57,.19,.19,.05) graph, 2^20 x 2^20, 2^24 distinct edges, GCN values
1/deg(row), B = 2^20 x 128 FP32 N(0,1) -- synthetic stand-in for the paper's GNN graphs.

A step is one pass of the whole hot path over that input: the device planner (validation,
extraction, windows/compaction/binning when enabled, residual chunks, cost-ordered work list)
followed by the one persistent execute launch, then the plan is released.  Inputs are resident
in HBM before timing; A (138 MB), B (512 MiB) and C (512 MiB) exceed the 129 MB L2, so no flush
is needed between steps.

  value      SpMM GFLOP/s = 2 * nnz * K / step time (device time, CUDA events, max over ranks)
  roofline   the execute kernel: algorithmic bytes (CSR + touched B rows + C) / its mean
             CUDA-event duration, against the measured HBM copy bandwidth
  e2e        the same metric through ns_spmm_host with pinned host buffers (H2D of A and B,
             plan, execute, D2H of C inside the timed region)
  cpu_baseline  the FP64 oracle on the host cores over the whole matrix (about 0.2 s on 16
             cores for the power-law graph; larger workloads take a bounded row sample), with a
             single-thread figure and the CPU model

--impl reference runs the oracle (the reference arm of this build) on the same workload, the
whole matrix every step, and prints the same metric.
With --gpus N > 1 (torchrun) every rank runs an independent replica (the path needs no
exchange); value sums the replicas' work over the slowest rank's time.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

PEAKS_PATH = os.path.join(ROOT, "MEASURED_PEAKS.json")
FALLBACK_HBM = 6800.0
# the headline metric, printed identically by both arms
METRIC = "SpMM GFLOP/s (2*nnz*K/s) & % HBM roofline"


def _peaks():
    try:
        with open(PEAKS_PATH) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM, "fallback"


class ClockSampler:
    """nvidia-smi clocks and throttle reasons, sampled every 20 ms.  The sampler is started and
    has delivered its first sample before the timed region begins (`with` entry waits for it);
    `summary()` keeps the samples that arrived between `start()` and `stop()` (a sample arrives
    a few ms after it is taken), or, for a region shorter than the interval, the first sample
    after `start()`."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []  # (arrival time, line)
        self.t0 = self.t1 = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "20"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
            deadline = time.perf_counter() + 5.0
            while not self.lines and time.perf_counter() < deadline and self.proc.poll() is None:
                time.sleep(0.005)
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append((time.perf_counter(), line.strip()))

    def start(self):
        self.t0 = time.perf_counter()

    def stop(self):
        self.t1 = time.perf_counter()
        time.sleep(0.05)  # let the samples taken inside the region arrive

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        rows = self.lines
        if self.t0 is not None and self.t1 is not None:
            inside = [ln for t, ln in rows if self.t0 <= t <= self.t1 + 0.03]
            after = [ln for t, ln in rows if t >= self.t0][:1]
            picked = inside or after
        else:
            picked = [ln for _, ln in rows]
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in picked:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"], "samples": 0}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": float(max(mx)),
                "reasons": sorted(reasons), "samples": len(sm)}


# DRAM traffic of the execute kernel per launch: dram__bytes_read.sum + dram__bytes_write.sum
# from one ncu capture (summarised in profiles/), keyed by workload and tune.  It is valid only for
# the kernel source it was taken on: the digest of the execute kernel's sources must match,
# otherwise the roofline reports traffic as null.
EXEC_SOURCES = ("ns_exec.cu", "ns_contig.cu", "ns_exec_f32.cu", "ns_residual.cuh", "ns_mem.cuh",
                "ns_internal.cuh", "ns_dense.cuh", "ns_dense_tc.cuh", "ns_ptx.cuh")
MEASURED_TRAFFIC = {
    # (workload, tau_tile, chunk_nnz, l2_hints): (source digest, bytes per launch)
    ("powerlaw", 2147483647, 512, 1): ("c218fd6215f19630", 1772762112 + 551939072),
    ("powerlaw", 2147483647, 256, 1): ("c218fd6215f19630", 1786630656 + 597434624),
    ("powerlaw", 2147483647, 1024, 1): ("c218fd6215f19630", 1757437440 + 535467776),
}


def exec_source_digest() -> str:
    import hashlib
    h = hashlib.sha256()
    for f in EXEC_SOURCES:
        with open(os.path.join(ROOT, "paper_2606_22482_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def measured_traffic(workload: str, tune) -> float | None:
    rec = MEASURED_TRAFFIC.get((workload, int(tune.tau_tile), int(tune.chunk_nnz), int(tune.l2_hints)))
    if rec is None or rec[0] != exec_source_digest():
        return None
    return rec[1]


def make_workload(name: str, seed: int):
    import synth
    if name == "powerlaw":
        A, B = synth.config_powerlaw(seed)
        desc = {"workload": "powerlaw-rmat-2^20-16.7Mnnz-K128-fp32", "m": A["m"], "n": A["n"],
                "nnz": A.nnz, "K": 128, "b_dtype": "f32", "seed": seed,
                "graph": "RMAT(.57,.19,.19,.05) relabelled, GCN values"}
    elif name == "powerlaw-community":
        A, B = synth.config_powerlaw(seed, community=True)
        desc = {"workload": "powerlaw-rmat-2^20-16.7Mnnz-K128-fp32-community-rows", "m": A["m"], "n": A["n"],
                "nnz": A.nnz, "K": 128, "b_dtype": "f32", "seed": seed,
                "graph": "RMAT(.57,.19,.19,.05) relabelled, rows in seeded community order, GCN values"}
    elif name == "attention":
        A, B = synth.config_attention(seed)
        desc = {"workload": "block-sparse-attention-32768-K128-fp32", "m": A["m"], "n": A["n"],
                "nnz": A.nnz, "K": 128, "b_dtype": "f32", "seed": seed}
    elif name == "attention-bf16":
        A, B = synth.config_attention(seed)
        desc = {"workload": "block-sparse-attention-32768-K128-bf16", "m": A["m"], "n": A["n"],
                "nnz": A.nnz, "K": 128, "b_dtype": "bf16", "seed": seed}
    elif name == "small":
        A, B = synth.config_small(seed)
        desc = {"workload": "uniform-4096-16nnz-K32-fp32", "m": A["m"], "n": A["n"],
                "nnz": A.nnz, "K": 32, "b_dtype": "f32", "seed": seed}
    else:
        raise SystemExit(f"unknown workload {name}")
    return A, B, desc


def algorithmic_bytes(A, K: int, b_bytes: int) -> int:
    n_touched = int(np.count_nonzero(np.bincount(A["colidx"], minlength=A["n"])))
    return 4 * (A["m"] + 1) + 8 * A.nnz + b_bytes * K * n_touched + 4 * A["m"] * K, n_touched


def cpu_sample_rows(A, target_nnz: int, seed: int = 7):
    """A row sample of about target_nnz nonzeros (uniform over rows, so the degree mix holds)."""
    rng = np.random.default_rng(seed)
    m = A["m"]
    frac = min(1.0, target_nnz / max(A.nnz, 1))
    if frac >= 1.0:
        return np.arange(m, dtype=np.int32), int(A.nnz)
    rows = np.nonzero(rng.random(m) < frac)[0].astype(np.int32)
    lens = np.diff(A["rowptr"].astype(np.int64))[rows]
    return rows, int(lens.sum())


def cpu_model() -> str:
    """The host CPU's model name (lscpu), for the record beside the CPU baseline."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        fields = dict(ln.split(":", 1) for ln in out.splitlines() if ":" in ln)
        name = fields.get("Model name", "").strip()
        vendor = fields.get("Vendor ID", "").strip()
        return f"{vendor} {name}".strip() or "unknown"
    except Exception:
        import platform
        return platform.processor() or "unknown"


def oracle_single_thread(A, B, K, bf16: bool, seconds_budget: float = 4.0) -> dict:
    """The oracle on one host core, on a row sample sized for about seconds_budget."""
    import oracle
    rows, nnz_s = cpu_sample_rows(A, 100_000, seed=5)
    t0 = time.perf_counter()
    oracle.spmm(A, B, rows=rows, threads=1, b_bf16=bf16)
    rate = 2.0 * nnz_s * K / max(time.perf_counter() - t0, 1e-9)
    rows, nnz_s = cpu_sample_rows(A, int(rate * seconds_budget / (2.0 * K)), seed=13)
    t0 = time.perf_counter()
    oracle.spmm(A, B, rows=rows, threads=1, b_bf16=bf16)
    dt = time.perf_counter() - t0
    return {"value": 2.0 * nnz_s * K / dt / 1e9, "unit": "GFLOP/s", "cores": 1,
            "sample": f"{len(rows)} uniformly sampled rows ({nnz_s} nnz, {nnz_s / A.nnz:.1%} of A), "
                      f"FP64, {dt:.1f} s"}


def run_cpu_oracle(A, B, K, seconds_budget: float, threads: int, bf16: bool = False, C_gpu=None):
    """Time the oracle, as it stands, on all host cores: the whole matrix when that fits about
    seconds_budget, else a uniform row sample of that size.  With C_gpu (the device result,
    copied back after the timed region) the same oracle rows give its error against FP64."""
    import oracle
    rows, nnz_s = cpu_sample_rows(A, 200_000)
    t0 = time.perf_counter()
    oracle.spmm(A, B, rows=rows, threads=threads, b_bf16=bf16)
    t1 = time.perf_counter()
    rate = 2.0 * nnz_s * K / max(t1 - t0, 1e-9)   # flop/s on the probe
    target = int(min(A.nnz, max(200_000, rate * seconds_budget / (2.0 * K))))
    rows, nnz_s = cpu_sample_rows(A, target, seed=11)
    t0 = time.perf_counter()
    ref = oracle.spmm(A, B, rows=rows, threads=threads, b_bf16=bf16)
    dt = time.perf_counter() - t0
    out = {"value": 2.0 * nnz_s * K / dt / 1e9, "unit": "GFLOP/s", "cores": threads,
           "kind": "oracle",
           "sample": f"{len(rows)} rows ({nnz_s} nnz, {nnz_s / A.nnz:.1%} of A), FP64, {dt:.2f} s",
           "cpu_model": cpu_model(),
           "single_thread": oracle_single_thread(A, B, K, bf16)}
    acc = accuracy(A, C_gpu, rows, ref) if C_gpu is not None else None
    return out, acc


def accuracy(A, C_gpu, rows, ref) -> dict:
    """Error of the device result on `rows` against the FP64 oracle's values `ref` there."""
    diff = np.asarray(C_gpu[rows], dtype=np.float64) - ref
    dn, rn = np.linalg.norm(diff, axis=1), np.linalg.norm(ref, axis=1)
    nz = rn > 0
    return {"rel_frobenius_vs_fp64": float(np.linalg.norm(dn) / max(np.linalg.norm(rn), 1e-300)),
            "max_row_rel_err": float((dn[nz] / rn[nz]).max()) if nz.any() else 0.0,
            "zero_rows_exact": bool(np.all(dn[~nz] == 0)),
            "rows_checked": int(len(rows)), "of_rows": int(A["m"])}


def accuracy_sample(A, B, K, bf16: bool, C_gpu, threads: int, target_nnz: int = 400_000) -> dict:
    """The device result against the FP64 oracle on a uniform row sample (no timing): the
    accuracy figure of a bench line that skips the CPU baseline."""
    import oracle
    rows, _ = cpu_sample_rows(A, target_nnz, seed=11)
    return accuracy(A, C_gpu, rows, oracle.spmm(A, B, rows=rows, threads=threads, b_bf16=bf16))


def replicas_result(ms_step: float, flops_per_rank: float, ws: int, device) -> tuple:
    """Whole-job step time and throughput of `ws` independent replicas (no data-path collective):
    the slowest rank's step time (max over ranks) and all ranks' flops over it, in GFLOP/s.
    Every rank calls it; with ws > 1 the process group must be initialised."""
    if ws > 1:
        import torch
        import torch.distributed as dist
        t = torch.tensor([ms_step], dtype=torch.float64, device=device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        ms_step = float(t.item())
    return ms_step, flops_per_rank * ws / (ms_step * 1e-3) / 1e9


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="powerlaw",
                    choices=["powerlaw", "powerlaw-community", "attention", "attention-bf16", "small",
                             "batched", "serve", "gcn"])
    ap.add_argument("--epochs", type=int, default=200, help="GCN epochs (--workload gcn)")
    ap.add_argument("--rebalance", action="store_true",
                    help="choose tau by the epoch-level re-balance loop (Section 5.3) instead")
    ap.add_argument("--rate", type=float, default=2000.0, help="serve: Poisson arrivals per second")
    ap.add_argument("--duration", type=float, default=30.0, help="serve: seconds of arrivals")
    ap.add_argument("--pool", type=int, default=1024, help="serve: graphs in the pool")
    ap.add_argument("--inflight", type=int, default=256, help="serve: requests admitted at once")
    ap.add_argument("--serve-budget", type=float, default=64.0, help="serve: HBM budget (GiB)")
    ap.add_argument("--plain-requests", type=int, default=2000,
                    help="serve: requests of the trace also run one at a time (plain path)")
    ap.add_argument("--serve-trace", default=None, help="serve: write per-request times to this .npz")
    ap.add_argument("--serve-checks", type=int, default=400,
                    help="serve: about this many served results compared with the oracle")
    ap.add_argument("--tau", default="auto", help="'auto' (autotuner), 'inf' or an integer")
    ap.add_argument("--seed", type=int, default=0)
    ap.add_argument("--l2", type=int, default=None, choices=[0, 1, 2],
                    help="override the L2 policy of the tune (2: planner-marked hot B rows)")
    ap.add_argument("--tn", type=int, default=None, help="override the column-slice width TN")
    ap.add_argument("--chunk", type=int, default=None, help="override the residual chunk size W")
    ap.add_argument("--tm", type=int, default=None, choices=[16, 32, 64], help="override the window height TM")
    ap.add_argument("--tk", type=int, default=None, choices=[16, 32], help="override the tile width TK")
    ap.add_argument("--reorder", type=int, default=None,
                    help="Section 6.1 local reordering: windows per cluster (0 = off)")
    ap.add_argument("--no-cpu", action="store_true", help="skip the cpu_baseline leg")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--schedule", default="auto", choices=["auto", "overlapped", "serial"],
                    help="plan each step on a second stream overlapping the previous execute, or "
                         "serially; auto: the faster of the two in the warm-up")
    args = ap.parse_args()

    ws, rank, local = dist_env()
    threads = len(os.sched_getaffinity(0)) if hasattr(os, "sched_getaffinity") else os.cpu_count()

    if args.impl == "reference":
        if rank != 0:
            return
        A, B, desc = make_workload(args.workload, args.seed)
        K = B.shape[1]
        bf16 = desc["b_dtype"] == "bf16"
        import oracle
        if bf16:
            import synth
            B = synth.bf16_bits(B)
        # every step is the whole matrix (the power-law graph takes about 0.2 s on 16 cores)
        rows, nnz_s = cpu_sample_rows(A, A.nnz)
        times = []
        for i in range(args.warmup + args.steps):
            t0 = time.perf_counter()
            oracle.spmm(A, B, rows=rows, threads=threads, b_bf16=bf16)
            dt = time.perf_counter() - t0
            if i >= args.warmup:
                times.append(dt)
        t = float(np.mean(times))
        val = 2.0 * nnz_s * K / t / 1e9
        sample = f"the whole matrix ({len(rows)} rows, {nnz_s} nnz) per step, FP64 oracle"
        print(json.dumps({
            "impl": "reference", "metric": METRIC, "value": val,
            "unit": "GFLOP/s", "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": t * 1e3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": desc,
            "cpu_baseline": {"value": val, "unit": "GFLOP/s", "cores": threads, "kind": "oracle",
                             "sample": sample, "cpu_model": cpu_model(),
                             "single_thread": oracle_single_thread(A, B, K, bf16)},
            "e2e": {"value": val, "unit": "GFLOP/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        }))
        return

    import torch
    import torch.distributed as dist

    if args.workload == "batched":
        return bench_batched(args, threads)
    if args.workload == "serve":
        return bench_serve(args, threads)
    if args.workload == "gcn":
        return bench_gcn(args, threads)
    if ws > 1:
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    import paper_2606_22482_gb300 as ns

    A, B, desc = make_workload(args.workload, args.seed + rank)
    K = B.shape[1]
    bf16 = desc["b_dtype"] == "bf16"
    DT = ns.NS_BF16 if bf16 else ns.NS_F32
    At = {k: (torch.from_numpy(v).to(dev) if isinstance(v, np.ndarray) else v) for k, v in A.items()}
    if bf16:
        import synth
        B = synth.bf16_bits(B)
        Bt = torch.from_numpy(B.view(np.int16)).to(dev).view(torch.bfloat16)
    else:
        Bt = torch.from_numpy(B).to(dev)
    Ct = torch.empty((A["m"], K), device=dev)
    stream = torch.cuda.current_stream()

    # ---- tune: the autotuner picks (TM, tau) from dry runs (untimed, done once) ----
    tune = ns.tune_default()
    tune_src = "default"
    if args.tau == "inf":
        tune.tau_tile = ns.NS_TAU_INF
        tune_src = "fixed tau=inf"
    elif args.tau != "auto":
        tune.tau_tile = int(args.tau)
        tune_src = f"fixed tau={args.tau}"
    else:
        try:
            # each timed step plans afresh: the autotuner weighs plan time fully (plan_runs = 1)
            tune = ns.autotune(At, K, DT, plan_runs=1.0)
            tune_src = "autotuned (objective: plan + execute)"
        except Exception as e:  # autotuner unavailable: pure CUDA-core plan
            tune.tau_tile = ns.NS_TAU_INF
            tune_src = f"default (autotune unavailable: {str(e)[:60]})"

    if args.l2 is not None:
        tune.l2_hints = args.l2
        tune_src += f", l2_hints={args.l2}"
    if args.tn is not None:
        tune.TN = args.tn
        tune_src += f", TN={args.tn}"
    if args.tm is not None:
        tune.TM = args.tm
        tune_src += f", TM={args.tm}"
    if args.tk is not None:
        tune.TK = args.tk
        tune_src += f", TK={args.tk}"
    if args.reorder is not None:
        tune.reorder = args.reorder
        tune_src += f", reorder={args.reorder}"
    if args.chunk is not None:
        tune.chunk_nnz = args.chunk
        tune.absorb_cap = args.chunk
        tune_src += f", chunk_nnz={args.chunk}"
    rebalance_rep = None
    if args.rebalance:
        start = ns.tune_default()
        start.TM = args.tm if args.tm is not None else 16
        tune, rebalance_rep = ns.rebalance(At, K, DT, Bt, Ct, start=start, eps=0.05, max_iter=10)
        tune_src = f"epoch-level re-balance (Section 5.3), TM={tune.TM}"

    # Each step plans afresh and executes.  Overlapped schedule: the plans go on a second stream,
    # so step i + 1's plan runs while step i's execute is on the GPU (the execute waits for its
    # own plan); a plan is released two steps later, so its memory is never the next plan's.
    # Serial schedule: plan, then execute, on one stream.  Nothing is skipped either way: every
    # step validates A, partitions it and executes.  Unless --schedule fixes it, both are timed
    # in the warm-up (untimed) and the faster one is kept: overlap pays when the execute leaves
    # L2 to itself (a large B streamed from HBM), not when the plan's passes evict the L2-resident
    # B the execute gathers from.
    side_stream = torch.cuda.Stream()
    plan_stream = side_stream
    live = []

    def step(ev=None, pev=None):
        if pev is not None:
            pev[0].record(plan_stream)
        p = ns.spmm_plan(At, K, DT, tune, stream=plan_stream)
        if pev is not None:
            pev[1].record(plan_stream)
        if ev is not None:
            ev[0].record(stream)
        p.execute(Bt, Ct, stream=stream)
        if ev is not None:
            ev[1].record(stream)
        live.append(p)
        while len(live) > 2:
            live.pop(0).close()

    def run_steps(n):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(n):
            step()
        torch.cuda.synchronize()
        dt = (time.perf_counter() - t0) / n
        for p in live:
            p.close()
        live.clear()
        return dt

    schedule_probe = {}
    for name in (("overlapped", "serial") if args.schedule == "auto" else (args.schedule,)):
        plan_stream = side_stream if name == "overlapped" else stream
        run_steps(max(args.warmup, 3))
        schedule_probe[name] = run_steps(max(args.warmup, 5)) * 1e3
    schedule = min(schedule_probe, key=schedule_probe.get)
    plan_stream = side_stream if schedule == "overlapped" else stream
    with ns.spmm_plan(At, K, DT, tune) as p:
        st = p.stats()

    exec_events = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
                   for _ in range(args.steps)]
    plan_events = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
                   for _ in range(args.steps)]
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    if ws > 1:
        dist.barrier()
    torch.cuda.synchronize()
    launches0 = ns.launch_count()
    with ClockSampler(local) as clk:
        clk.start()
        t_start.record(stream)
        plan_stream.wait_stream(stream)
        for i in range(args.steps):
            step(exec_events[i], plan_events[i])
        t_end.record(stream)
        torch.cuda.synchronize()
        clk.stop()
    for p in live:
        p.close()
    live.clear()
    launches = ns.launch_count() - launches0
    if ws > 1:
        dist.barrier()
    ms_total = t_start.elapsed_time(t_end)
    exec_ms = float(np.mean([a.elapsed_time(b) for a, b in exec_events]))
    plan_gpu_ms = float(np.mean([a.elapsed_time(b) for a, b in plan_events]))
    ms_step = ms_total / args.steps

    flops = 2.0 * A.nnz * K
    ms_step, value = replicas_result(ms_step, flops, ws, dev)
    hbm, peak_src = _peaks()
    alg_bytes, n_touched = algorithmic_bytes(A, K, 2 if bf16 else 4)
    achieved = alg_bytes / (exec_ms * 1e-3) / 1e9

    # ---- e2e: host buffers through ns_spmm_host ----
    e2e = None
    if not args.no_e2e:
        Ah = {k: (torch.from_numpy(v).pin_memory().numpy() if isinstance(v, np.ndarray) else v)
              for k, v in A.items()}
        Bh = torch.from_numpy(B).pin_memory().numpy()
        Ch = torch.empty((A["m"], K), dtype=torch.float32).pin_memory().numpy()
        for _ in range(2):
            ns.spmm_host(Ah, Bh, Ch, DT, tune)
        n_e2e = max(3, min(args.steps, 10))
        t0 = time.perf_counter()
        for _ in range(n_e2e):
            ns.spmm_host(Ah, Bh, Ch, DT, tune)
        dt = (time.perf_counter() - t0) / n_e2e
        h2d = 4 * (A["m"] + 1) + 8 * A.nnz + B.nbytes
        e2e = {"value": flops * ws / dt / 1e9, "unit": "GFLOP/s", "h2d_bytes_per_step": int(h2d),
               "d2h_bytes_per_step": int(Ch.nbytes), "ms_per_step": dt * 1e3}
        ns.lib.ns_release_cache()

    if rank != 0:
        if ws > 1:
            dist.destroy_process_group()
        return
    cpu = acc = None
    if not args.no_cpu:
        # the last timed step's C, read back after the timed region, against the FP64 oracle
        cpu, acc = run_cpu_oracle(A, B, K, 12.0, threads, bf16, C_gpu=Ct.cpu().numpy())
    else:
        acc = accuracy_sample(A, B, K, bf16, Ct.cpu().numpy(), threads)
    out = {
        "metric": METRIC,
        "value": value, "unit": "GFLOP/s", "n_gpus": ws, "steps": args.steps,
        "warmup": max(args.warmup, 3), "ms_per_step": ms_step, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "bf16" if bf16 else "f32", "data": "synthetic",
        "config": dict(desc, parallelism=f"replicas x{ws}", l2="inputs larger than L2 (A+B+C 1.16 GB)",
                       step=("device plan + one persistent execute launch"
                             + (" (plans on a second stream: a step's plan overlaps the previous execute)"
                                if schedule == "overlapped" else "")), tune=tune.as_dict(),
                       tune_source=tune_src, plan=st),
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s",
                     "frac": achieved / hbm, "traffic": measured_traffic(args.workload, tune),
                     "source_digest": exec_source_digest(),
                     "kernel": "k_exec (persistent execute)", "peak_source": f"{peak_src} hbm_gbs",
                     "algorithmic_bytes": alg_bytes, "n_touched": n_touched,
                     "kernel_ms": exec_ms, "frac_of_8000": achieved / 8000.0},
        "plan_ms": plan_gpu_ms,
        "plan_schedule": {"used": schedule, "warmup_ms_per_step": schedule_probe,
                          "note": "plan_ms is the plan's span on its stream; overlapped, it includes "
                                  "the wait for the previous execute's SMs"},
        "rebalance": rebalance_rep,
        "rel_frobenius_vs_fp64": acc["rel_frobenius_vs_fp64"] if acc else None,
        "accuracy": acc,
        "cpu_baseline": cpu,
        "e2e": e2e,
        "gpu_launches": int(launches),
        "clocks": clk.summary(),
    }
    print(json.dumps(out))
    if ws > 1:
        dist.destroy_process_group()


# ---------------------------------------------------------------------------------------------
# batched form: 512 uneven graphs, K = 64, one persistent launch replayed from a CUDA graph
# ---------------------------------------------------------------------------------------------
def bench_batched(args, threads):
    import torch
    import oracle
    import synth
    import paper_2606_22482_gb300 as ns
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(0)
    graphs, Bs = synth.config_batched(args.seed)
    K = 64
    Ad = [{k: (torch.from_numpy(v).to(dev) if isinstance(v, np.ndarray) else v) for k, v in g.items()}
          for g in graphs]
    Bd = [torch.from_numpy(b).to(dev) for b in Bs]
    Cd = [torch.empty((g["m"], K), device=dev) for g in graphs]
    nnz = sum(g.nnz for g in graphs)
    # tune on the largest graph (project autotuner), applied to every graph
    big = int(np.argmax([g.nnz for g in graphs]))
    try:
        tune = ns.autotune(Ad[big], K, ns.NS_F32)
        src = "autotuned on the largest graph"
    except Exception as e:
        tune = ns.tune_default()
        src = f"default ({str(e)[:40]})"
    if args.chunk is not None:
        tune.chunk_nnz = tune.absorb_cap = args.chunk
        src += f", W={args.chunk} by flag"
    else:
        try:  # W timed on the whole batch (untimed tuning, like the dry runs above)
            tune, _ = ns.batch_autotune(Ad, [K] * len(graphs), ns.NS_F32, Bd, Cd, start=tune)
            src += f", W={tune.chunk_nnz} timed on the whole batch"
        except Exception as e:
            src += f" (batch W sweep unavailable: {str(e)[:40]})"
    t0 = time.perf_counter()
    bt = ns.Batch(Ad, [K] * len(graphs), ns.NS_F32, tune)
    plan_s = time.perf_counter() - t0
    stream = torch.cuda.current_stream()
    for _ in range(max(args.warmup, 3)):
        bt.execute(Bd, Cd)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    l0 = ns.launch_count()
    with ClockSampler(0) as clk:
        clk.start()
        e0.record(stream)
        for _ in range(args.steps):
            bt.execute(Bd, Cd)
        e1.record(stream)
        torch.cuda.synchronize()
        clk.stop()
    ms = e0.elapsed_time(e1) / args.steps
    # every graph of the batch against the FP64 oracle (after the timed region)
    errs = [oracle.rel_frobenius(Cd[g].cpu().numpy(), oracle.spmm(graphs[g], Bs[g], threads=threads))
            for g in range(len(graphs))]
    n_touched = sum(int(np.count_nonzero(np.bincount(g["colidx"], minlength=g["n"]))) for g in graphs)
    alg = sum(4 * (g["m"] + 1) + 8 * g.nnz + 4 * g["m"] * K for g in graphs) + 4 * K * n_touched
    hbm, src_pk = _peaks()
    print(json.dumps({
        "metric": "SpMM GFLOP/s (2*nnz*K/s), batched form", "value": 2.0 * nnz * K / (ms * 1e-3) / 1e9,
        "unit": "GFLOP/s", "n_gpus": 1, "steps": args.steps, "warmup": max(args.warmup, 3),
        "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32", "data": "synthetic",
        "config": {"workload": "batched-512-graphs-K64-fp32", "graphs": len(graphs), "nnz": nnz,
                   "step": "one persistent launch (CUDA graph replay) over all graphs",
                   "tune": tune.as_dict(), "tune_source": src, "plan_s": plan_s, **bt.stats()},
        "roofline": {"bound": "hbm", "achieved": alg / (ms * 1e-3) / 1e9, "peak": hbm, "unit": "GB/s",
                     "frac": alg / (ms * 1e-3) / 1e9 / hbm, "traffic": None, "peak_source": src_pk},
        "rel_frobenius_vs_fp64": max(errs), "accuracy": {"max_rel_frobenius_per_graph": max(errs),
                                                          "graphs_checked": len(errs)},
        "gpu_launches": ns.launch_count() - l0,
        "clocks": clk.summary()}))


# ---------------------------------------------------------------------------------------------
# GNN workload: a 2-layer GCN forward for many epochs on the power-law graph, one plan for all
# ---------------------------------------------------------------------------------------------
def bench_gcn(args, threads):
    import torch
    import oracle
    import synth
    import paper_2606_22482_gb300 as ns
    from paper_2606_22482_gb300.gcn import GCN
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(0)
    A, X = synth.config_powerlaw(args.seed)
    K = 128
    At = {k: (torch.from_numpy(v).to(dev) if isinstance(v, np.ndarray) else v) for k, v in A.items()}
    rng = np.random.default_rng(args.seed + 7)
    Ws = [torch.from_numpy((rng.standard_normal((K, K)) / np.sqrt(K)).astype(np.float32)).to(dev)
          for _ in range(2)]
    Xt = torch.from_numpy(X).to(dev)
    stream = torch.cuda.current_stream()
    tune = ns.tune_default()
    tune.tau_tile = ns.NS_TAU_INF
    if args.chunk is not None:
        tune.chunk_nnz = tune.absorb_cap = args.chunk
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
    for _ in range(2):  # pool warm-up
        ns.spmm_plan(At, K, ns.NS_F32, tune).close()
    torch.cuda.synchronize()
    ev[0].record(stream)
    plan = ns.spmm_plan(At, K, ns.NS_F32, tune)
    ev[1].record(stream)
    torch.cuda.synchronize()
    plan_ms = ev[0].elapsed_time(ev[1])
    net = GCN(plan, Ws)
    for _ in range(max(args.warmup, 3)):
        net.forward(Xt)
    torch.cuda.synchronize()
    l0 = ns.launch_count()
    with ClockSampler(0) as clk:
        clk.start()
        ev[2].record(stream)
        for _ in range(args.epochs):
            out = net.forward(Xt)
        ev[3].record(stream)
        torch.cuda.synchronize()
        clk.stop()
    ms_epoch = ev[2].elapsed_time(ev[3]) / args.epochs
    launches = ns.launch_count() - l0
    # the SpMM part alone (same plan, same operands)
    XW = torch.empty((A["n"], K), device=dev)
    torch.matmul(Xt, Ws[0], out=XW)
    C = torch.empty((A["m"], K), device=dev)
    ev[2].record(stream)
    for _ in range(20):
        plan.execute(XW, C)
    ev[3].record(stream)
    torch.cuda.synchronize()
    spmm_ms = ev[2].elapsed_time(ev[3]) / 20
    # parity of the last layer's SpMM on sampled rows: its GEMM input read back from the device
    H1 = torch.relu(C)  # layer-1 output of the run above (same plan, same operands)
    XW2 = torch.matmul(H1, Ws[1])
    plan.execute(XW2, C)
    torch.cuda.synchronize()
    err = oracle.rel_frobenius(C.cpu().numpy(), oracle.spmm(A, XW2.cpu().numpy(), threads=threads))
    plan.close()
    nnz = A.nnz
    total_ms = plan_ms + args.epochs * ms_epoch
    print(json.dumps({
        "metric": "GCN 2-layer forward, epochs/s (one SpMM plan for all epochs)",
        "value": 1e3 / ms_epoch, "unit": "epochs/s", "n_gpus": 1, "steps": args.epochs,
        "warmup": max(args.warmup, 3), "ms_per_step": ms_epoch, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "gcn-2layer-powerlaw-rmat-2^20-K128-fp32", "nnz": nnz, "K": K,
                   "layers": 2, "epochs": args.epochs, "tune": tune.as_dict(),
                   "gemm": "torch.matmul (cuBLAS), FP32 without TF32"},
        "plan_ms": plan_ms, "spmm_ms": spmm_ms,
        "spmm_share_of_epoch": 2 * spmm_ms / ms_epoch,
        "plan_share_of_run": plan_ms / total_ms,
        "spmm_gflops": 2.0 * nnz * K / (spmm_ms * 1e-3) / 1e9,
        "rel_frobenius_vs_fp64": err, "accuracy": {"spmm": "layer-2 SpMM, every row"},
        "gpu_launches": launches, "clocks": clk.summary()}))


# ---------------------------------------------------------------------------------------------
# served form: open-loop Poisson arrivals, continuous batching vs one request at a time
# ---------------------------------------------------------------------------------------------
def _serve_graph_job(args):
    import synth
    n, seed = args
    return synth.serve_graph(int(n), seed=seed)


def make_serve_pool(count: int, seed: int, workers: int):
    """The serving pool: `count` RMAT graphs (lognormal node counts, median 20k, sigma 1.2, at
    most 2M nodes, average degree 16), generated by a spawn-started process pool."""
    import multiprocessing as mp
    from concurrent.futures import ProcessPoolExecutor
    import synth
    sizes = synth.serve_pool_sizes(count, seed)
    jobs = [(int(n), 1000 + i) for i, n in enumerate(sizes)]
    order = np.argsort(-sizes)                   # largest first: the pool finishes together
    out = [None] * count
    with ProcessPoolExecutor(max_workers=max(1, workers), mp_context=mp.get_context("spawn")) as ex:
        for i, g in zip(order, ex.map(_serve_graph_job, [jobs[i] for i in order], chunksize=1)):
            out[i] = g
    return sizes, out


class PinnedPool:
    """Page-locked float32 buffers for results, reused by power-of-two size class."""

    def __init__(self):
        import torch
        self.torch = torch
        self.free = {}

    @staticmethod
    def size_class(n: int) -> int:
        return 1 << (max(1, n) - 1).bit_length()

    def prewarm(self, cls: int, count: int) -> None:
        lst = self.free.setdefault(cls, [])
        while len(lst) < count:
            lst.append(self.torch.empty(cls, dtype=self.torch.float32).pin_memory())

    def get(self, m: int, K: int):
        n = max(1, m * K)
        cls = self.size_class(n)
        lst = self.free.setdefault(cls, [])
        t = lst.pop() if lst else self.torch.empty(cls, dtype=self.torch.float32).pin_memory()
        return t, t.numpy()[:m * K].reshape(m, K)

    def put(self, t):
        self.free.setdefault(t.numel(), []).append(t)


def bench_serve(args, threads):
    import torch
    import oracle
    import paper_2606_22482_gb300 as ns
    t_setup = time.perf_counter()
    sizes, graphs = make_serve_pool(args.pool, args.seed, threads)
    t_pool = time.perf_counter() - t_setup
    torch.cuda.set_device(0)
    rng = np.random.default_rng(args.seed)
    n_req = int(args.rate * args.duration)
    arr = np.cumsum(rng.exponential(1.0 / args.rate, size=n_req))
    req_g = rng.integers(0, len(graphs), size=n_req)
    req_K = rng.choice([32, 64, 128], size=n_req)
    req_bf = rng.integers(0, 2, size=n_req).astype(bool)
    nnz = np.array([g.nnz for g in graphs], dtype=np.int64)
    flops = float((2.0 * nnz[req_g] * req_K).sum())
    # one pinned random block per dtype: the B of a request is its first n x K elements
    max_el = int(max(g["n"] for g in graphs)) * 128
    gen = torch.Generator().manual_seed(args.seed + 7)
    Bf32 = torch.randn(max_el, generator=gen, dtype=torch.float32).pin_memory()
    Bb16 = torch.randn(max_el, generator=gen, dtype=torch.float32).to(torch.bfloat16).pin_memory()
    Bf32_np, Bb16_np = Bf32.numpy(), Bb16.view(torch.int16).numpy().view(np.uint16)

    def b_of(i):
        g, K = int(req_g[i]), int(req_K[i])
        blk = Bb16_np if req_bf[i] else Bf32_np
        return blk[:graphs[g]["n"] * K].reshape(graphs[g]["n"], K)

    check_every = max(1, n_req // args.serve_checks)
    check_rows = {}

    def rows_to_check(i):
        m = graphs[int(req_g[i])]["m"]
        if m <= 2048:
            return np.arange(m, dtype=np.int32)
        return np.sort(np.random.default_rng(i).choice(m, 2048, replace=False)).astype(np.int32)

    pool = PinnedPool()
    # result buffers of about 50 ms of arrivals per size class, page-locked before the trace
    # (pinning memory takes driver locks that would stall the server's threads mid-trace)
    cls_of = np.array([PinnedPool.size_class(graphs[int(g)]["m"] * int(K)) for g, K in zip(req_g, req_K)])
    budget = 24 << 30
    for c in sorted(set(cls_of.tolist())):
        cnt = int((cls_of == c).sum())
        want = min(cnt, max(2, int(np.ceil(args.rate * 0.05 * cnt / n_req))))
        want = min(want, max(1, budget // (4 * c)))
        budget -= want * 4 * c
        pool.prewarm(c, want)
    tune = ns.tune_default()
    sv = ns.Server(hbm_budget_bytes=int(args.serve_budget * (1 << 30)), max_inflight=args.inflight,
                   max_queue=1 << 16, max_graphs=len(graphs) + 16, tune=tune)
    gids = [sv.register(g) for g in graphs]
    # warm: the planner builds every graph's plan once (one plan per graph serves every K and
    # dtype under this tune) and the widest requests (K = 128, FP32) fill the server's device
    # block cache; plans stay resident for the trace
    t_w = ns.now()
    warm = {}
    for g in range(len(graphs)):
        Ct, Cv = pool.get(graphs[g]["m"], 128)
        warm[sv.submit(gids[g], Bf32_np[:graphs[g]["n"] * 128].reshape(-1, 128), Cv, ns.NS_F32)] = Ct
    plan_wait = []
    while warm:
        for tk in list(warm):
            done, st = sv.poll(tk)
            if done:
                pool.put(warm.pop(tk))
                if st["t_planned"] > 0:
                    plan_wait.append(st["t_planned"] - t_w)
        time.sleep(0.0005)
    t_warm = ns.now() - t_w

    # ---- the timed trace ----
    lat = np.zeros(n_req)
    # admission wait, launch, device + copies (host view); then the device part on the GPU's clock:
    # B uploaded, kernel done, C copied, completion seen by the server
    parts = np.zeros((n_req, 7))
    out_rows = {}
    pending = {}
    launches0 = ns.launch_count()
    with ClockSampler(0) as clk:
        clk.start()
        t0 = ns.now()
        i = 0
        while i < n_req or pending:
            now = ns.now() - t0
            while i < n_req and arr[i] <= now:
                g, K, bf = int(req_g[i]), int(req_K[i]), bool(req_bf[i])
                Ct, Cv = pool.get(graphs[g]["m"], K)
                tk = sv.submit(gids[g], b_of(i), Cv, ns.NS_BF16 if bf else ns.NS_F32, t_arrival=t0 + arr[i])
                pending[tk] = (i, Ct, Cv)
                i += 1
            for tk in list(pending):
                done, st = sv.poll(tk)
                if done:
                    j, Ct, Cv = pending.pop(tk)
                    ta = t0 + arr[j]
                    lat[j] = st["t_done"] - ta
                    parts[j] = (st["t_admit"] - ta, st["t_start"] - st["t_admit"], st["t_done"] - st["t_start"],
                                st["t_h2d"] - st["t_start"], st["t_exec"] - st["t_h2d"], st["t_d2h"] - st["t_exec"],
                                st["t_done"] - st["t_d2h"])
                    if j % check_every == 0:
                        r = rows_to_check(j)
                        out_rows[j] = (r, Cv[r].copy())
                    pool.put(Ct)
            time.sleep(0.0001)
        wall = ns.now() - t0
        clk.stop()
    launches = ns.launch_count() - launches0
    sv.close()
    if args.serve_trace:
        np.savez(args.serve_trace, arrival=arr, lat=lat, parts=parts, g=req_g, K=req_K, bf16=req_bf,
                 nodes=np.array([graphs[int(g)]["n"] for g in req_g]))

    # ---- accuracy of the served results (sampled requests, sampled rows) vs the FP64 oracle ----
    errs = {False: [], True: []}
    for j, (r, Cr) in out_rows.items():
        g, bf = int(req_g[j]), bool(req_bf[j])
        ref = oracle.spmm(graphs[g], b_of(j), rows=r, b_bf16=bf, threads=threads)
        errs[bf].append(oracle.rel_frobenius(Cr, ref))

    # ---- the plain path: the first requests of the same trace, one at a time (plan + execute +
    # copies through ns_spmm_host, as a caller without the server would do it) ----
    n_plain = min(n_req, args.plain_requests)
    lat_p = np.zeros(n_plain)
    Cp, Cpv = pool.get(int(max(g["m"] for g in graphs)), 128)
    tp = time.perf_counter()
    for j in range(n_plain):
        now = time.perf_counter() - tp
        if arr[j] > now:
            time.sleep(arr[j] - now)
        g, K, bf = int(req_g[j]), int(req_K[j]), bool(req_bf[j])
        ns.spmm_host(graphs[g], b_of(j), Cp.numpy()[:graphs[g]["m"] * K].reshape(-1, K),
                     ns.NS_BF16 if bf else ns.NS_F32, tune)
        lat_p[j] = time.perf_counter() - tp - arr[j]
    wall_p = time.perf_counter() - tp
    flops_p = float((2.0 * nnz[req_g[:n_plain]] * req_K[:n_plain]).sum())

    pct = lambda a, q: float(np.percentile(a, q) * 1e3) if len(a) else None
    worst = int(np.argmax(lat))
    # size classes as the server forms them: B + C above 32 MB is a bulk request
    io = np.array([graphs[int(g)]["n"] * int(K) * (2 if bf else 4) + graphs[int(g)]["m"] * int(K) * 4
                   for g, K, bf in zip(req_g, req_K, req_bf)], dtype=np.int64)
    bulk = io > (32 << 20)
    by_class = {name: {"share": float(sel.mean()), "p50_ms": pct(lat[sel], 50), "p99_ms": pct(lat[sel], 99),
                       "device_and_copies_p99_ms": pct(parts[sel, 2], 99)}
                for name, sel in (("small", ~bulk), ("bulk", bulk))}
    h2d = float(sum(graphs[int(g)]["n"] * int(K) * (2 if bf else 4) for g, K, bf in zip(req_g, req_K, req_bf)))
    d2h = float(sum(graphs[int(g)]["m"] * int(K) * 4 for g, K in zip(req_g, req_K)))
    all_err = errs[False] + errs[True]
    print(json.dumps({
        "metric": "served SpMM throughput & p50/p99 latency", "value": flops / wall / 1e9,
        "unit": "GFLOP/s", "n_gpus": 1, "steps": n_req, "warmup": len(graphs),
        "ms_per_step": wall / n_req * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "mixed f32/bf16", "data": "synthetic",
        "config": {"workload": f"serve-poisson-{args.rate:g}/s-{args.duration:g}s-pool{args.pool}",
                   "requests": n_req, "K": "{32,64,128}", "b_dtype": "50/50 f32/bf16",
                   "graph_nodes_median": float(np.median(sizes)), "graph_nodes_max": int(sizes.max()),
                   "pool_nnz": int(nnz.sum()), "max_inflight": args.inflight,
                   "hbm_budget_gib": args.serve_budget, "tune": tune.as_dict(),
                   "l2": "every request copies its B in and its C out (host buffers)"},
        "served": {"requests_per_s": n_req / wall, "offered_per_s": args.rate,
                   "p50_ms": pct(lat, 50), "p99_ms": pct(lat, 99), "max_ms": pct(lat, 100),
                   "GFLOP_per_s": flops / wall / 1e9,
                   "breakdown_p50_ms": {"admission_wait": pct(parts[:, 0], 50), "launch": pct(parts[:, 1], 50),
                                        "device_and_copies": pct(parts[:, 2], 50)},
                   "breakdown_p99_ms": {"admission_wait": pct(parts[:, 0], 99), "launch": pct(parts[:, 1], 99),
                                        "device_and_copies": pct(parts[:, 2], 99)},
                   "device_breakdown_p99_ms": {"h2d_after_launch": pct(parts[:, 3], 99), "execute": pct(parts[:, 4], 99),
                                               "d2h": pct(parts[:, 5], 99), "seen_by_server": pct(parts[:, 6], 99)},
                   "slowest_request": {"ms": lat[worst] * 1e3, "nodes": int(graphs[int(req_g[worst])]["n"]),
                                       "K": int(req_K[worst]), "bf16": bool(req_bf[worst]),
                                       "parts_ms": dict(zip(["admission_wait", "launch", "device_and_copies",
                                                             "h2d_after_launch", "execute", "d2h", "seen_by_server"],
                                                            [float(x * 1e3) for x in parts[worst]]))},
                   "first_n_p50_ms": pct(lat[:n_plain], 50), "first_n_p99_ms": pct(lat[:n_plain], 99),
                   "by_size_class": by_class},
        "plain": {"requests": n_plain, "requests_per_s": n_plain / wall_p, "p50_ms": pct(lat_p, 50),
                  "p99_ms": pct(lat_p, 99), "GFLOP_per_s": flops_p / wall_p / 1e9,
                  "how": "the first requests of the trace, one at a time through ns_spmm_host"},
        "planning": {"graphs": len(graphs), "warm_s": t_warm, "pool_generation_s": t_pool,
                     "plan_ready_p50_s": float(np.median(plan_wait)) if plan_wait else None},
        "rel_frobenius_vs_fp64": max(all_err) if all_err else None,
        "accuracy": {"f32_max": max(errs[False]) if errs[False] else None,
                     "bf16_max": max(errs[True]) if errs[True] else None,
                     "requests_checked": len(all_err),
                     "rows": "all rows of graphs up to 2048 nodes, else 2048 sampled rows"},
        "e2e": {"value": flops / wall / 1e9, "unit": "GFLOP/s", "h2d_bytes_per_step": h2d / n_req,
                "d2h_bytes_per_step": d2h / n_req},
        "gpu_launches": int(launches),
        "clocks": clk.summary(),
    }))


if __name__ == "__main__":
    main()

#!/usr/bin/env python3
"""Benchmark: local approximate GP predictions per second on one GB300.

Workload (the paper-scale 2-d problem, Sec. 3.4/4.1 scale): design N=40000 uniform on
[-2,2]^2 with z = x1 exp(-x1^2 - x2^2), 10000 predictive locations on a 100x100 grid
over [-1.97,1.97]^2, lengthscale d=0.5, nugget g=1e-6, n0=6 -> n=50 by ALC over the
1000 nearest candidates.  One step = the whole path for all 10000 locations: kernel (a)
(candidate sets) then kernels (b)+(c) (greedy design + predictive equations).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--precision both|fp64|mixed]
  python bench.py --impl reference ...   # the CPU oracle on host cores (a baseline)

The headline value is the mixed-precision path (float-float screen, FP64 decisions and
predictions); the plain FP64 path is timed in the same run and reported under
"variants".  Prints one JSON line.  Under torchrun every rank runs the full workload on its own GPU
(independent problems, no collective on the data path: weak scaling); `value` is all
ranks' predictions over the slowest rank's time.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "local-GP predictions/sec (n=50, 1000 cand) FP64 plain vs mixed; serving p99 ms"
UNIT = "predictions/s"
FP64_PEAK_TFLOPS_DERIVED = 152 * 2 * 2 * 2.07e9 / 1e12   # SMs x DFMA/clk x 2 flop x max clock
# FP64 ALC screens in 64-bit fixed point: three 32 x 32 + 64-bit multiply-adds (8 lanes per clock
# and SM sub-partition) do a term's two flops
FX_PEAK_TFLOPS_DERIVED = 152 * 32 * 2.07e9 / 3 * 2 / 1e12
EXP_FLOPS = 20      # FP64 flops counted per double-precision exp (measured: about 20 DFMA each)


def kernel_source_hash(unit: str | None = None) -> str:
    """sha256 over CUDA sources with their comments and blank space removed: DRAM counters
    recorded for another revision of a kernel's code are stale (the sources hold no string
    literal with a comment marker).  unit: a translation unit of the library (such as
    "select_mixed.cu"), hashed with the local headers it includes, transitively; None:
    every source of the library."""
    import hashlib
    import re
    h = hashlib.sha256()
    dirs = [os.path.join(ROOT, "paper_1303_0383_gb300", "csrc"), os.path.join(ROOT, "include")]

    def find(fn):
        for d in dirs:
            if os.path.isfile(os.path.join(d, fn)):
                return os.path.join(d, fn)
        return None

    if unit is None:
        files = [(fn, os.path.join(dirs[0], fn)) for fn in sorted(os.listdir(dirs[0]))]
    else:
        seen, todo = {}, [unit]
        while todo:
            fn = todo.pop()
            path = find(fn)
            if fn in seen or path is None:
                continue
            seen[fn] = path
            todo += re.findall(r'^\s*#\s*include\s+"([^"]+)"', open(path, encoding="utf-8").read(),
                               flags=re.M)
        files = sorted(seen.items())
    for fn, path in files:
        src = open(path, encoding="utf-8").read()
        src = re.sub(r"/\*.*?\*/", " ", src, flags=re.S)
        src = re.sub(r"//[^\n]*", "", src)
        code = "\n".join(" ".join(line.split()) for line in src.splitlines() if line.strip())
        h.update(fn.encode())
        h.update(code.encode())
    return h.hexdigest()


def env_rank():
    return int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")), \
        int(os.environ.get("LOCAL_RANK", "0"))


def select_flops_per_location(n0, n, M, p, method="alc"):
    """Algorithmic FP64 flops of the O(j)-per-candidate greedy design for one location:
    every candidate still in the pool at step j (j = 0..n-2) costs 2j (the Cholesky-row
    dot) + 3p (squared distance) + 1 + EXP_FLOPS (its correlation to the new point)
    + 7 (new row entry, v and cov updates, ALC score); plus 3p + 1 + EXP_FLOPS per
    candidate for K(x, c) at the start."""
    total = M * (3 * p + 1 + EXP_FLOPS)
    for j in range(n - 1):
        pool = M - (j + 1)
        total += pool * (2 * j + 3 * p + 1 + EXP_FLOPS + 7)
    return float(total)


FP32_PEAK_TOPS_DERIVED = 152 * 128 * 2.07e9 / 1e12   # SMs x FP32 lanes/clk x max clock


def mixed_fp32_ops_per_location(n0, n, M, p):
    """FP32 operations (add, multiply or fused multiply-add, each one) of the float-float
    screen for one location: every pool candidate at step j costs 12j + 6 (the compensated
    row dot: TwoProd with cross terms and TwoSum per term, one renormalisation) + 20p + 3
    (squared distance of coordinates pre-scaled by 1/sqrt(theta)) + 66 (float-float
    exponential) + 9 (new row entry) + 42 (v and cov updates) + 6 (screen score)."""
    total = 0
    for j in range(n - 1):
        pool = M - (j + 1)
        total += pool * (12 * j + 6 + 20 * p + 3 + 66 + 9 + 42 + 6)
    return float(total)


def mspe_mixed_fp32_ops_per_location(n0, n, M, p):
    """FP32 operations of the float-float MSPE screen for one location: every pool
    candidate at step j costs 36j + 18 (three compensated row dots, u_s.u_c, u_s.ud_c and
    q_j.u_c) + 20p + 3 (squared distance) + 11 (scaling by 1/theta) + 66 (exponential) + 14
    (Kd(s, c)) + 18 (two new row entries) + 42 (v and cov) + 75 (the four derivative sums)
    + 170 (J(c): four float-float divisions, eight products, six sums) + 6 (tracking)."""
    total = 0
    for j in range(n - 1):
        pool = M - (j + 1)
        total += pool * (36 * j + 18 + 20 * p + 3 + 11 + 66 + 14 + 18 + 42 + 75 + 170 + 6)
    return float(total)


def factor_stream_bytes_per_location(n, M):
    """Bytes of candidate factor rows the screen reads for one location: every pool
    candidate at step j reads its j float-float entries (8 bytes each)."""
    return float(sum((M - (j + 1)) * j * 8 for j in range(n - 1)))


def paper_form_flops_per_location(n0, n, M):
    """The paper's O(j^2)-per-candidate form (K_j^{-1} times K(X_j, X_cand) every step)."""
    return float(sum(2 * j * j * (M - j) for j in range(n0, n)))


def dense_flops_per_location(n0, n, M, p):
    """Algorithmic FP64 flops of the paper's explicit-inverse form (lagp_select_dense_dev)
    for one location: every pool candidate at a greedy step with j design points costs
    j(j+1) (the quadratic form k_j(c)^T K_j^{-1} k_j(c) over the upper triangle, FMA = 2)
    + 2j (its dot with K_j^{-1} k_j(x)) + 4 (v, cov, score); every step adds 6j^2 (K_j^{-1}
    k_j(x), K_j^{-1} k_j(s) and the partition inverse update) and, but for the last,
    3p + 1 + EXP_FLOPS per candidate for the new point's correlations; plus 3p + 1 +
    EXP_FLOPS per candidate for K(x, c) at the start."""
    total = M * (3 * p + 1 + EXP_FLOPS)
    for j in range(n):
        if j >= n0:
            total += (M - j) * (j * (j + 1) + 2 * j + 4)
        total += 6 * j * j
        if j + 1 < n:
            total += M * (3 * p + 1 + EXP_FLOPS)
    return float(total)


def mspe_flops_per_location(n0, n, M, p):
    """Algorithmic FP64 flops of the MSPE design in the Cholesky basis for one location:
    every pool candidate at step j costs 6j (three j-dots: u_c, its derivative row and the
    Q-row product) + 3p + 1 + EXP_FLOPS (its correlation to the new point) + 40 (entries,
    v, the derivative terms and J(c)); plus O(j^2) per step for the new rows of L^-1, Q, R."""
    total = M * (3 * p + 1 + EXP_FLOPS)
    for j in range(n - 1):
        pool = M - (j + 1)
        total += pool * (6 * j + 3 * p + 1 + EXP_FLOPS + 40) + 6 * j * j
    return float(total)


# The single-design workloads: generator, the (method, precision) variants timed, the
# headline variant, the CPU-oracle sample size (about 10-30 s of work on 16 cores), the
# untimed oracle sample for the accuracy of another method's variants, and the paper's own
# rate for the same problem where it gives one.
def _workloads():
    from paper_1303_0383_gb300 import inputs
    return {
        "paper-2d": dict(make=inputs.paper_2d, variants=[("alc", "fp64"), ("alc", "mixed")],
                         head=("alc", "mixed"), cpu=1600, paper=None),
        "smooth-8d": dict(make=inputs.smooth_8d, variants=[("alc", "fp64"), ("alc", "mixed"), ("mspe", "fp64"),
                                                            ("mspe", "mixed")],
                          head=("alc", "mixed"), cpu=120, acc_other=64, paper=None),
        "grid-2d": dict(make=inputs.grid_2d, variants=[("alc", "fp64"), ("alc", "mixed"), ("mspe", "fp64"), ("mspe", "mixed"), ("nn", "fp64")],
                        head=("alc", "mixed"), cpu=1600,
                        paper={"value": 10000 / 30.0, "what": "Sec. 4.1: about 30 s for 10K locations, "
                               "40K-point 2-d design, ALC, n=50, fixed theta, 8 threads on a 4-core iMac"}),
        "borehole": dict(make=lambda: inputs.borehole(4000, 500),
                         variants=[("alc", "fp64"), ("alc", "mixed"), ("mspe", "fp64"), ("mspe", "mixed"), ("nn", "fp64")],
                         head=("alc", "mixed"), cpu=500,
                         paper={"value": 500 / 23.2, "what": "Table 1 alc.nomle: 23.2 s for 500 locations "
                                "(fit + predict), N=4000, n=50, 8 threads on a 4-core iMac"}),
        "borehole-8000": dict(make=lambda: inputs.borehole(8000, 1000),
                              variants=[("alc", "fp64"), ("alc", "mixed"), ("mspe", "fp64"), ("mspe", "mixed"), ("nn", "fp64")],
                              head=("alc", "mixed"), cpu=1000,
                              paper={"value": 1000 / 45.1, "what": "Table SM.1 alc.nomle: 45.1 s for 1000 "
                                     "locations (fit + predict), N=8000, n=50, 8 threads on a 4-core iMac"}),
    }


def vkey(method, prec):
    return prec if method == "alc" else "%s_%s" % (method, prec)


class ClockSampler:
    """nvidia-smi clock/throttle sampling during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        import tempfile
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), "--query-gpu=" + self.FIELDS,
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None
        time.sleep(0.3)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.2)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                rows.append((float(parts[1]), float(parts[2]), parts[5:9], float(parts[3])))
            except ValueError:
                continue
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i, v in enumerate(r[2]) if v == "Active"})
        counts = {nm: sum(1 for r in rows if r[2][i] == "Active") for i, nm in enumerate(names)}
        return {"sm_mhz": statistics.median(r[0] for r in rows),
                "sm_max_mhz": max(r[1] for r in rows), "reasons": reasons,
                "reason_samples": {k: v for k, v in counts.items() if v},
                "samples": len(rows), "power_w_max": max(r[3] for r in rows)}


def cpu_oracle_sample(w, n_loc: int, seed: int = 0, method: str = "alc"):
    """Times the CPU oracle (as it stands) on a seeded sample of the workload's locations.
    Returns (locations per second, cores, seconds, the sample's location indices, the
    oracle's outputs for them)."""
    import oracle
    oracle.build()
    locs = np.sort(np.random.default_rng(seed).choice(w.T, size=n_loc, replace=False))
    cores = os.cpu_count() or 1
    t0 = time.perf_counter()
    r = oracle.predict(w.X, w.Z, w.XX[locs], w.n0, w.n, w.ncand, w.d, w.g, method, nthreads=cores)
    dt = time.perf_counter() - t0
    assert (r["status"] == 0).all()
    return n_loc / dt, cores, dt, locs, r


def accuracy_vs_oracle(w, locs, ora, r, method, prec):
    """The parity protocol of the tests (oracle/parity.py) on the oracle's sample: errors of
    mean, s2 and var against the FP64 oracle along the GPU's path, selection match rate,
    forced paths and near-tie steps, values admitted by each adjudication clause; for the
    mixed screens, the FP64 re-score passes of the last timed call (all locations)."""
    from oracle.parity import check_sample
    gpu = {"idx": r["idx_np"], "mean": r["mean"], "s2": r["s2"], "var": r["var"]}
    out = check_sample(w, list(locs), ora, gpu, method)
    out["sample"] = "%d seeded locations of the %d" % (len(locs), w.T)
    if prec == "mixed" and method != "nn":
        out["fp64_rescore_passes"] = r["rescores"]
        out["fp64_rescore_fraction_of_steps"] = r["rescores"] / float(w.T * (w.n - w.n0))
    return out


def run_reference(args):
    rank, world, _ = env_rank()
    if rank != 0:
        return 0
    from paper_1303_0383_gb300 import inputs
    w = inputs.paper_2d()
    sample = args.ref_sample
    for _ in range(args.warmup):
        cpu_oracle_sample(w, max(8, sample // 8), seed=999)
    times = []
    cores = os.cpu_count() or 1
    for k in range(args.steps):
        _, cores, dt, _, _ = cpu_oracle_sample(w, sample, seed=k)
        times.append(dt)
    value = sample * len(times) / sum(times)
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * sum(times) / len(times), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": w.name, "N": w.N, "p": w.p, "T": w.T, "n0": w.n0, "n": w.n,
                   "ncand": w.ncand, "d": w.d, "g": w.g, "method": "alc",
                   "step": "oracle on a seeded sample of %d of the %d locations" % (sample, w.T)},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": "%d seeded locations per step of the %d" % (sample, w.T)},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def e2e_timing(args, w, M, method, prec, flush, idx_dev):
    """Host entry point lagp_predict with pinned host buffers: the copy of XX in and of
    every output back are inside each timed call."""
    import torch
    from paper_1303_0383_gb300 import lagp
    T = w.XX.shape[0]
    design = lagp.Design(w.X, w.Z)
    XXh = torch.empty((T, w.p), dtype=torch.float64, pin_memory=True).numpy()
    XXh[:] = w.XX
    outh = dict(mean=torch.empty(T, dtype=torch.float64, pin_memory=True).numpy(),
                s2=torch.empty(T, dtype=torch.float64, pin_memory=True).numpy(),
                var=torch.empty(T, dtype=torch.float64, pin_memory=True).numpy(),
                idx=torch.empty((T, w.n), dtype=torch.int32, pin_memory=True).numpy(),
                status=torch.empty(T, dtype=torch.int8, pin_memory=True).numpy())
    for _ in range(max(1, args.warmup)):
        design.predict(XXh, w.n0, w.n, M, w.d, w.g, method, prec, out=outh)
    times = []
    for _ in range(args.steps):
        flush.add_(1.0)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        design.predict(XXh, w.n0, w.n, M, w.d, w.g, method, prec, out=outh)
        times.append(time.perf_counter() - t0)
    design.close()
    assert np.array_equal(outh["idx"], idx_dev.cpu().numpy()), "host and device paths disagree"
    return 1e3 * sum(times) / len(times)


def time_precision(args, w, prec, X, Z, XX, flush, stream, lagp, torch, method="alc"):
    """Warm up, then time args.steps steps of kernel (a) + kernels (b)+(c) with CUDA events
    per kernel on the launching stream (L2 flushed between steps, outside the events)."""
    dev = X.device
    T, M = w.T, w.ncand
    cand = torch.empty((T, M), dtype=torch.int32, device=dev)
    mean = torch.empty(T, dtype=torch.float64, device=dev)
    s2, var = torch.empty_like(mean), torch.empty_like(mean)
    idx = torch.empty((T, w.n), dtype=torch.int32, device=dev)
    status = torch.empty(T, dtype=torch.int8, device=dev)
    ws_knn = lagp.workspace(lagp.lagp_knn_workspace_bytes(w.N, T, M), dev)
    ws_sel = lagp.workspace(lagp.lagp_select_workspace_bytes(T, w.p, w.n, M, method, prec), dev)

    def step(evs=None):
        if evs:
            evs[0].record(stream)
        lagp.lagp_knn_dev(X, XX, M, cand, ws_knn, stream)
        if evs:
            evs[1].record(stream)
        lagp.lagp_select_dev(X, Z, XX, cand, w.n0, w.n, w.d, w.g, method, prec, mean, s2, var,
                             idx, status, ws_sel, stream)
        if evs:
            evs[2].record(stream)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    assert int((status != 0).sum()) == 0, "failed locations in warm-up"
    launches0 = lagp.lagp_launch_count()
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(3)] for _ in range(args.steps)]
    barrier(torch)
    for k in range(args.steps):
        flush.add_(1.0)                 # evict L2 between timed steps (not timed)
        step(evs[k])
    barrier(torch)
    launches = lagp.lagp_launch_count() - launches0
    knn_ms = [e[0].elapsed_time(e[1]) for e in evs]
    sel_ms = [e[1].elapsed_time(e[2]) for e in evs]
    step_ms = [a + b for a, b in zip(knn_ms, sel_ms)]
    rescores = lagp.lagp_select_rescore_count(ws_sel, method, prec, stream)
    return dict(ms=sum(step_ms) / len(step_ms), knn_ms=sum(knn_ms) / len(knn_ms),
                sel_ms=sum(sel_ms) / len(sel_ms), launches=int(launches), idx=idx,
                idx_np=idx.cpu().numpy(), mean=mean.cpu().numpy(), s2=s2.cpu().numpy(),
                var=var.cpu().numpy(), rescores=rescores)


def max_over_ranks(values, device=None):
    """Element-wise maximum of a list of floats over the ranks of the process group (the
    slowest rank's time is the job's); the values themselves when not distributed."""
    import torch
    if not (torch.distributed.is_available() and torch.distributed.is_initialized()):
        return [float(v) for v in values]
    t = torch.tensor([float(v) for v in values], dtype=torch.float64,
                     device=device if device is not None else "cpu")
    torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
    return [float(v) for v in t.cpu()]


def barrier(torch):
    if torch.distributed.is_available() and torch.distributed.is_initialized():
        torch.distributed.barrier()
    if torch.cuda.is_available():
        torch.cuda.synchronize()


FP32_FMA_PEAK_TFLOPS_DERIVED = 152 * 128 * 2 * 2.07e9 / 1e12   # SMs x FP32 lanes x 2 flop x max clock


def roofline_for(prec, w, sel_ms, traffic, method="alc"):
    """Roofline of kernels (b)+(c) for one launch over all T locations.  "frac" is always
    the method's algorithmic work (FP64-equivalent flops of the O(j)-per-candidate design:
    FMA = 2, exp = 20) per second of the launch against the peak of the pipe that does
    it: FP64 DFMA for the FP64 MSPE kernel, integer multiply-adds for the fixed-point screen of
    FP64 ALC, FP32 FMA for the mixed screens (which carry that
    work in float-float on the FP32 pipes).  For the mixed screens "issued" gives the
    second figure: the FP32 operations the float-float arithmetic actually issues, against
    the FP32 lane peak (one operation per lane-cycle)."""
    T, M = w.T, w.ncand
    if method == "nn":
        return None  # no scoring: kernels (b)+(c) only evaluate the predictive equations
    alg = (mspe_flops_per_location if method == "mspe" else select_flops_per_location)(
        w.n0, w.n, M, w.p)
    achieved = alg * T / (sel_ms / 1e3) / 1e12
    name = {("alc", "fp64"): "select_mixed_kernel, fixed point", ("alc", "mixed"): "select_mixed_kernel",
            ("mspe", "fp64"): "select_mspe_kernel",
            ("mspe", "mixed"): "select_mspe_mixed_kernel"}[(method, prec)]
    out = {"kernel": name + " (kernels b+c)", "bound": "alu", "achieved": achieved,
           "unit": "TFLOP/s", "traffic": traffic, "work_per_location": alg,
           "work_unit": "FP64-equivalent flops of the O(j)-per-candidate design (FMA = 2, exp = 20)"}
    if prec == "fp64" and method == "alc":
        out.update(peak=FX_PEAK_TFLOPS_DERIVED, frac=achieved / FX_PEAK_TFLOPS_DERIVED,
                   peak_source="derived integer: 152 SMs x 32 IMAD.WIDE lanes x 2.07 GHz, 3 per FMA")
        return out
    if prec == "fp64":
        out.update(peak=FP64_PEAK_TFLOPS_DERIVED, frac=achieved / FP64_PEAK_TFLOPS_DERIVED,
                   peak_source="derived FP64: 152 SMs x 2 DFMA/clk x 2 flop x 2.07 GHz")
        return out
    out.update(peak=FP32_FMA_PEAK_TFLOPS_DERIVED, frac=achieved / FP32_FMA_PEAK_TFLOPS_DERIVED,
               peak_source="derived FP32: 152 SMs x 128 FMA lanes x 2 flop x 2.07 GHz; the work "
                           "runs in float-float on these pipes")
    ops = (mspe_mixed_fp32_ops_per_location if method == "mspe" else mixed_fp32_ops_per_location)(
        w.n0, w.n, M, w.p)
    issued = ops * T / (sel_ms / 1e3) / 1e12
    streams = 2 if method == "mspe" else 1
    out["issued"] = {"achieved": issued, "peak": FP32_PEAK_TOPS_DERIVED, "unit": "T op/s",
                     "frac": issued / FP32_PEAK_TOPS_DERIVED, "work_per_location": ops,
                     "work_unit": "FP32 operations the float-float screen issues (add, mul or FMA = 1)",
                     "peak_source": "derived FP32: 152 SMs x 128 lanes x 2.07 GHz (one operation per lane-cycle)",
                     "fp32_ops_per_algorithmic_flop": ops / alg}
    out["factor_stream_tbs"] = streams * factor_stream_bytes_per_location(w.n, M) * T / (sel_ms / 1e3) / 1e12
    out["factor_stream_note"] = "factor-row bytes read per second (shared memory + L2 + DRAM), kernels (b)+(c) time"
    return out


def stored_traffic(prec):
    tpath = os.path.join(ROOT, "profiles", "select_traffic.json")
    if not os.path.exists(tpath):
        return None
    try:
        for tj in json.load(open(tpath)).get("entries", []):
            if tj.get("precision") == prec and \
                    tj.get("source_sha256") == kernel_source_hash(tj.get("unit")):
                return tj.get("bytes_per_launch")
    except Exception:
        return None
    return None


def time_stagewise(args, w, method, prec, stages, X, Z, XX, flush, stream, lagp, torch):
    """The stagewise scheme of Sec. 4.2 (lagp.predict_stagewise's calls, with CUDA events
    between them): candidates, design at theta0, local MLE, stages-1 times (design at the
    estimates, MLE), predictive equations on the last design.  Returns timings, the
    outputs of the last step and the mean Newton iterations."""
    dev = X.device
    T, M, n, N, p = w.T, w.ncand, w.n, w.N, w.p
    tmin, tmax = w.d / 100.0, w.d * 100.0
    f64, i32 = torch.float64, torch.int32
    cand = torch.empty((T, M), dtype=i32, device=dev)
    mean = torch.empty(T, dtype=f64, device=dev)
    s2, var = torch.empty_like(mean), torch.empty_like(mean)
    idx = torch.empty((T, n), dtype=i32, device=dev)
    status = torch.empty(T, dtype=torch.int8, device=dev)
    mst = torch.empty(T, dtype=torch.int8, device=dev)
    theta = torch.empty(T, dtype=f64, device=dev)
    th1 = torch.empty_like(theta)
    iters = torch.empty(T, dtype=i32, device=dev)
    ws_knn = lagp.workspace(lagp.lagp_knn_workspace_bytes(N, T, M), dev)
    ws_sel = lagp.workspace(lagp.lagp_select_workspace_bytes(T, p, n, M, method, prec), dev)
    ws_mle = lagp.workspace(lagp.lagp_mle_workspace_bytes(T, n), dev)
    ws_pr = lagp.workspace(lagp.lagp_design_predict_workspace_bytes(T, n), dev)
    it_sum = [0]

    def step(evs=None):
        marks = []
        rec = (lambda: marks.append(torch.cuda.Event(enable_timing=True)) or marks[-1].record(stream)) \
            if evs is not None else (lambda: None)
        rec()
        lagp.lagp_knn_dev(X, XX, M, cand, ws_knn, stream)
        rec()
        lagp.lagp_select_dev(X, Z, XX, cand, w.n0, n, w.d, w.g, method, prec, mean, s2, var, idx,
                             status, ws_sel, stream)
        rec()
        lagp.lagp_mle_dev(X, Z, idx, w.d, w.g, tmin, tmax, theta, iters, mst, 100, 1e-8, ws_mle,
                          stream)
        rec()
        for _ in range(stages - 1):
            th1.copy_(theta)
            lagp.lagp_select_theta_dev(X, Z, XX, cand, w.n0, n, th1, w.g, method, prec, mean, s2,
                                       var, idx, status, ws_sel, stream)
            rec()
            lagp.lagp_mle_dev(X, Z, idx, th1, w.g, tmin, tmax, theta, iters, mst, 100, 1e-8,
                              ws_mle, stream)
            rec()
        lagp.lagp_design_predict_dev(X, Z, XX, idx, theta, w.g, mean, s2, var, status, ws_pr,
                                     stream)
        rec()
        if evs is not None:
            evs.append(marks)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    assert int((status != 0).sum()) == 0 and int((mst != 0).sum()) == 0, "failed locations"
    launches0 = lagp.lagp_launch_count()
    evs = []
    barrier(torch)
    for k in range(args.steps):
        flush.add_(1.0)
        step(evs)
    barrier(torch)
    launches = lagp.lagp_launch_count() - launches0
    names = ["knn", "select", "mle"]
    for k in range(2, stages + 1):
        names += ["select_theta_%d" % k, "mle_%d" % k]
    names.append("predict")
    kern = {nm: sum(m[i].elapsed_time(m[i + 1]) for m in evs) / len(evs) for i, nm in enumerate(names)}
    ms = sum(kern.values())
    return dict(ms=ms, kernels_ms=kern, launches=int(launches), idx=idx,
                mean=mean.cpu().numpy(), s2=s2.cpu().numpy(),
                newton_iters=float(iters.double().mean()))


def accuracy(w, mean, s2):
    """Out-of-sample accuracy against the known response at XX (the paper's Sec. 5 metrics):
    RMSE, sqrt(1 - NSE) = sd(error) / sd(response), and the coverage of the 95% Student-t
    interval with n degrees of freedom."""
    if w.ZZ is None:
        return None
    from scipy import stats
    err = mean - w.ZZ
    q = stats.t.ppf(0.975, w.n)
    cover = float(np.mean(np.abs(err) <= q * np.sqrt(s2)))
    return {"rmse": float(np.sqrt(np.mean(err ** 2))),
            "sqrt_1_minus_nse": float(np.std(err) / np.std(w.ZZ)), "coverage95": cover}


# The paper's rates for its stagewise rows (with local MLE), where it states the
# predictive-set size: Table 1 (borehole N=4000, 500 locations) and Table SM.1 (N=8000,
# 1000 locations), seconds for fit + predict on 8 threads of a 4-core iMac.
PAPER_STAGEWISE = {("borehole", 1): 500 / 23.5, ("borehole", 2): 500 / 46.3,
                   ("borehole-8000", 1): 1000 / 46.2, ("borehole-8000", 2): 1000 / 92.3}


def print_stagewise(args, w, spec, variants, clocks, world):
    head = spec["head"]
    hk = vkey(head[0] + (str(args.stages) if args.stages > 1 else "") + "_mle", head[1])
    if hk not in variants:
        hk = next(iter(variants))
    paper = PAPER_STAGEWISE.get((args.workload, args.stages))
    line = {
        "metric": "local-GP predictions/sec, stagewise scheme with local MLE (Sec. 4.2), %d stage(s)"
                  % args.stages,
        "value": variants[hk]["value"], "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": variants[hk]["ms_per_step"], "higher_is_better": True,
        "scaling": "weak", "vs_baseline": variants[hk]["value"] / paper if paper else None,
        "dtype": "f64" if head[1] == "fp64" else "f32x2+f64", "data": "synthetic",
        "config": {"workload": w.name, "N": w.N, "p": w.p, "T": w.T, "n0": w.n0, "n": w.n,
                   "ncand": w.ncand, "theta0": w.d, "g": w.g, "tmin": w.d / 100, "tmax": w.d * 100,
                   "stages": args.stages, "l2": "flushed between timed steps (256 MB write)"},
        "clocks": clocks, "gpu_launches": variants[hk]["gpu_launches"], "variants": variants,
    }
    if paper:
        line["paper_context"] = {"value": paper, "unit": UNIT,
                                 "what": "the paper's %s row (fit + predict, 8 threads, 4-core iMac)"
                                         % (head[0] + ("2" if args.stages == 2 else ""))}
    print(json.dumps(line), flush=True)
    return 0


def _with(args, **kw):
    a = argparse.Namespace(**vars(args))
    for k, v in kw.items():
        setattr(a, k, v)
    return a


def measure_single(args, wname, steps, warmup, e2e, cpu_n, acc_n_other, world=1, rank=0,
                   locations=0):
    """One single-design workload, every (method, precision) variant of it: kernel (a) +
    kernels (b)+(c) timed per step with CUDA events on the launching stream (L2 flushed
    between steps), the host entry point lagp_predict timed end to end, clocks sampled
    during the timed region.  Then (rank 0) the CPU oracle is timed on a seeded sample
    (cpu_n locations, all host cores: the cpu_baseline) and every variant's outputs are
    checked against the oracle's on that sample (variants of another method: an untimed
    sample of acc_n_other locations).  Returns the line's pieces."""
    import torch
    from paper_1303_0383_gb300 import lagp
    spec = _workloads()[wname]
    w = spec["make"]()
    if locations:
        w.XX = np.ascontiguousarray(w.XX[:locations])
        if w.ZZ is not None:
            w.ZZ = w.ZZ[:locations]
        w.name += " (first %d locations)" % locations
    variants_run = [v for v in spec["variants"] if args.precision == "both" or v[1] == args.precision]
    head = spec["head"] if spec["head"] in variants_run else variants_run[0]
    dev = torch.device("cuda", torch.cuda.current_device())
    stream = torch.cuda.current_stream()
    X, Z, XX = (torch.as_tensor(a).to(dev) for a in (w.X, w.Z, w.XX))
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)  # > L2
    a2 = _with(args, steps=steps, warmup=warmup)
    sampler = ClockSampler(int(os.environ.get("CUDA_VISIBLE_DEVICES", "0").split(",")[0])
                           if os.environ.get("CUDA_VISIBLE_DEVICES", "").isdigit()
                           else torch.cuda.current_device())
    sampler.start()
    res = {}
    for method, prec in variants_run:
        k = vkey(method, prec)
        res[k] = time_precision(a2, w, prec, X, Z, XX, flush, stream, lagp, torch, method=method)
        # e2e: the host C ABI (lagp_predict) with pinned host buffers, copies inside the region
        res[k]["e2e_ms"] = e2e_timing(a2, w, w.ncand, method, prec, flush, res[k]["idx"]) \
            if e2e else float("nan")
    clocks = sampler.stop()
    del flush
    if world > 1:
        for r in res.values():
            r["ms"], r["e2e_ms"], r["sel_ms"] = max_over_ranks([r["ms"], r["e2e_ms"], r["sel_ms"]], dev)
    if rank != 0:
        return None
    variants = {}
    for method, prec in variants_run:
        k = vkey(method, prec)
        r = res[k]
        variants[k] = {
            "method": method, "precision": prec,
            "value": world * w.T / (r["ms"] / 1e3), "ms_per_step": r["ms"],
            "kernels_ms": {"knn": r["knn_ms"], "select": r["sel_ms"]},
            "e2e": {"value": world * w.T / (r["e2e_ms"] / 1e3) if r["e2e_ms"] == r["e2e_ms"] else None,
                    "ms_per_step": r["e2e_ms"]},
            "gpu_launches": r["launches"],
            "roofline": roofline_for(prec, w, r["sel_ms"],
                                     stored_traffic(prec) if (method == "alc" and wname == "paper-2d"
                                                              and not locations) else None,
                                     method=method),
            "accuracy": accuracy(w, r["mean"], r["s2"]),
        }
    cpu = {"value": None, "cores": None, "seconds": 0.0, "n": 0}
    if cpu_n:
        n_cpu = min(cpu_n, w.T)
        val, cores, dt, locs, ora = cpu_oracle_sample(w, n_cpu, method=head[0])
        cpu = {"value": val, "cores": cores, "seconds": dt, "n": n_cpu}
        samples = {head[0]: (locs, ora)}
        for method, prec in variants_run:
            if method not in samples:
                n_o = min(acc_n_other, w.T)
                _, _, _, l2, o2 = cpu_oracle_sample(w, n_o, seed=1, method=method)
                samples[method] = (l2, o2)
            locs_m, ora_m = samples[method]
            variants[vkey(method, prec)]["accuracy_vs_oracle"] = accuracy_vs_oracle(
                w, locs_m, ora_m, res[vkey(method, prec)], method, prec)
    return dict(w=w, spec=spec, head=head, res=res, variants=variants, clocks=clocks, cpu=cpu)


def run_gpu(args):
    import torch
    rank, world, local = env_rank()
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    from paper_1303_0383_gb300 import lagp
    lagp.load()
    if args.stages:
        return run_stagewise(args, world, rank)
    spec = _workloads()[args.workload]
    m = measure_single(args, args.workload, args.steps, args.warmup, not args.no_e2e,
                       0 if args.no_cpu else (args.cpu_sample or spec["cpu"]),
                       spec.get("acc_other", 64), world, rank, args.locations)
    if rank != 0:
        if world > 1:
            torch.distributed.destroy_process_group()
        return 0
    w, head, res, variants = m["w"], m["head"], m["res"], m["variants"]
    T = w.T
    h2d = T * w.p * 8
    d2h = T * (8 * 3 + 4 * w.n + 1)
    hk = vkey(*head)
    H = res[hk]
    paper = m["spec"]["paper"]
    line = {
        "metric": METRIC, "value": variants[hk]["value"], "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": H["ms"],
        "higher_is_better": True, "scaling": "weak",
        "vs_baseline": (variants[hk]["value"] / paper["value"]) if paper else None,
        "dtype": "f64" if head[1] == "fp64" else "f32x2+f64",
        "data": "synthetic",
        "config": {"workload": w.name, "N": w.N, "p": w.p, "T": w.T, "n0": w.n0, "n": w.n,
                   "ncand": w.ncand, "d": w.d, "g": w.g, "method": head[0], "precision": head[1],
                   "l2": "flushed between timed steps (256 MB write)",
                   "parallelism": "replicas only: each GPU runs the whole workload"},
        "clocks": m["clocks"],
        "e2e": {"value": variants[hk]["e2e"]["value"], "unit": UNIT,
                "ms_per_step": H["e2e_ms"], "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                "api": "lagp_predict (host buffers, pinned)"},
        "gpu_launches": H["launches"],
        "kernels_ms": variants[hk]["kernels_ms"],
        "roofline": variants[hk]["roofline"],
        "accuracy_vs_oracle": variants[hk].get("accuracy_vs_oracle"),
        "variants": variants,
        "paper_form_effective_tflops": {
            k: paper_form_flops_per_location(w.n0, w.n, w.ncand) * T / (res[k]["sel_ms"] / 1e3) / 1e12
            for k in res if not k.startswith("nn")},
        "cpu_baseline": {"value": m["cpu"]["value"], "unit": UNIT, "cores": m["cpu"]["cores"],
                         "kind": "oracle",
                         "sample": "%d seeded locations of the %d, %s (%.1f s wall)" %
                                   (m["cpu"]["n"], w.T, head[0], m["cpu"]["seconds"])},
    }
    if paper:
        line["paper_context"] = {"value": paper["value"], "unit": UNIT, "what": paper["what"]}
    # The other workloads, each timed under its own clock record: only on the default
    # invocation at one GPU (they are measurements of their own, not part of the step).
    if world == 1 and args.extras and args.workload == "paper-2d" and not args.locations:
        xs, xw = min(args.steps, 5), 3
        for name in [x for x in args.extras.split(",") if x]:
            t0 = time.perf_counter()
            if name == "smooth-8d":
                line["smooth_8d"] = extra_single(args, "smooth-8d", xs, xw)
            elif name == "batched":
                line["batched"] = {prec: measure_batched(args, prec, xs, xw, args.batch_T)
                                   for prec in ("mixed", "fp64")}
            elif name == "dense":
                line["dense_ab"] = dense_ab_pair(10000, 1000, 3, 3)
            elif name == "serving":
                line["serving"] = measure_serving([float(r) for r in args.extra_serve_rates.split(",")],
                                                  args.extra_serve_seconds, ["mixed", "fp64"])
            line.setdefault("extras_wall_s", {})[name] = time.perf_counter() - t0
    print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


def measure_dense_ab(wname, T_sub, steps, warmup):
    """The A/B of the two forms of ALC on one workload's first T_sub locations, candidate
    lists computed once: kernels (b)+(c) of the paper's explicit-inverse form
    (lagp_select_dense_dev, O(j^2) per candidate) against the Cholesky-row kernels
    (lagp_select_dev, O(j)), FP64 and mixed, each timed with CUDA events over `steps`
    launches after `warmup` (L2 flushed between launches).  Agreement of the paper form's
    designs with the exact greedy designs (the Cholesky-row FP64 kernel's, which the parity
    tests pin to the oracle), and the paper form's roofline against the FP64 pipe."""
    import torch
    from paper_1303_0383_gb300 import lagp
    w = _workloads()[wname]["make"]()
    w.XX = np.ascontiguousarray(w.XX[:T_sub])
    T, M, dev = w.T, w.ncand, torch.device("cuda", torch.cuda.current_device())
    stream = torch.cuda.current_stream()
    X, Z, XX = (torch.as_tensor(a).to(dev) for a in (w.X, w.Z, w.XX))
    cand = torch.empty((T, M), dtype=torch.int32, device=dev)
    lagp.lagp_knn_dev(X, XX, M, cand, lagp.workspace(lagp.lagp_knn_workspace_bytes(w.N, T, M), dev),
                      stream)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    vis = os.environ.get("CUDA_VISIBLE_DEVICES", "")
    sampler = ClockSampler(int(vis) if vis.isdigit() else torch.cuda.current_device())
    sampler.start()
    res = {}
    for key in ("dense", "fp64", "mixed"):
        mean = torch.empty(T, dtype=torch.float64, device=dev)
        s2, var = torch.empty_like(mean), torch.empty_like(mean)
        idx = torch.empty((T, w.n), dtype=torch.int32, device=dev)
        status = torch.empty(T, dtype=torch.int8, device=dev)
        if key == "dense":
            ws = lagp.workspace(lagp.lagp_select_dense_workspace_bytes(T, w.p, w.n, M), dev)
            run = lambda: lagp.lagp_select_dense_dev(X, Z, XX, cand, w.n0, w.n, w.d, w.g, mean, s2,
                                                     var, idx, status, ws, stream)
        else:
            ws = lagp.workspace(lagp.lagp_select_workspace_bytes(T, w.p, w.n, M, "alc", key), dev)
            run = (lambda k=key: lagp.lagp_select_dev(X, Z, XX, cand, w.n0, w.n, w.d, w.g, "alc", k,
                                                      mean, s2, var, idx, status, ws, stream))
        for _ in range(warmup):
            run()
        torch.cuda.synchronize()
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
               for _ in range(steps)]
        for a, b in evs:
            flush.add_(1.0)
            a.record(stream)
            run()
            b.record(stream)
        torch.cuda.synchronize()
        res[key] = dict(ms=sum(a.elapsed_time(b) for a, b in evs) / steps,
                        idx=idx.cpu().numpy(), s2=s2.cpu().numpy(),
                        failed=int((status != 0).sum()))
    clocks = sampler.stop()
    d, f = res["dense"], res["fp64"]
    same = (d["idx"] == f["idx"]).all(axis=1)
    overlap = np.array([len(np.intersect1d(a, b)) / w.n for a, b in zip(d["idx"], f["idx"])])
    first = np.array([int(np.argmax(a != b)) if (a != b).any() else w.n
                      for a, b in zip(d["idx"], f["idx"])])
    ratio = d["s2"] / f["s2"]
    alg = dense_flops_per_location(w.n0, w.n, M, w.p)
    achieved = alg * T / (d["ms"] / 1e3) / 1e12
    return {
        "workload": w.name, "T": T, "n0": w.n0, "n": w.n, "ncand": M, "g": w.g,
        "steps": steps, "warmup": warmup, "l2": "flushed between timed launches (256 MB write)",
        "ms": {"dense_fp64": d["ms"], "cholesky_row_fp64": f["ms"], "cholesky_row_mixed": res["mixed"]["ms"]},
        "dense_over_cholesky_row_fp64": d["ms"] / f["ms"],
        "dense_over_cholesky_row_mixed": d["ms"] / res["mixed"]["ms"],
        "failed_locations": {k: r["failed"] for k, r in res.items()},
        "dense_designs": {
            "equal_to_exact_greedy": float(same.mean()),
            "mean_overlap_with_exact_greedy": float(overlap.mean()),
            "median_first_differing_step": float(np.median(first[~same])) if (~same).any() else None,
            "s2_ratio_to_exact_greedy": {"median": float(np.median(ratio)),
                                         "p99": float(np.quantile(ratio, 0.99)),
                                         "max": float(ratio.max()), "min": float(ratio.min())}},
        "roofline": {"kernel": "select_dense_kernel (kernels b+c)", "bound": "alu",
                     "achieved": achieved, "unit": "TFLOP/s", "peak": FP64_PEAK_TFLOPS_DERIVED,
                     "frac": achieved / FP64_PEAK_TFLOPS_DERIVED, "work_per_location": alg,
                     "work_unit": "FP64 flops of the paper's explicit-inverse form (FMA = 2, exp = 20)",
                     "peak_source": "derived FP64: 152 SMs x 2 DFMA/clk x 2 flop x 2.07 GHz"},
        "clocks": clocks,
    }


def dense_ab_pair(T2, T8, steps, warmup):
    """The A/B of the two forms on paper-2d (first T2 locations) and smooth-8d (first T8)."""
    return {"paper-2d": measure_dense_ab("paper-2d", T2, steps, warmup),
            "smooth-8d": measure_dense_ab("smooth-8d", T8, steps, warmup)}


def run_dense_ab(args):
    """--workload dense-ab: the A/B of the paper's explicit-inverse form against the
    Cholesky-row kernels alone, one JSON line (rank 0 of one GPU; --locations caps both
    workloads' location counts)."""
    from paper_1303_0383_gb300 import lagp
    lagp.load()
    T2 = args.locations or 10000
    T8 = min(args.locations or 1000, 1000)
    ab = dense_ab_pair(T2, T8, args.steps, args.warmup)
    print(json.dumps({"metric": "ALC kernels (b)+(c) ms: the paper's explicit-inverse form vs the "
                                "Cholesky-row form", "unit": "ms", "higher_is_better": False,
                      "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
                      "dtype": "f64 (paper form) / f64 and f32x2+f64 (Cholesky-row)",
                      "data": "synthetic", "dense_ab": ab}), flush=True)
    return 0


def extra_single(args, wname, steps, warmup):
    """A single-design workload as an extra key of the default line: every variant's rate,
    its roofline, its error against the oracle, its clocks (no end-to-end timing)."""
    spec = _workloads()[wname]
    m = measure_single(_with(args, precision="both"), wname, steps, warmup, False, spec["cpu"],
                       spec.get("acc_other", 64))
    w = m["w"]
    return {"workload": w.name, "N": w.N, "p": w.p, "T": w.T, "n0": w.n0, "n": w.n, "ncand": w.ncand,
            "d": w.d, "g": w.g, "steps": steps, "warmup": warmup, "unit": UNIT,
            "l2": "flushed between timed steps (256 MB write)", "clocks": m["clocks"],
            "variants": m["variants"],
            "cpu_baseline": {"value": m["cpu"]["value"], "unit": UNIT, "cores": m["cpu"]["cores"],
                             "kind": "oracle", "sample": "%d seeded locations, alc (%.1f s wall)"
                             % (m["cpu"]["n"], m["cpu"]["seconds"])}}


def run_stagewise(args, world, rank):
    import torch
    from paper_1303_0383_gb300 import lagp
    spec = _workloads()[args.workload]
    w = spec["make"]()
    if args.locations:
        w.XX = np.ascontiguousarray(w.XX[: args.locations])
        if w.ZZ is not None:
            w.ZZ = w.ZZ[: args.locations]
        w.name += " (first %d locations)" % args.locations
    variants_run = [v for v in spec["variants"] if args.precision == "both" or v[1] == args.precision]
    dev = torch.device("cuda", torch.cuda.current_device())
    stream = torch.cuda.current_stream()
    X, Z, XX = (torch.as_tensor(a).to(dev) for a in (w.X, w.Z, w.XX))
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    sampler = ClockSampler(torch.cuda.current_device())
    sampler.start()
    res = {}
    for method, prec in variants_run:
        # the stagewise scheme with local MLE: the paper's alc/mspe (1 stage) and alc2/mspe2
        # (2 stages) rows; device buffers only (no host API for it)
        k = vkey(method + (str(args.stages) if args.stages > 1 else "") + "_mle", prec)
        res[k] = time_stagewise(args, w, method, prec, args.stages, X, Z, XX, flush, stream, lagp, torch)
    clocks = sampler.stop()
    for r in res.values():
        if world > 1:
            r["ms"] = max_over_ranks([r["ms"]], dev)[0]
    if rank != 0:
        return 0
    variants = {k: {"value": world * w.T / (r["ms"] / 1e3), "ms_per_step": r["ms"],
                    "kernels_ms": r["kernels_ms"], "gpu_launches": r["launches"],
                    "newton_iters_mean": r["newton_iters"], "accuracy": accuracy(w, r["mean"], r["s2"])}
                for k, r in res.items()}
    return print_stagewise(args, w, spec, variants, clocks, world)


_BATCH_ORACLE: dict = {}


def batched_accuracy(B, idx, mean, s2, var, n_sample=48):
    """The parity protocol (oracle/parity.py) on a seeded sample of a batch's locations: each
    against the oracle on its own design, n and candidate count.  The sample is drawn from
    the locations with n <= 80 and at most 1500 candidates (the oracle's cost grows as
    n^2 M: seconds per location at n = 200, M = 4000); the oracle's designs are computed once
    per batch and shared by both precisions, on the host cores (ctypes calls release the
    interpreter lock)."""
    from concurrent.futures import ThreadPoolExecutor

    import oracle
    from oracle.parity import check_location
    from paper_1303_0383_gb300.inputs import Workload
    rng = np.random.default_rng(4)
    elig = np.nonzero((B.n <= 80) & (B.ncand <= 1500))[0]
    locs = np.sort(rng.choice(elig, size=min(n_sample, len(elig)), replace=False))
    off = np.concatenate([[0], np.cumsum(B.n)]).astype(np.int64)

    def one_workload(t):
        W = B.designs[int(B.design_of[t])]
        x = np.ascontiguousarray(B.XX[t, : W.p][None, :])
        return Workload("batched location %d" % t, W.X, W.Z, x, n0=W.n0, n=int(B.n[t]),
                        ncand=int(B.ncand[t]), d=W.d, g=W.g)

    key = (B.name, B.T, tuple(locs))
    if key not in _BATCH_ORACLE:
        def solve(t):
            w1 = one_workload(t)
            cand = oracle.knn(w1.X, w1.XX, w1.ncand)[0]
            return cand, oracle.local_design(w1.X, w1.Z, w1.XX[0], cand, w1.n0, w1.n, w1.d, w1.g, "alc")
        with ThreadPoolExecutor(max_workers=os.cpu_count() or 4) as ex:
            _BATCH_ORACLE[key] = list(ex.map(solve, locs))
    from oracle.parity import CLAUSES
    same = failed = forced = near = 0
    errs = {"mean": [], "s2": [], "var": []}
    by_clause: dict = {}
    first = None
    for t, (cand, ora) in zip(locs, _BATCH_ORACLE[key]):
        try:
            info = check_location(one_workload(t), 0, cand, idx[off[t]:off[t + 1]], mean[t], s2[t],
                                  "alc", gpu_var=var[t], ora=ora)
        except AssertionError as e:
            failed += 1
            first = first or str(e)[:300]
            continue
        same += not info["forced"]
        forced += info["forced"]
        near += info["near_ties"]
        failed += not info["ok_vals"]
        for k in errs:
            errs[k].append(info["err_" + k])
        for k2, c in enumerate(info["clauses"]):
            if c:
                e = info["adj_%d" % k2][0]
                nv, mv = by_clause.get(c, (0, 0.0))
                by_clause[c] = (nv + 1, max(mv, e))
    out = {"locations": int(len(locs)), "selection_match_rate": same / max(len(locs), 1),
           "forced_path_locations": forced, "near_tie_steps": near, "failed": failed,
           "sample": "%d seeded locations with n <= 80 and at most 1500 candidates" % len(locs)}
    for k, v in errs.items():
        v = np.asarray(v) if v else np.zeros(1)
        out["max_rel_err_" + k] = float(v.max())
        out["median_rel_err_" + k] = float(np.median(v))
    out["adjudicated"] = {CLAUSES[c]: {"values": nv, "max_rel_err": mv}
                          for c, (nv, mv) in sorted(by_clause.items())}
    if first:
        out["first_failure"] = first
    return out


def measure_batched(args, prec, steps, warmup, batch_T):
    """Workload 4: uneven local problems over three resident designs in one persistent
    launch, CUDA-graph replay, launch shape tuned on the first batch."""
    import torch
    from paper_1303_0383_gb300 import inputs, lagp
    lagp.load()
    B = inputs.batched_uneven(batch_T)
    dev = torch.device("cuda", torch.cuda.current_device())
    designs = [dict(X=torch.as_tensor(w.X, device=dev), Z=torch.as_tensor(w.Z, device=dev),
                    n0=w.n0, theta=w.d, g=w.g) for w in B.designs]
    T = B.T
    XX = torch.as_tensor(B.XX, device=dev)
    mean = torch.empty(T, dtype=torch.float64, device=dev)
    s2, var = torch.empty_like(mean), torch.empty_like(mean)
    idx = torch.empty(int(B.n.sum()), dtype=torch.int32, device=dev)
    status = torch.empty(T, dtype=torch.int8, device=dev)
    ws = lagp.workspace(lagp.lagp_predict_batch_workspace_bytes(designs, B.design_of, B.n,
                                                                B.ncand, "alc", prec), dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream()
    flags = lagp.LAGP_BATCH_TUNE | lagp.LAGP_BATCH_GRAPH

    def step():
        lagp.lagp_predict_batch_dev(designs, XX, B.design_of, B.n, B.ncand, "alc", prec, mean, s2,
                                    var, idx, status, flags, ws, stream)

    t0 = time.perf_counter()
    step()                       # tunes the launch shape for this signature
    torch.cuda.synchronize()
    tune_s = time.perf_counter() - t0
    for _ in range(warmup):
        step()                   # captures the graph, then replays
    torch.cuda.synchronize()
    assert int((status != 0).sum()) == 0
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(steps)]
    sampler = ClockSampler(torch.cuda.current_device())
    sampler.start()
    launches0 = lagp.lagp_launch_count()
    torch.cuda.synchronize()
    for k in range(steps):
        flush.add_(1.0)
        evs[k][0].record(stream)
        step()
        evs[k][1].record(stream)
    torch.cuda.synchronize()
    clocks = sampler.stop()
    ms = sum(a.elapsed_time(b) for a, b in evs) / steps
    acc = batched_accuracy(B, idx.cpu().numpy(), mean.cpu().numpy(), s2.cpu().numpy(),
                           var.cpu().numpy())
    return {"metric": "local-GP predictions/sec, batched uneven problems", "value": T / (ms / 1e3),
            "unit": UNIT, "steps": steps, "warmup": warmup, "ms_per_step": ms,
            "dtype": "f32x2+f64" if prec == "mixed" else "f64",
            "config": {"workload": B.name, "precision": prec, "method": "alc",
                       "flags": "tune+graph", "first_call_s": tune_s,
                       "l2": "flushed between timed steps (256 MB write)"},
            "clocks": clocks,
            # the library's kernels per step (graph replays count the kernels they hold)
            "gpu_launches": (lagp.lagp_launch_count() - launches0) / steps,
            "accuracy_vs_oracle": acc}


def run_batched(args):
    precs = ["mixed", "fp64"] if args.precision == "both" else [args.precision]
    out = {p: measure_batched(args, p, args.steps, args.warmup, args.batch_T) for p in precs}
    line = dict(out[precs[0]])
    line.update(n_gpus=1, higher_is_better=True, data="synthetic", variants=out)
    print(json.dumps(line), flush=True)
    return 0


_SERVE_ORACLE: dict = {}


def served_accuracy(designs, ncand, picked):
    """The parity protocol on served locations (the first location of every 23rd request at
    the headline rate, at most 48): each against the oracle on its design, n and candidate
    count.  picked: (design, x, n, result row) tuples.  The oracle's designs are cached by
    request, so both precisions (which serve the same seeded requests) share them."""
    from concurrent.futures import ThreadPoolExecutor

    import oracle
    from oracle.parity import check_location
    from paper_1303_0383_gb300.inputs import Workload

    def workload(d, x, n):
        W = designs[d]
        return Workload("served location", W.X, W.Z, np.ascontiguousarray(x[None, :]), n0=W.n0,
                        n=n, ncand=ncand[d], d=W.d, g=W.g)

    keys = [(d, x.tobytes(), n) for d, x, n, _ in picked]
    todo = [(k, d, x, n) for k, (d, x, n, _) in zip(keys, picked) if k not in _SERVE_ORACLE]

    def solve(item):
        _, d, x, n = item
        w1 = workload(d, x, n)
        cand = oracle.knn(w1.X, w1.XX, w1.ncand)[0]
        return cand, oracle.local_design(w1.X, w1.Z, w1.XX[0], cand, w1.n0, w1.n, w1.d, w1.g, "alc")
    with ThreadPoolExecutor(max_workers=os.cpu_count() or 4) as ex:
        for item, res in zip(todo, ex.map(solve, todo)):
            _SERVE_ORACLE[item[0]] = res
    same = failed = 0
    worst = {"mean": 0.0, "s2": 0.0, "var": 0.0}
    for k, (d, x, n, r) in zip(keys, picked):
        cand, ora = _SERVE_ORACLE[k]
        try:
            info = check_location(workload(d, x, n), 0, cand, r["idx"], r["mean"], r["s2"], "alc",
                                  gpu_var=r["var"], ora=ora)
        except AssertionError:
            failed += 1
            continue
        same += not info["forced"]
        failed += not info["ok_vals"]
        for q in worst:
            worst[q] = max(worst[q], info["err_" + q])
    return {"locations": len(picked), "selection_match_rate": same / max(len(picked), 1),
            "failed": failed, "max_rel_err_mean": worst["mean"], "max_rel_err_s2": worst["s2"],
            "max_rel_err_var": worst["var"],
            "sample": "the first location of every 23rd request at the headline rate"}


def measure_serving(rates, seconds, precs):
    """Workload 5: Poisson arrivals of requests (1..4096 locations, log-uniform) against
    the three resident designs with n in {50, 100}; p50/p99 latency and throughput per
    arrival rate, for the server in each precision, with the clocks of each precision's
    run."""
    import torch
    from paper_1303_0383_gb300 import inputs, lagp
    lagp.load()
    B = inputs.batched_uneven(1)
    dev = torch.device("cuda", torch.cuda.current_device())
    descs = [dict(X=torch.as_tensor(w.X, device=dev), Z=torch.as_tensor(w.Z, device=dev),
                  n0=w.n0, theta=w.d, g=w.g) for w in B.designs]
    ncand = [1000, 2000, 2000]
    lo, hi = [-2.0, 0.0, 0.0], [2.0, 1.0, 1.0]
    results = {}
    for prec in precs:
        srv = lagp.Server(descs, "alc", prec, nmax=100, ncand_max=2000, max_batch=16384,
                          memory_budget=24 << 30, max_slots=3)
        # warm-up: one request per design and n
        for d in range(3):
            for n in (50, 100):
                rid = srv.submit(d, np.random.default_rng(d).uniform(lo[d], hi[d], (64, B.designs[d].p)),
                                 n, ncand[d])
                srv.wait(rid, -1)
                srv.results(rid)
        sampler = ClockSampler(torch.cuda.current_device())
        sampler.start()
        per_rate = {}
        picked = []
        for lam in rates:
            rng = np.random.default_rng(int(lam))
            sent, reqs = [], []
            start = time.perf_counter()
            t_next = 0.0
            while t_next < seconds:
                L = int(np.floor(np.exp(rng.uniform(0.0, np.log(4097.0)))))
                d = int(rng.integers(0, 3))
                n = int(rng.choice([50, 100]))
                x = rng.uniform(lo[d], hi[d], size=(L, B.designs[d].p))
                now = time.perf_counter() - start
                if t_next > now:
                    time.sleep(t_next - now)
                sent.append((srv.submit(d, x, n, ncand[d]), L))
                reqs.append((d, x, n))
                t_next += rng.exponential(L / lam)   # arrivals carry L locations at rate lam
            lat, locs = [], 0
            for k, (rid, L) in enumerate(sent):
                srv.wait(rid, -1)
                r = srv.results(rid)
                assert (r["status"] == 0).all()
                lat.append(r["latency_ms"])
                locs += L
                if lam == max(rates) and k % 23 == 0 and len(picked) < 48:
                    d, x, n = reqs[k]
                    picked.append((d, x[0].copy(), n, {q: r[q][0] for q in ("idx", "mean", "s2", "var")}))
            wall = time.perf_counter() - start
            lat = np.array(lat)
            per_rate[str(int(lam))] = {
                "requests": len(sent), "locations": locs,
                "throughput_locations_per_s": locs / wall,
                "p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
                "mean_ms": float(lat.mean())}
        clocks = sampler.stop()
        st = srv.stats()
        srv.close()
        results[prec] = {"rates": per_rate, "slots": st["slots"], "max_inflight": st["max_inflight"],
                         "batches": st["batches"], "clocks": clocks,
                         "accuracy_vs_oracle": served_accuracy(B.designs, ncand, picked)}
    top = str(int(max(rates)))
    head = "mixed" if "mixed" in results else precs[0]
    return {"metric": "serving p99 ms (Poisson arrivals, 1..4096 locations per request)",
            "value": results[head]["rates"][top]["p99_ms"], "unit": "ms", "higher_is_better": False,
            "config": {"workload": "serving over the 2-d/4-d/8-d designs, n in {50,100}, candidates "
                                   "1000/2000/2000, %g s of arrivals per rate" % seconds,
                       "rates_locations_per_s": rates, "headline_rate": top, "precision": head},
            "results": results}


def run_serving(args):
    precs = ["fp64", "mixed"] if args.precision == "both" else [args.precision]
    line = measure_serving([float(r) for r in args.serve_rates.split(",")], args.serve_seconds, precs)
    line.update(n_gpus=1, data="synthetic")
    print(json.dumps(line), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--precision", default="both", choices=["fp64", "mixed", "both"])
    ap.add_argument("--cpu-sample", type=int, default=0,
                    help="oracle sample size (0: the workload's default, about 10-30 s on 16 cores)")
    ap.add_argument("--ref-sample", type=int, default=160)
    ap.add_argument("--locations", type=int, default=0,
                    help="use only the first K locations (small case for profiling)")
    ap.add_argument("--no-e2e", action="store_true", help="skip the host-API timing")
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU oracle sample")
    ap.add_argument("--workload", default="paper-2d",
                    choices=["paper-2d", "smooth-8d", "grid-2d", "borehole", "borehole-8000", "batched",
                             "serving", "dense-ab"])
    ap.add_argument("--extras", default="smooth-8d,batched,dense,serving",
                    help="other workloads measured after the default paper-2d line and added to it "
                         "as keys (comma list; empty: none)")
    ap.add_argument("--no-extras", dest="extras", action="store_const", const="")
    ap.add_argument("--extra-serve-rates", default="1000,20000,50000")
    ap.add_argument("--extra-serve-seconds", type=float, default=10.0)
    ap.add_argument("--serve-rates", default="1000,5000,10000,20000,50000")
    ap.add_argument("--serve-seconds", type=float, default=30.0)
    ap.add_argument("--batch-T", type=int, default=20000)
    ap.add_argument("--stages", type=int, default=0,
                    help="time the stagewise scheme with local MLE (Sec. 4.2): 1 or 2 stages")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "batched":
        return run_batched(args)
    if args.workload == "serving":
        return run_serving(args)
    if args.workload == "dense-ab":
        return run_dense_ab(args)
    return run_gpu(args)


if __name__ == "__main__":
    sys.exit(main())

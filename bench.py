"""Benchmark of the temporally parallel LQT solver on one GB300 (or N replicas).

Workload: the 2-D point-mass tracking problem (n=4 states, m=2 inputs, the
paper's F and L of Sec. VI-A), t in [0, 100], T = 2^20 sub-intervals with
K = 4 RK4 steps each, X(t) and r(t) sampled on the half-step grid (1.35 GB of
inputs, larger than L2).  One step = one lqt_solve: element build + value scan
+ trajectory scan + controls + optimal cost.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Prints one JSON line.  `value` is sub-intervals per second over all ranks with
inputs resident on the device; `e2e` is the same metric through the host-buffer
entry point lqt_solve_host with the host<->device copies inside the timed
region.  Under torchrun every rank solves its own copy of the workload
(replicas: the method has no cross-GPU exchange at this size).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "LQT sub-intervals/s (build+scan+trajectory) vs sequential GPU sweep, same tol"
UNIT = "sub-intervals/s"
T_DEFAULT = 1 << 20
K_STEPS = 4
FP64_PEAK_TFLOPS = 152 * 4 * 0.5 * 2 * 2.07e9 / 1e12  # SMs x sub-partitions x DFMA/clk x flop x max clock
PROFILE_TRAFFIC = os.path.join(ROOT, "profiles", "build_kernel_point_mass_n4.md")


def algorithmic_build_flops_per_block(n: int, K: int) -> float:
    """The algorithmic FP64 work of one element build: K RK4 steps of the dense
    element right-hand side, K (40 n^3 + 60 n^2) flop (FMA = 2; no symmetric
    savings, no factor form): the per-unit figure the roofline uses."""
    return float(K * (40 * n ** 3 + 60 * n ** 2))


def build_flops_per_block(n: int, m_pad: int, K: int, has_c: bool) -> float:
    """FP64 operations of one element build (FMA = 2), as the kernel is written:
    per right-hand side A Lt and J Lt (2 n^2 M), Lt^T eta (n M), dA (n^2 (M+n)),
    db (n (M + n[c])), dC (n(n+1)/2 M), deta (n (n + M + n[c])), J F (n^3), dJ
    (n(n+1)/2 (M + 2 adds)), dzeta (M + n[c]); 4 right-hand sides and 7 axpys of
    the 3n^2/... state (n^2 + n + 2 n(n+1)/2 + n + 1 entries) per RK4 step."""
    ns = n * (n + 1) // 2
    c = n if has_c else 0
    fma = 2 * n * n * m_pad + n * m_pad + n * n * (m_pad + n) + n * (m_pad + c) + ns * m_pad + \
        n * (n + m_pad + c) + n ** 3 + ns * m_pad + m_pad + c
    adds = 2 * ns + 2
    rhs = 2 * fma + adds
    state = n * n + n + 2 * ns + n + 1
    step = 4 * rhs + 7 * 2 * state
    return float(K * step)


def alg_scan(n: int) -> float:
    """Algorithmic FP64 work of the value scan per sub-interval: about 22 n^3
    flop (a full combination in the reduce and a value-form combination in the
    down-sweep, dense products and LU)."""
    return 22.0 * n ** 3


def alg_traj(n: int) -> float:
    """Algorithmic FP64 work of the state scan per sub-interval: about 9 n^3
    flop (the one-sub-interval map and its composition)."""
    return 9.0 * n ** 3


def alg_solve(n: int, m: int, K: int) -> float:
    """Algorithmic FP64 work of one lqt_solve per sub-interval: element build,
    value scan, state scan and the control 2 m n."""
    return algorithmic_build_flops_per_block(n, K) + alg_scan(n) + alg_traj(n) + 2.0 * m * n


def alg_backward(n: int, m: int, K: int) -> float:
    """Algorithmic work of one lqt_backward per sub-interval: the elements
    recomputed once (one build) plus a vector-Jacobian product of every
    forward stage, each costing twice its stage (one product per operand):
    3 build + 2 (value scan + state scan)."""
    return 3.0 * algorithmic_build_flops_per_block(n, K) + 2.0 * (alg_scan(n) + alg_traj(n))


def alg_densify(n: int, m: int, K: int) -> float:
    """Algorithmic work of lqt_densify per sub-interval: K RK4 steps (4 stages)
    of the Riccati right-hand side (S F: 2n^3, (S Lt)(S Lt)^T: 4 n^2 m, the v
    equation 2 n^2 + 4 n m) and of the closed loop (2 n^2 + 4 n m)."""
    return float(K * (4 * (2 * n ** 3 + 4 * n * n * m + 2 * n * n + 4 * n * m) + 4 * (2 * n * n + 4 * n * m)))


def alg_method2(n: int, m: int, K: int) -> float:
    """lqt_solve_method2 per sub-interval: the backward and the forward element
    builds, the value scan and the prefix scan (22 n^3 each), the states from
    the prefixes (one LU with n + 1 right-hand sides, about 3 n^3)."""
    return 2.0 * algorithmic_build_flops_per_block(n, K) + 2.0 * alg_scan(n) + 3.0 * n ** 3 + 2.0 * m * n


def alg_invariant_solve(n: int, m: int, K: int) -> float:
    """lqt_solve_invariant per sub-interval: the per-sub-interval part of the
    time-invariant build (b, eta, zeta by K RK4 steps of matrix-vector
    products, about 24 K (n m + n^2) flop) plus the value and state scans."""
    return 24.0 * K * (n * m + n * n) + alg_scan(n) + alg_traj(n) + 2.0 * m * n


def scan_flops_per_block(n: int) -> float:
    """Approximate FP64 work of stages (b)+(c) per sub-interval: one full
    combination (reduce), one value-form combination with the map, the chunk
    composition and the state/control update."""
    full = 2 * (n ** 3 * (1 + 2 + 1 + 1.5 + 1 + 1.5) + 2 * n ** 3 / 3)
    value = 2 * (n ** 3 * (1 + 1 + 1 + 0.5) + n ** 3 / 3)
    comp = 2 * n ** 3
    return float(full + value + comp + 2 * 2 * n * n)


# ---------------------------------------------------------------------------
# clocks
# ---------------------------------------------------------------------------

class ClockSampler:
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.path = None

    def __enter__(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        if self.proc is None or not self.path:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        rows = []
        for ln in open(self.path):
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                rows.append((float(parts[0]), float(parts[1]), parts[4:8]))
            except ValueError:
                continue
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for _, _, flags in rows for i, f in enumerate(flags) if f.lower() == "active"})
        return {"sm_mhz": statistics.median(r[0] for r in rows), "sm_max_mhz": max(r[1] for r in rows),
                "reasons": reasons, "samples": len(rows)}


# ---------------------------------------------------------------------------
# helpers
# ---------------------------------------------------------------------------

def source_hash() -> str:
    """sha256 (first 16 hex digits) of the element-build kernel's own source:
    the right-hand side, RK4 driver and kernel in lqt_build.cu and the element
    types and stores of lqt_device.cuh that it uses."""
    csrc = os.path.join(ROOT, "paper_2212_11744_gb300", "csrc")
    build = open(os.path.join(csrc, "lqt_build.cu")).read()
    dev = open(os.path.join(csrc, "lqt_device.cuh")).read()
    parts = [
        build[build.index("// Right-hand side of the backward conditional HJB ODEs in s:"):
              build.index("// Terminal element a_T")],
        dev[:dev.index("// Packed element size")],
    ]
    i0 = dev.index("template <int N>\n__device__ __forceinline__ void store_public")
    parts.append(dev[i0:dev.index("template <int N>", i0 + 10)])
    h = hashlib.sha256()
    for part in parts:
        h.update(part.encode())
    return h.hexdigest()[:16]


def profiled_traffic():
    """DRAM bytes per build-kernel launch from the committed ncu summary, if it
    was taken on the current kernel source."""
    if not os.path.exists(PROFILE_TRAFFIC):
        return None
    txt = open(PROFILE_TRAFFIC).read()
    mh = re.search(r"source_hash:\s*([0-9a-f]+)", txt)
    mt = re.search(r"traffic_bytes_per_full_launch:\s*([0-9.eE+]+)", txt)
    if not mh or not mt or mh.group(1) != source_hash():
        return None
    return float(mt.group(1))


def dist_setup():
    """torchrun environment -> (world size, rank, local rank).  NCCL when CUDA is
    present, gloo otherwise (the CPU tests of the multi-rank logic)."""
    import torch
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if ws > 1:
        import torch.distributed as dist
        if torch.cuda.is_available():
            torch.cuda.set_device(local)
            dist.init_process_group("nccl", device_id=torch.device("cuda", local))
        else:
            dist.init_process_group("gloo")
    elif torch.cuda.is_available():
        torch.cuda.set_device(local)
    return ws, rank, local


def _dist_device():
    import torch
    import torch.distributed as dist
    return torch.device("cuda") if dist.get_backend() == "nccl" else torch.device("cpu")


def barrier(ws):
    """All ranks meet here (an all-reduce on the backend's device), then the
    local GPU, if any, is drained."""
    import torch
    if ws > 1:
        import torch.distributed as dist
        t = torch.zeros(1, device=_dist_device())
        dist.all_reduce(t)
    if torch.cuda.is_available():
        torch.cuda.synchronize()


def max_over_ranks(x: float, ws: int) -> float:
    import torch
    if ws == 1:
        return x
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=_dist_device())
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def probe_pipes() -> dict:
    """FP64 and FP32 FMA throughput on this device, measured with the
    library's probe kernel (lqt_probe_fma_rate: 8 independent FMA chains per
    thread, 256 threads per SM, one CTA per SM), best of three CUDA-event
    timings each; and the time of one warp-wide FP64 FMA instruction on one
    sub-partition with 1 and with 32 active lanes."""
    import torch

    import paper_2212_11744_gb300 as lqt
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    out = lqt.lqt_probe_fma_rate(0, sms, 256, 10, 32)

    def rate(prec, iters, threads):
        best = None
        for _ in range(3):
            ms = _events_ms(lambda: lqt.lqt_probe_fma_rate(prec, sms, threads, iters, 32, out=out), 1)
            best = ms if best is None else min(best, ms)
        return 2.0 * 8 * iters * sms * threads / (best * 1e-3) / 1e12

    res = {"sms": sms, "fp64_tflops": rate(0, 20000, 256), "fp32_tflops": rate(1, 100000, 256)}
    for lanes in (1, 32):
        ms = min(_events_ms(lambda: lqt.lqt_probe_fma_rate(0, 1, 32, 5000, lanes, out=out), 1) for _ in range(3))
        res[f"fp64_ns_per_warp_instruction_{lanes}_lanes"] = ms * 1e6 / (8 * 5000)
    res["how"] = "lqt_probe_fma_rate: 8 independent chains x <- x a + b per thread, 256 threads per SM"
    return res


def roofline(kernel: str, flop_per_unit: float, formula: str, units: float, ms: float, peak_measured,
             traffic=None, peak: float = None, note: str = None) -> dict:
    """The roofline object of one row: algorithmic FP64 flop per unit x units
    / the CUDA-event time, against the FP64 pipe's peak (derived from unit
    counts and clock) and beside it the rate the probe measured in this run."""
    peak = FP64_PEAK_TFLOPS if peak is None else peak
    ach = flop_per_unit * units / (ms * 1e-3) / 1e12
    r = {"bound": "alu", "kernel": kernel, "achieved": ach, "peak": peak, "unit": "TFLOP/s", "frac": ach / peak,
         "peak_measured": peak_measured, "frac_of_measured": (ach / peak_measured) if peak_measured else None,
         "traffic": traffic, "stage_ms": ms, "flop_per_unit": formula, "flop_per_unit_value": flop_per_unit,
         "units": units}
    if note:
        r["note"] = note
    return r


def cpu_baseline_sample(p, seconds_hint=True):
    """Times the oracle (single thread, as it stands) on the first Ts
    sub-intervals of the workload."""
    import oracle
    import workloads as W
    Ts = min(1 << 19, p.T)
    sub = W.truncate(p, Ts)
    t0 = time.perf_counter()
    oracle.solve(sub)
    dt = time.perf_counter() - t0
    return {"value": Ts / dt, "unit": UNIT, "cores": 1, "kind": "oracle",
            "sample": f"first {Ts} of the {p.T} sub-intervals (same grid and samples), one solve, {dt:.1f} s"}


def cpu_baseline_grid(g):
    """Times the oracle's grid method (block function, then values in the
    doubling order), single thread, on the whole problem."""
    import oracle
    t0 = time.perf_counter()
    oracle.grid_values(g, oracle.grid_block(g))
    dt = time.perf_counter() - t0
    return {"value": g.T / dt, "unit": "blocks/s", "cores": 1, "kind": "oracle",
            "sample": f"the whole G = {g.G}, T = {g.T} problem, {dt:.2f} s"}


def _oracle_timed(fn, units: float, unit: str, sample: str) -> dict:
    t0 = time.perf_counter()
    fn()
    dt = time.perf_counter() - t0
    return {"value": units / dt, "unit": unit, "cores": 1, "kind": "oracle", "sample": f"{sample}, {dt:.2f} s"}


def cpu_baseline_batch(probs, seconds_per_n: float = 1.5) -> dict:
    """The oracle on a fixed sample of the 4096-problem batch: for each state
    dimension, the first problems of that dimension in batch order until about
    seconds_per_n (at least one), giving a rate per dimension; the batch's
    oracle time is then the sum over dimensions of its sub-intervals of that
    dimension divided by that dimension's rate."""
    import oracle
    byn = {}
    for p in probs:
        byn.setdefault(p.n, []).append(p)
    rates, counts, secs = {}, {}, 0.0
    for n, ps in sorted(byn.items()):
        t0 = time.perf_counter()
        done, subs = 0, 0
        while done < len(ps) and (done == 0 or time.perf_counter() - t0 < seconds_per_n):
            oracle.solve(ps[done])
            subs += ps[done].T
            done += 1
        dt = time.perf_counter() - t0
        rates[n], counts[n] = subs / dt, done
        secs += dt
    total = sum(p.T for p in probs)
    est = sum(sum(p.T for p in ps) / rates[n] for n, ps in byn.items())
    return {"value": total / est, "unit": UNIT, "cores": 1, "kind": "oracle",
            "per_n_rate": {str(n): r for n, r in rates.items()},
            "sample": "per n, the first problems of that n in batch order: " +
                      ", ".join(f"n={n}: {c}" for n, c in counts.items()) +
                      f" problems ({secs:.1f} s in all); batch time = sum over n of its sub-intervals / rate"}


def cpu_baseline_adjoint(Ts: int = 256) -> dict:
    """The oracle's reverse mode (torch CPU autograd through its restatement)
    on the first Ts sub-intervals of the differentiable n = 8 workload,
    forward + backward."""
    import torch

    from oracle import lqt_torch as LT
    import workloads as W
    p = W.truncate(W.differentiable_n8(), Ts)

    def run():
        t = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64).requires_grad_()
        F, L, X, U, r, Xf, x0 = (t(p.F.values), t(p.L.values), t(p.X.values), t(p.U.values), t(p.r.values),
                                 t(p.Xf), t(p.x0))
        rf = t(p.rf) if p.rf is not None else None
        o = LT.solve(p, F, L, X, U, r, Xf, rf, x0)
        loss = o["cost"] + ((o["x"][-1] - torch.tensor(p.extra["x_target"])) ** 2).sum()
        loss.backward()

    return _oracle_timed(run, Ts, UNIT + " (forward + backward)",
                         f"the first {Ts} of the {1 << 14} sub-intervals, reverse mode")


def cpu_baseline_densify(Ts: int = 1 << 14) -> dict:
    import oracle
    import workloads as W
    p = W.truncate(W.point_mass_2d(T=T_DEFAULT, K=K_STEPS), Ts)
    return _oracle_timed(lambda: oracle.densify(p, oracle.solve(p)), Ts * p.K, "sub-steps/s (solve + densify)",
                         f"the first {Ts} sub-intervals of the point mass")


def cpu_baseline_method2(Ts: int = 1 << 14) -> dict:
    import oracle
    import workloads as W
    p = W.truncate(W.point_mass_2d(T=T_DEFAULT, K=K_STEPS), Ts)

    def run():
        sol = oracle.solve(p)
        oracle.trajectory_method2(p, sol["S"], sol["v"])

    return _oracle_timed(run, Ts, UNIT, f"the first {Ts} sub-intervals of the point mass (values, then Method 2)")


# ---------------------------------------------------------------------------
# reference arm: the oracle as it stands, on the host cores
# ---------------------------------------------------------------------------

def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import oracle
    import workloads as W
    oracle.build()
    p = W.point_mass_2d(T=T_DEFAULT, K=K_STEPS)
    Ts = 1 << 16
    sub = W.truncate(p, Ts)
    for _ in range(args.warmup):
        oracle.solve(sub)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        oracle.solve(sub)
    dt = (time.perf_counter() - t0) / args.steps
    value = Ts / dt
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": workload_config(p),
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                         "sample": f"first {Ts} of the {p.T} sub-intervals per step"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))


def workload_config(p):
    return {"workload": f"point_mass_2d n={p.n} m={p.m} T={p.T} K={p.K} t=[0,100] X,r per RK4 half-step",
            "T": p.T, "n": p.n, "m": p.m, "K": p.K,
            "l2": f"inputs larger than L2 ({p.nbytes_inputs() / 1e9:.2f} GB of coefficient samples)"}


# ---------------------------------------------------------------------------
# the other rows of the hot path, measured beside the headline
# ---------------------------------------------------------------------------

def _events_ms(fn, reps, stream=None):
    import torch
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(reps):
        fn()
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / reps


def _relmax(a, b):
    return float((a - b).abs().max() / b.abs().max().clamp_min(1e-12))


def tune_candidates(n: int):
    """First-level chunk lengths the batch autotuner tries for state dimension
    n (0 = the library's own choice): all of them where a solve of the class
    takes well under a second, three where it takes seconds (n = 16)."""
    return (0, 2, 4, 8, 16, 32) if n <= 8 else (0, 8, 32)


def measure_rows(T_headline, pk=None):
    """Batched (4096 problems), mixed precision (point mass at T = 2^20 and the
    n = 64 workload), adjoint (n = 8, T = 2^14), the short double-integrator
    solve and the next rows.  Each entry is timed with CUDA events after a
    warm-up and carries a roofline object (algorithmic FP64 flop per unit x
    units / its time, against the FP64 pipe peak; pk = the probe's measured
    FP64 rate); failures are recorded, not raised."""
    import torch

    import paper_2212_11744_gb300 as lqt
    import workloads as W
    rows = {}

    def guard(name, fn):
        try:
            rows[name] = fn()
        except Exception as exc:  # keep the headline line even if a row fails
            rows[name] = {"error": repr(exc)[:300]}

    def batched():
        from paper_2212_11744_gb300.batch import BatchSet
        probs = [W.batched_member(b) for b in range(4096)]
        bset = BatchSet(probs)
        bts = bset.batches
        chunks = {n: bt.autotune(candidates=tune_candidates(n), reps=3 if n <= 8 else 2) for n, bt in bts.items()}
        outs = bset.new_outputs()
        s = torch.cuda.Stream()
        bset.solve(outs, stream=s)
        torch.cuda.synchronize()
        g = bset.capture(outs, stream=s)
        g.replay()
        torch.cuda.synchronize()
        ms = _events_ms(g.replay, 2)
        per = {str(n): _events_ms(lambda bt=bt, o=outs[n]: bt.solve(out=o), 1) for n, bt in bts.items()}
        total = int(sum(p.T for p in probs))
        subs_n = {n: int(bt.T.sum()) for n, bt in bts.items()}
        st = lqt.lqt_get_status()
        flop = sum(alg_solve(n, max(1, n // 2), 4) * subs_n[n] for n in bts)
        rl = roofline("the four batched solves (one CUDA graph, one stream per n)", flop / total,
                      "sum over n of K (40 n^3 + 60 n^2) + 22 n^3 + 9 n^3 + 2 m n per sub-interval, averaged",
                      total, ms, pk)
        rl["per_n"] = {str(n): roofline(f"lqt_solve_batched n={n}", alg_solve(n, max(1, n // 2), 4),
                                        "K (40 n^3 + 60 n^2) + 22 n^3 + 9 n^3 + 2 m n", subs_n[n], per[str(n)], pk)
                       for n in bts}
        return {"workload": "4096 LQT problems, n in {2,4,8,16} (m = n/2), T in [256, 8192], K = 4, one CUDA graph "
                            "of four batched solves (one per n, each on its own stream)",
                "value": total / (ms * 1e-3), "unit": UNIT, "ms": ms, "sub_intervals": total,
                "per_n_ms": per, "per_n_count": {str(n): bt.B for n, bt in bts.items()},
                "per_n_sub_intervals": {str(n): v for n, v in subs_n.items()},
                "tuned_chunk": {str(n): c for n, c in chunks.items()},
                "tuning_ms": {str(n): {str(c): t for c, t in bt.tuned_timings().items()} for n, bt in bts.items()},
                "status": st, "roofline": rl,
                "cpu_baseline": cpu_baseline_batch(probs)}

    def mixed():
        out = {}
        p = W.point_mass_2d(T=T_headline, K=K_STEPS)
        dp = lqt.DeviceProblem(p)
        ws = torch.empty(lqt.lqt_workspace_size(dp, lqt.LQT_WS_SOLVE), dtype=torch.uint8, device="cuda")
        a, b = lqt.new_solution(dp), lqt.new_solution(dp)
        lqt.lqt_solve(dp, out=a, ws=ws)
        lqt.lqt_solve_mixed(dp, out=b, ws=ws)
        ms64 = _events_ms(lambda: lqt.lqt_solve(dp, out=a, ws=ws), 3)
        ms32 = _events_ms(lambda: lqt.lqt_solve_mixed(dp, out=b, ws=ws), 3)
        import oracle
        got = {k: b[k].cpu().numpy() for k in ("S", "v", "zeta", "x", "u")}
        f64 = {k: a[k].cpu().numpy() for k in ("S", "v", "zeta", "x", "u")}
        del ws, a, b, dp
        ref = oracle.solve(p)
        relm = lambda x, y: float(np.abs(x - y).max() / max(np.abs(y).max(), 1e-300))
        fl = alg_solve(p.n, p.m, p.K)
        out["point_mass_T2^20"] = {
            "value": p.T / (ms32 * 1e-3), "unit": UNIT, "ms_mixed": ms32, "ms_f64": ms64,
            "rel_err_vs_oracle": {k: relm(got[k], ref[k]) for k in got},
            "rel_err_f64_path_vs_oracle": {k: relm(f64[k], ref[k]) for k in f64},
            "roofline": roofline("lqt_solve_mixed n=4", fl, "K (40 n^3 + 60 n^2) + 22 n^3 + 9 n^3 + 2 m n "
                                 "(FP32 products counted as FP64 work)", p.T, ms32, pk),
            "roofline_f64": roofline("lqt_solve n=4", fl, "K (40 n^3 + 60 n^2) + 22 n^3 + 9 n^3 + 2 m n", p.T, ms64,
                                     pk)}
        del got, f64, ref
        p = W.large_state_n64(T=1 << 16)
        dp = lqt.DeviceProblem(p)
        a = lqt.lqt_solve(dp)
        b = lqt.lqt_solve_mixed(dp)
        ms64 = _events_ms(lambda: lqt.lqt_solve(dp, out=a), 1)
        ms32 = _events_ms(lambda: lqt.lqt_solve_mixed(dp, out=b), 1)
        got = {k: b[k].cpu().numpy() for k in ("S", "v", "zeta", "x", "u")}
        S64, v64 = a["S"].cpu().numpy(), a["v"].cpu().numpy()
        del a, b, dp
        # the oracle cannot fold all 2^16 n = 64 elements in seconds: values at
        # the last 256 boundaries against its solve of the last 256
        # sub-intervals, states at the first 257 against its rollout with the
        # FP64 path's values (the checks of tests/test_gpu_mixed.py)
        Ts, T = 256, p.T
        tail = oracle.solve(W.window(p, T - Ts, Ts))
        head = W.window(p, 0, Ts)
        xr, ur = oracle.trajectory(head, oracle.build_elements(head, 0, Ts + 1), S64[:Ts + 1], v64[:Ts + 1], p.x0)
        err = {k: relm(got[k][T - Ts:], tail[k]) for k in ("S", "v", "zeta")}
        err["x"] = relm(got["x"][:Ts + 1], xr)
        err["u"] = relm(got["u"][:Ts + 1], ur)
        fl = alg_solve(p.n, p.m, p.K)
        out["large_state_n64_T2^16"] = {
            "value": p.T / (ms32 * 1e-3), "unit": UNIT, "ms_mixed": ms32, "ms_f64": ms64,
            "f64_value": p.T / (ms64 * 1e-3), "rel_err_vs_oracle": err,
            "rel_err_sample": "values at the last 256 boundaries, states and controls at the first 257",
            "roofline": roofline("lqt_solve_mixed n=64", fl, "K (40 n^3 + 60 n^2) + 22 n^3 + 9 n^3 + 2 m n "
                                 "(FP32 products counted as FP64 work)", p.T, ms32, pk),
            "roofline_f64": roofline("lqt_solve n=64", fl, "K (40 n^3 + 60 n^2) + 22 n^3 + 9 n^3 + 2 m n", p.T,
                                     ms64, pk)}
        out["note"] = ("errors: max |mixed - oracle| / max |oracle| per output; asserted <= 1e-4 in "
                       "tests/test_gpu_mixed.py at these sizes")
        out["cpu_baseline"] = cpu_baseline_sample(W.truncate(W.point_mass_2d(T=T_headline, K=K_STEPS), 1 << 17))
        return out

    def adjoint():
        p = W.differentiable_n8()
        dp = lqt.DeviceProblem(p)
        fwd = lqt.lqt_solve(dp)
        gx = torch.zeros(p.T + 1, p.n, dtype=torch.float64, device="cuda")
        gx[-1] = 2.0 * (fwd["x"][-1] - torch.tensor(p.extra["x_target"], device="cuda"))
        ws = torch.empty(lqt.lqt_workspace_size(dp, lqt.LQT_WS_BACKWARD), dtype=torch.uint8, device="cuda")
        lqt.lqt_backward(dp, fwd, gx=gx, g_cost=1.0, ws=ws)
        fms = _events_ms(lambda: lqt.lqt_solve(dp, out=fwd), 3)
        bms = _events_ms(lambda: lqt.lqt_backward(dp, fwd, gx=gx, g_cost=1.0, ws=ws), 3)
        return {"workload": "n=8, m=4, T=2^14, K=4; loss = cost + |x_T - x_target|^2; gradients w.r.t. F, L, X, U, "
                            "r, Xf, x0", "value": p.T / ((fms + bms) * 1e-3), "unit": UNIT + " (forward + backward)",
                "ms_forward": fms, "ms_backward": bms, "backward_over_forward": bms / fms,
                "workspace_bytes": int(ws.numel()),
                "roofline": roofline("lqt_backward n=8", alg_backward(p.n, p.m, p.K),
                                     "3 K (40 n^3 + 60 n^2) + 2 (22 n^3 + 9 n^3): the elements recomputed once, "
                                     "each forward stage's vector-Jacobian product at twice its work", p.T, bms, pk),
                "roofline_forward": roofline("lqt_solve n=8", alg_solve(p.n, p.m, p.K),
                                             "K (40 n^3 + 60 n^2) + 22 n^3 + 9 n^3 + 2 m n", p.T, fms, pk),
                "cpu_baseline": cpu_baseline_adjoint()}

    def small():
        """The double integrator (T = 1024, K = 10): at this size a solve is
        ~60 dependent short launches, so it is also timed captured in one CUDA
        graph (the calls allocate nothing and never synchronise)."""
        p = W.double_integrator()
        dp = lqt.DeviceProblem(p)
        ws = torch.empty(lqt.lqt_workspace_size(dp, lqt.LQT_WS_SOLVE), dtype=torch.uint8, device="cuda")
        o = lqt.lqt_solve(dp, ws=ws)
        ms = _events_ms(lambda: lqt.lqt_solve(dp, out=o, ws=ws), 20)
        st = torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st):
            lqt.lqt_solve(dp, out=o, ws=ws)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                lqt.lqt_solve(dp, out=o, ws=ws)
        torch.cuda.synchronize()
        graph.replay()
        ms_graph = _events_ms(graph.replay, 20)
        return {"workload": "double integrator n=2, T=1024, K=10", "value": p.T / (ms_graph * 1e-3), "unit": UNIT,
                "ms_graph": ms_graph, "ms_stream_launches": ms, "value_stream_launches": p.T / (ms * 1e-3),
                "roofline": roofline("lqt_solve n=2 (one CUDA graph)", alg_solve(p.n, p.m, p.K),
                                     "K (40 n^3 + 60 n^2) + 22 n^3 + 9 n^3 + 2 m n", p.T, ms_graph, pk),
                "status": lqt.lqt_get_status(), "cpu_baseline": cpu_baseline_sample(p)}

    def densify():
        p = W.point_mass_2d(T=T_headline, K=K_STEPS)
        dp = lqt.DeviceProblem(p)
        ws = torch.empty(lqt.lqt_workspace_size(dp, lqt.LQT_WS_SOLVE), dtype=torch.uint8, device="cuda")
        sol = lqt.lqt_solve(dp, ws=ws)
        d = lqt.lqt_densify(dp, sol)
        wsd = torch.empty(lqt.lqt_workspace_size(dp, lqt.LQT_WS_DENSIFY), dtype=torch.uint8, device="cuda")
        dms = _events_ms(lambda: lqt.lqt_densify(dp, sol, out=d, ws=wsd), 3)
        sms = _events_ms(lambda: lqt.lqt_solve(dp, out=sol, ws=ws), 3)
        fine = p.T * p.K
        return {"workload": "point mass T=2^20, K=4: solution at all 4 194 305 RK4 sub-steps from the boundary "
                            "solution", "value": fine / ((sms + dms) * 1e-3), "unit": "sub-steps/s (solve + densify)",
                "ms_densify": dms, "ms_solve": sms, "status": lqt.lqt_get_status(),
                "roofline": roofline("densify_kernel n=4", alg_densify(p.n, p.m, p.K),
                                     "K [4 (2 n^3 + 4 n^2 m + 2 n^2 + 4 n m) + 4 (2 n^2 + 4 n m)] per sub-interval",
                                     p.T, dms, pk),
                "cpu_baseline": cpu_baseline_densify()}

    def method2():
        p = W.point_mass_2d(T=T_headline, K=K_STEPS)
        dp = lqt.DeviceProblem(p)
        ws = torch.empty(lqt.lqt_workspace_size(dp, lqt.LQT_WS_SOLVE_METHOD2), dtype=torch.uint8, device="cuda")
        m2 = lqt.lqt_solve_method2(dp, ws=ws)
        m1 = lqt.lqt_solve(dp)
        ms = _events_ms(lambda: lqt.lqt_solve_method2(dp, out=m2, ws=ws), 3)
        formula = "2 K (40 n^3 + 60 n^2) + 2 (22 n^3) + 3 n^3 + 2 m n"
        row = {"workload": "point mass T=2^20, K=4: values by the suffix scan, states by Method 2 (forward-ODE "
                           "elements, prefix scan)", "value": p.T / (ms * 1e-3), "unit": UNIT, "ms": ms,
               "rel_diff_vs_method1": {k: _relmax(m2[k], m1[k]) for k in ("x", "u")},
               "roofline": roofline("lqt_solve_method2 n=4", alg_method2(p.n, p.m, p.K), formula, p.T, ms, pk),
               "status": lqt.lqt_get_status(), "cpu_baseline": cpu_baseline_method2()}
        del ws, m2, m1
        # the team kernels: a warp per element and combination (n = 16), a
        # 256-thread CTA (n = 64)
        for name, q in (("n16_m8_K4_T65536", W.batched_member(7, T=1 << 16, n=16)),
                        ("n64_m16_K2_T4096", W.large_state_n64(T=1 << 12))):
            dq = lqt.DeviceProblem(q)
            wq = torch.empty(lqt.lqt_workspace_size(dq, lqt.LQT_WS_SOLVE_METHOD2), dtype=torch.uint8, device="cuda")
            oq = lqt.lqt_solve_method2(dq, ws=wq)
            mq = _events_ms(lambda: lqt.lqt_solve_method2(dq, out=oq, ws=wq), 2)
            row[name] = {"ms": mq, "value": q.T / (mq * 1e-3), "unit": UNIT, "status": lqt.lqt_get_status(),
                         "roofline": roofline(f"lqt_solve_method2 n={q.n}", alg_method2(q.n, q.m, q.K), formula,
                                              q.T, mq, pk)}
            del wq, oq
        return row

    def invariant():
        """The 4096-problem batch and the n = 64 problem with the time-invariant
        element build (every problem there has constant F, L, U, X and a uniform
        grid)."""
        from paper_2212_11744_gb300.batch import BatchSet
        probs = [W.batched_member(b) for b in range(4096)]
        bset = BatchSet(probs)
        bts = bset.batches
        bset.set_invariant_build(True)
        chunks = {n: bt.autotune(candidates=tune_candidates(n), reps=3) for n, bt in bts.items()}
        outs = bset.new_outputs()
        s = torch.cuda.Stream()
        bset.solve(outs, stream=s)
        torch.cuda.synchronize()
        g = bset.capture(outs, stream=s)
        g.replay()
        torch.cuda.synchronize()
        ms = _events_ms(g.replay, 2)
        per = {str(n): _events_ms(lambda bt=bt, o=outs[n]: bt.solve(out=o), 1) for n, bt in bts.items()}
        total = int(sum(p.T for p in probs))
        subs_n = {n: int(bt.T.sum()) for n, bt in bts.items()}
        form = "24 K (n m + n^2) + 22 n^3 + 9 n^3 + 2 m n per sub-interval"
        flop = sum(alg_invariant_solve(n, max(1, n // 2), 4) * subs_n[n] for n in bts)
        rl = roofline("the four batched solves, time-invariant build (one CUDA graph)", flop / total,
                      form + ", averaged", total, ms, pk)
        rl["per_n"] = {str(n): roofline(f"lqt_solve_batched n={n}, time-invariant build",
                                        alg_invariant_solve(n, max(1, n // 2), 4), form, subs_n[n], per[str(n)], pk)
                       for n in bts}
        res = {"workload": "the 4096-problem batch (as a4) with the time-invariant element build",
               "value": total / (ms * 1e-3), "unit": UNIT, "ms": ms, "per_n_ms": per,
               "tuned_chunk": {str(n): c for n, c in chunks.items()},
               "tuning_ms": {str(n): {str(c): t for c, t in bt.tuned_timings().items()} for n, bt in bts.items()},
               "status": lqt.lqt_get_status(), "roofline": rl,
               "cpu_baseline": "as a4 (the oracle's general element build is the reference of this build)"}
        del bts, bset, outs, g
        p = W.large_state_n64(T=1 << 16)
        dp = lqt.DeviceProblem(p)
        try:
            o = lqt.lqt_solve_invariant(dp)
            ims = _events_ms(lambda: lqt.lqt_solve_invariant(dp, out=o), 1)
            res["large_state_n64_T2^16_ms"] = ims
            res["large_state_n64_T2^16_roofline"] = roofline(
                "lqt_solve_invariant n=64", alg_invariant_solve(p.n, p.m, p.K), form, p.T, ims, pk)
        except lqt.LQTError as exc:
            res["large_state_n64_T2^16"] = str(exc)
        return res

    def grid():
        """The nonlinear example of Sec. VI-B on state grids of 20, 40, 60 (the
        paper's) and 201 points, 10^4 blocks of 1/10 with 10 Euler steps each:
        block function plus values at every block boundary.  The unit of work
        is a candidate g_k + f_k of a grid minimisation; evaluated in FP64 each
        costs one FP64 add, so `vs_fp64_add_peak` > 1 is what the kernel's FP32
        screen gains over that bound."""
        import workloads as Wk
        T = 10000
        out = {"workload": "falling body dx/dt = 1 - x^2/10 + u on [-6, 6], T = 10^4 blocks, 10 steps per block, "
                           "App. E interpolated minimum", "unit": "blocks/s", "per_G": {}}
        add_peak = FP64_PEAK_TFLOPS * 1e12 / 2  # DFMA issue slots per second
        for G in (20, 40, 60, 201):
            g = Wk.falling_body(G=G, T=T)
            wb = torch.empty(lqt.lqt_grid_workspace_size(g, 0), dtype=torch.uint8, device="cuda")
            wv = torch.empty(lqt.lqt_grid_workspace_size(g, 1), dtype=torch.uint8, device="cuda")
            Vb = lqt.lqt_grid_block(g, ws=wb)
            V = lqt.lqt_grid_values(g, Vb, ws=wv)

            def path():
                lqt.lqt_grid_block(g, out=Vb, ws=wb)
                lqt.lqt_grid_values(g, Vb, out=V, ws=wv)

            for _ in range(3):
                path()
            ms_stream = _events_ms(path, 5)
            vms = _events_ms(lambda: lqt.lqt_grid_values(g, Vb, out=V, ws=wv), 5)
            # the same calls captured once in a CUDA graph (the ~40 dependent
            # launches of a small grid are launch-latency bound)
            st = torch.cuda.Stream()
            st.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(st):
                path()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=st):
                    path()
            torch.cuda.synchronize()
            graph.replay()
            ms = _events_ms(graph.replay, 5)
            L = T.bit_length()
            pops = sum(bin(e).count("1") for e in range(1, T + 1))
            cand = ((g.substeps - 1) + (L - 1)) * G ** 3 + pops * G * G
            outs_g = ((g.substeps - 1) + (L - 1)) * G ** 2 + pops * G
            fl = cand + 16 * outs_g
            out["per_G"][str(G)] = {"ms": ms, "ms_stream_launches": ms_stream, "ms_values": vms,
                                    "value": T / (ms * 1e-3), "candidates": cand,
                                    "candidates_per_s": cand / (ms * 1e-3),
                                    "vs_fp64_add_peak": cand / (ms * 1e-3) / add_peak,
                                    "roofline": roofline(
                                        f"grid min-plus kernels G={G} (one CUDA graph)", fl / T,
                                        "candidates (one FP64 add each) + 16 flop per output entry for the App. E "
                                        "refinement (its 3 divisions counted as 1 flop each), per block",
                                        T, ms, (pk / 2) if pk else None, peak=FP64_PEAK_TFLOPS / 2,
                                        note="peak: FP64 pipe issue rate (one add per lane slot)")}
            del graph
        out["value"] = out["per_G"]["60"]["value"]
        out["status"] = lqt.lqt_get_status()
        out["cpu_baseline"] = cpu_baseline_grid(Wk.falling_body(G=60, T=T))
        return out

    guard("a4_batched", batched)
    guard("a5_mixed", mixed)
    guard("a6_adjoint", adjoint)
    guard("double_integrator_T1024", small)
    guard("next1_densify", densify)
    guard("next2_method2", method2)
    guard("next3_invariant", invariant)
    guard("next4_grid", grid)
    return rows


def same_tol_sequential(p, par_value: float) -> dict:
    """The paper's sequential method as one GPU thread (lqt_solve_sequential)
    at the parallel path's accuracy.  Truth: the oracle's sequential method
    (O2) with 8K RK4 steps per sub-interval.  The parallel path runs with K
    steps; the sequential sweep's step count is the smallest multiple of K
    whose error (max over S, v, x of max |. - truth| / max |truth|) is at most
    the parallel path's.  Done on the first 2^14 sub-intervals of the
    workload's grid (the timed sample), and on the whole t in [0, 100] at
    T = 2^10 and 2^12, where discretisation error, not rounding, sets the
    step count."""
    import torch

    import oracle
    import paper_2212_11744_gb300 as lqt
    import workloads as W

    def err(a, ref):
        return max(float(np.abs(a[k].cpu().numpy() - ref[k]).max() / np.abs(ref[k]).max()) for k in ("S", "v", "x"))

    def case(q, time_it):
        K = q.K
        truth = oracle.sequential(W.resample(q, 8 * K))
        dq = lqt.DeviceProblem(q)
        par = lqt.lqt_solve(dq)
        torch.cuda.synchronize()
        e_par = err(par, truth)
        tried = {}
        ks = None
        for mult in range(1, 9):
            Ks = mult * K
            dqs = lqt.DeviceProblem(W.resample(q, Ks) if Ks != K else q)
            sq = lqt.lqt_solve_sequential(dqs)
            torch.cuda.synchronize()
            tried[str(Ks)] = err(sq, truth)
            if tried[str(Ks)] <= e_par:
                ks = Ks
                break
        res = {"T": q.T, "K_parallel": K, "rel_err_parallel_vs_O2_8K": e_par, "K_sequential_same_tol": ks,
               "rel_err_sequential_vs_O2_8K": tried}
        if time_it and ks is not None:
            dqs = lqt.DeviceProblem(W.resample(q, ks) if ks != K else q)
            sq = lqt.lqt_solve_sequential(dqs)
            ms = _events_ms(lambda: lqt.lqt_solve_sequential(dqs, out=sq), 1)
            pms = _events_ms(lambda: lqt.lqt_solve(dq, out=par), 3)
            res.update({"ms_sequential": ms, "ms_parallel": pms, "value": q.T / (ms * 1e-3),
                        "value_parallel_same_T": q.T / (pms * 1e-3), "speedup_same_T": ms / pms})
        return res

    head = case(W.truncate(p, min(1 << 14, p.T)), True)
    coarse = {str(T): case(W.point_mass_2d(T=T, K=p.K), True) for T in (1 << 10, 1 << 12)}
    out = {"value": head.get("value"), "unit": UNIT, "T_timed": head["T"],
           "K_sequential_same_tol": head["K_sequential_same_tol"],
           "speedup_parallel_over_sequential": (par_value / head["value"]) if head.get("value") else None,
           "sample": head, "coarse_grids": coarse,
           "tol_note": "errors against the oracle's sequential method at 8K RK4 steps per sub-interval; the "
                       "sequential sweep's steps searched over multiples of K; the headline speed-up divides the "
                       "T = 2^20 parallel rate by the sequential rate on the first 2^14 sub-intervals"}
    return out


# ---------------------------------------------------------------------------
# our arm
# ---------------------------------------------------------------------------

def run_ours(args):
    import torch

    import paper_2212_11744_gb300 as lqt
    import workloads as W

    ws_, rank, local = dist_setup()
    p = W.point_mass_2d(T=args.T, K=K_STEPS)
    dp = lqt.DeviceProblem(p)
    stream = torch.cuda.current_stream()
    ws = torch.empty(lqt.lqt_workspace_size(dp, lqt.LQT_WS_SOLVE), dtype=torch.uint8, device="cuda")
    out = lqt.new_solution(dp)

    def step():
        lqt.lqt_solve(dp, out=out, ws=ws, stream=stream)

    for _ in range(args.warmup):
        step()
    barrier(ws_)
    st = lqt.lqt_get_status(stream)
    if st != 0:
        raise RuntimeError("device status: " + lqt.lqt_strerror(st))
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clk:
        barrier(ws_)
        e0.record(stream)
        for _ in range(args.steps):
            step()
        e1.record(stream)
        torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / args.steps
    launches_per_step = lqt.lqt_last_launch_count()
    ms = max_over_ranks(ms, ws_)
    value = p.T * ws_ / (ms * 1e-3)

    # dominant stage: element build, timed alone (same stream, events)
    el = lqt.new_elements(dp)
    wsb = torch.empty(lqt.lqt_workspace_size(dp, lqt.LQT_WS_BUILD), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        lqt.lqt_build_elements(dp, out=el, ws=wsb, stream=stream)
    reps = max(3, args.steps)
    e0.record(stream)
    for _ in range(reps):
        lqt.lqt_build_elements(dp, out=el, ws=wsb, stream=stream)
    e1.record(stream)
    torch.cuda.synchronize()
    build_ms = e0.elapsed_time(e1) / reps
    m_pad = 1 if p.m <= 1 else 2 if p.m <= 2 else 4 if p.m <= 4 else 8
    fl_build = algorithmic_build_flops_per_block(p.n, p.K) * p.T
    achieved = fl_build / (build_ms * 1e-3) / 1e12
    achieved_impl = build_flops_per_block(p.n, m_pad, p.K, p.c is not None) * p.T / (build_ms * 1e-3) / 1e12
    del el, wsb

    # end to end through the host-buffer entry point
    hp = lqt.HostProblem(p, pinned=True)
    hout = lqt.host_solution(hp, pinned=True)
    wsh = torch.empty(lqt.lqt_workspace_size(hp, lqt.LQT_WS_SOLVE) + lqt.lqt_host_staging_size(hp) + 4096,
                      dtype=torch.uint8, device="cuda")
    lqt.lqt_solve_host(hp, wsh, out=hout, stream=stream)
    e2e_steps = max(2, min(args.steps, 5))
    barrier(ws_)
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        lqt.lqt_solve_host(hp, wsh, out=hout, stream=stream)
    e2e_s = max_over_ranks((time.perf_counter() - t0) / e2e_steps, ws_)
    h2d = sum(t.numel() * t.element_size() for t in hp.keep)
    d2h = sum(t.numel() * t.element_size() for t in hout.values())
    np.testing.assert_array_equal(hout["x"].numpy(), out["x"].cpu().numpy())
    del wsh

    # the sequential one-thread GPU sweep at the same tolerance
    seq = same_tol_sequential(p, value / ws_) if rank == 0 else None
    pk = probe_pipes() if rank == 0 else None

    rows = measure_rows(args.T, pk["fp64_tflops"]) if (args.rows and rank == 0) else None

    if rank == 0:
        cpu = cpu_baseline_sample(p)
        traffic = profiled_traffic()
        clocks = clk.summary()
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws_, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": dict(workload_config(p), parallelism=f"replicas x{ws_}"),
            "gpu_launches": launches_per_step * args.steps,
            "roofline": {"bound": "alu", "kernel": "build_kernel<4,2> (stage a, with its prepare/terminal launches)",
                         "achieved": achieved, "peak": FP64_PEAK_TFLOPS, "unit": "TFLOP/s",
                         "frac": achieved / FP64_PEAK_TFLOPS, "traffic": traffic,
                         "peak_source": "FP64 pipe: 152 SMs x 4 sub-partitions x 0.5 DFMA/clk x 2 flop x 2.07 GHz",
                         "peak_measured": pk["fp64_tflops"] if pk else None,
                         "frac_of_measured": achieved / pk["fp64_tflops"] if pk else None,
                         "stage_ms": build_ms,
                         "flop_per_unit": "K (40 n^3 + 60 n^2) per sub-interval (dense element right-hand side)",
                         "achieved_as_implemented": achieved_impl,
                         "frac_as_implemented": achieved_impl / FP64_PEAK_TFLOPS},
            "roofline_step": roofline("lqt_solve n=4 (whole step)", alg_solve(p.n, p.m, p.K),
                                      "K (40 n^3 + 60 n^2) + 22 n^3 + 9 n^3 + 2 m n per sub-interval", p.T, ms,
                                      pk["fp64_tflops"] if pk else None),
            "e2e": {"value": p.T * ws_ / e2e_s, "unit": UNIT, "h2d_bytes_per_step": h2d,
                    "d2h_bytes_per_step": d2h},
            "sequential_gpu": seq,
            "pipes_measured": pk,
            "cpu_baseline": cpu,
            "clocks": clocks,
            "rows": rows,
        }
        print(json.dumps(line), file=sys.stderr)
        print(json.dumps(result_line(line)))
    if ws_ > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def result_line(full):
    """The one line on stdout: the result and what qualifies it, below 2000
    characters, so that a reader of a log's tail gets it whole.  The full record,
    with every row's notes, is one JSON line on stderr."""
    pick = lambda d, *keys: {k: d[k] for k in keys} if d else d
    line = {k: v for k, v in full.items() if k not in ("roofline_step", "pipes_measured", "rows")}
    line["roofline"] = pick(full["roofline"], "bound", "kernel", "achieved", "peak", "unit", "frac", "traffic")
    line["sequential_gpu"] = pick(full["sequential_gpu"], "value", "unit", "T_timed", "speedup_parallel_over_sequential")
    line["cpu_baseline"] = pick(full["cpu_baseline"], "value", "unit", "cores")
    return line


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--T", type=int, default=T_DEFAULT)
    ap.add_argument("--rows", type=int, default=1, help="also measure the batched, mixed-precision and adjoint rows")
    args = ap.parse_args()
    if args.warmup < 3 and args.impl == "ours":
        args.warmup = 3
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()

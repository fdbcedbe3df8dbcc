#!/usr/bin/env python3
"""Benchmark: matrix-free CP-ALS of the DF particle-particle-ladder tensor on GB300.

Workload: one PPL instance with o=20 occupied, v=200 virtual, X=600 auxiliary
orbitals and CP rank R=800, seeded synthetic inputs shaped like the paper's
molecules (paper_2503_10380_gb300/inputs.py).  One step = one ALS sweep
(modes a, b, i, j) with TF32x3 tensor-core MTTKRPs (tf32 hi/lo split,
accumulator restarted every K block) and FP64 Gram / Cholesky / solve / fit.
BF16x3 is timed beside it with its energy error.  Prints one JSON line on rank 0.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                  [--workload single|batch|precision|sequence] [--precision bf16x3|tf32|tf32x3]

For N > 1 (one process per GPU under torchrun) every rank runs an
independent replica (the method has no exchange step on one instance):
value = N * K / max over ranks of the timed region.
"""

from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "CP-ALS sweeps/s & MTTKRP TFLOP/s at ≤0.1 kcal/mol ΔE vs plain FP64 on GPU"
SEED = 0
KCAL = 627.509474
MAIN_CFG = (60, 600, 1800, 2400)   # the largest single-GPU configuration (o, v, X, R)
CFG1 = (20, 200, 600, 800)
CFG2 = (40, 400, 1200, 1600)
O, V, XAUX, RANK = CFG1            # the instance the oracle's flop rate is timed on for estimates
ACC_SWEEPS_MAIN = 2                # sweeps compared against the FP64 GPU form (about 3 s per FP64 sweep)
E2E_SWEEPS, E2E_STEPS = 10, 2
def _workload(cfg):
    return f"cp-als-ppl single instance o={cfg[0]} v={cfg[1]} X={cfg[2]} R={cfg[3]}, graph-replayed ALS sweeps"


WORKLOAD = _workload(MAIN_CFG)


def set_main_cfg(cfg):
    """Run the single-instance benchmark (and the reference arm) on another size."""
    global MAIN_CFG, WORKLOAD
    MAIN_CFG = tuple(cfg)
    WORKLOAD = _workload(MAIN_CFG)


def alg_flops(o, v, X, R):
    """Algorithmic MTTKRP flops of one sweep: 4 o^2 v^2 R + 16 X v^2 R."""
    return 4.0 * o * o * v * v * R + 16.0 * X * v * v * R


def reduce_max(x: float, world: int, dev=None) -> float:
    """Max over ranks (the slowest replica sets the whole-job time)."""
    if world <= 1:
        return x
    import torch
    t = torch.tensor([float(x)], dtype=torch.float64, device=dev if dev is not None else "cpu")
    torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
    return float(t.item())


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def oracle_cores():
    try:
        from threadpoolctl import threadpool_info
        n = [i.get("num_threads") for i in threadpool_info() if i.get("user_api") == "blas"]
        if n:
            return int(max(n)), "threadpoolctl"
    except Exception:
        pass
    return os.cpu_count() or 1, "nproc (BLAS default thread count)"


def time_oracle_sweeps(inp, R_s, nsweeps):
    """Time `nsweeps` FP64 oracle sweeps of the rank-R_s problem on the host cores."""
    import numpy as np
    from oracle import ppl_oracle as orc
    U = {m: inp.factors[m][:, :R_s].copy() for m in orc.MODES}
    lam = np.ones(R_s)
    Bvv = np.ascontiguousarray(inp.Bvv)
    t0 = time.perf_counter()
    for _ in range(nsweeps):
        U, lam, _ = orc.als_sweep(Bvv, inp.tau, U, lam)
    return time.perf_counter() - t0


def oracle_estimate(o, v, X, R):
    """CPU baseline for a size too large to time the oracle on: one FP64 oracle sweep of
    the o=20 v=200 X=600 R=800 instance is timed on the host cores and its MTTKRP-flop
    rate is scaled to (o, v, X, R).  Labelled as an estimate."""
    from paper_2503_10380_gb300 import inputs
    inp = inputs.make_inputs(O, V, XAUX, RANK, seed=SEED)
    t = time_oracle_sweeps(inp, RANK, 1)
    rate = alg_flops(O, V, XAUX, RANK) / t
    cores, how = oracle_cores()
    return {"value": rate / alg_flops(o, v, X, R), "unit": "sweeps/s", "cores": cores, "kind": "oracle",
            "estimate": True,
            "sample": f"estimate: one FP64 oracle sweep of o={O} v={V} X={XAUX} R={RANK} took {t:.2f} s "
                      f"({rate / 1e9:.1f} GFLOP/s of MTTKRP flops), scaled by 4o^2v^2R + 16Xv^2R to "
                      f"o={o} v={v} X={X} R={R}; threads from {how}"}


class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.idx = gpu_index
        self.p = None
        try:
            self.p = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                       "-lms", "50"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.p = None

    def stop(self):
        if self.p is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        self.p.terminate()
        try:
            out, _ = self.p.communicate(timeout=5)
        except Exception:
            self.p.kill()
            out, _ = self.p.communicate()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                if int(f[0]) != self.idx:
                    continue
                sm.append(float(f[1]))
                smax.append(float(f[2]))
            except ValueError:
                continue
            for name, val in zip(names, f[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        d = json.load(open(p))
        return d, "measured"
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}, "fallback"


def traffic_from_profile(key: str, prof_name: str = "mttkrp_tc_cfg4_traffic.json",
                         src_names=("ppl_tc.cu", "ppl_cpd.cu")):
    """DRAM bytes per sweep from a committed ncu summary (profiles/<prof_name>)
    if it was taken on the current sources of the kernels and their
    orchestration; else None."""
    prof = os.path.join(ROOT, "profiles", prof_name)
    try:
        d = json.load(open(prof))
        for src_name in src_names:
            src = os.path.join(ROOT, "paper_2503_10380_gb300", "csrc", src_name)
            h = hashlib.sha256(open(src, "rb").read()).hexdigest()
            if d.get(src_name.replace(".cu", "") + "_sha256") != h:
                return None
        return d.get(key)
    except Exception:
        return None


def tensor_peak(pk, precision):
    """Algorithmic-flop peak of a tensor-core precision: the dtype's sustained
    rate divided by the MMAs issued per product (three for the split forms).
    pk: measure_peaks() of this run (TF32); bf16 from MEASURED_PEAKS.json."""
    bf16 = peaks()[0]["bf16_tflops_sustained"]
    tf32 = pk["tf32_tflops_sustained"]
    return {"bf16x3": (bf16 / 3.0, "sustained bf16 (MEASURED_PEAKS.json) / 3 (three bf16 MMAs per product)"),
            "tf32": (tf32, "sustained TF32 measured in this run"),
            "tf32x3": (tf32 / 3.0, "sustained TF32 measured in this run / 3 (three tf32 MMAs per product)")}[precision]


def main_config(world):
    """The workload's identity, the same dict in both arms."""
    o, v, X, R = MAIN_CFG
    gb = (o * o * v * v + X * (o + v) ** 2) * 8 / 1e9
    return {"workload": WORKLOAD, "o": o, "v": v, "X": X, "R": R,
            "l2": f"inputs larger than L2 (tau and B {gb:.2f} GB)",
            "parallelism": "replicas" if world > 1 else "single GPU"}


class _HostInputs:
    """The oracle's view of one instance: B_vv, tau and the initial factors on the host."""

    def __init__(self, Bvv, tau, factors):
        self.Bvv, self.tau, self.factors = Bvv, tau, factors


def host_inputs(cfg, dev=None):
    """Seeded inputs of `cfg` for the oracle.  Generated with the torch version of
    the generator (on the GPU when there is one: setup only, outside every timed
    region) and copied to host numpy arrays."""
    import numpy as np
    import torch
    from paper_2503_10380_gb300 import inputs
    o, v, X, R = cfg
    d = dev if dev is not None else ("cuda" if torch.cuda.is_available() else "cpu")
    B, tau, fac = inputs.make_inputs_torch(o, v, X, R, seed=SEED, device=d)
    Bvv = np.ascontiguousarray(B[:, o:, o:].cpu().numpy())
    tau_h = tau.cpu().numpy()
    del B, tau
    if torch.cuda.is_available():
        torch.cuda.empty_cache()
    return _HostInputs(Bvv, tau_h, fac)


def oracle_sample(inp, R, budget_s, nsweeps=2):
    """Oracle sweeps/s of the full rank-R problem from sweeps over its first R_s
    rank columns: the MTTKRP work of a column does not depend on the others and
    the R_s-column solves are a negligible part, so the full problem's sweep
    takes R / R_s times as long.  R_s is sized from a calibration sweep so that
    the timed sweeps take about budget_s."""
    t_cal = time_oracle_sweeps(inp, 8, 1)
    R_s = int(max(8, min(R, budget_s / nsweeps / (t_cal / 8))))
    t = time_oracle_sweeps(inp, R_s, nsweeps)
    return (nsweeps * R_s / R) / t, R_s, t


def run_reference(args, world, rank):
    if rank != 0:
        return
    o, v, X, R = MAIN_CFG
    inp = host_inputs(MAIN_CFG)
    # each step: one oracle sweep over the first R_s rank columns, R_s sized so
    # that the whole --steps K --warmup W run stays within about 150 s
    budget = 150.0
    t_cal = time_oracle_sweeps(inp, 8, 1)
    R_s = int(max(8, min(R, (budget / max(args.steps + args.warmup, 1)) / (t_cal / 8))))
    for _ in range(args.warmup):
        time_oracle_sweeps(inp, R_s, 1)
    t = time_oracle_sweeps(inp, R_s, args.steps)
    value = (args.steps * R_s / R) / t
    cores, how = oracle_cores()
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "sweeps/s", "n_gpus": 1,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000.0 / value,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic (seeded; shapes of the paper's molecules)",
        "config": main_config(1),
        "cpu_baseline": {"value": value, "unit": "sweeps/s", "cores": cores, "kind": "oracle",
                         "sample": f"{args.steps} FP64 oracle sweeps over the first {R_s} of {R} rank columns, "
                                   f"scaled by {R}/{R_s}; threads from {how}"},
        "e2e": {"value": value, "unit": "sweeps/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def measure_peaks(dev, stream):
    """Peaks measured in this run (the roofline denominators): TF32 dense
    throughput of a square cuBLAS GEMM (8192^3, TF32 allowed), best of 10 (burst)
    and back to back for about 2 s (sustained); FP64 FMA throughput of the
    library's own probe kernel.  Measurement only: nothing on the hot path calls
    cuBLAS."""
    import torch
    from paper_2503_10380_gb300 import binding
    prev = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = True
    n = 8192
    a = torch.randn(n, n, device=dev)
    b = torch.randn(n, n, device=dev)
    for _ in range(3):
        c = a @ b
    torch.cuda.synchronize()
    best = 1e30
    for _ in range(10):
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        c = a @ b
        e1.record(stream)
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    reps = max(1, int(2000.0 / best))
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(reps):
        c = a @ b
    e1.record(stream)
    torch.cuda.synchronize()
    sust = e0.elapsed_time(e1) / reps
    torch.backends.cuda.matmul.allow_tf32 = prev
    del a, b, c
    torch.cuda.empty_cache()
    fl = 2.0 * n ** 3
    fp64 = binding.ppl_probe_fp64_peak(stream.cuda_stream)
    return {"tf32_tflops": fl / (best * 1e-3) / 1e12, "tf32_tflops_sustained": fl / (sust * 1e-3) / 1e12,
            "fp64_tflops": fp64,
            "how": "tf32: torch.matmul 8192^3 with TF32 allowed, best of 10 (burst) and back to back for ~2 s "
                   "(sustained); fp64: ppl_probe_fp64_peak (independent FMA chains on every SM, best of 3)"}


def fp64_solve_flops(o, v, R):
    """Algorithmic FP64 flops of the four mode updates of one sweep, per mode
    R^3/3 (Cholesky) + 2 dim R^2 (the two triangular solves of M V^-1) + 2 dim R^2
    (the new factor's Gram matrix)."""
    return 4 * (R ** 3 / 3.0) + 4.0 * R * R * (2 * v + 2 * o)


def _factors_host(cp):
    return {k: t.cpu().numpy().copy() for k, t in cp.factors().items()}


def factor_errors(F, F64):
    """Relative error of every factor against the FP64 GPU form: normwise, and
    the worst element relative to the largest entry of its column."""
    import numpy as np
    out = {}
    for m in F64:
        a, b = np.atleast_2d(F[m]), np.atleast_2d(F64[m])
        col = np.max(np.abs(a - b), axis=0) / np.maximum(np.max(np.abs(b), axis=0), 1e-300)
        out[m] = {"norm": float(np.linalg.norm(a - b) / np.linalg.norm(b)), "col_max": float(np.max(col))}
    return out


def _time_sweeps(cp, n, stream):
    import torch
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(stream)
    cp.sweep(n, want_hist=False)
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / n


def _phases(cp, n=3):
    acc = None
    for _ in range(n):
        cp.sweep(1, want_hist=False)
        ph = cp.phase_ms()
        acc = ph if acc is None else {k: acc[k] + ph[k] for k in acc}
    return {k: acc[k] / n for k in acc}


MTTKRP_PHASES = ("tau_r", "chain_a", "chain_b", "s_and_p")
SOLVE_PHASES = ("solve_a", "solve_b", "solve_ij")


def accuracy_vs_fp64(B, tau, fac, precision, r_chunk, k, stream, E_exact=None, mttkrp_modes="abij", normR2=None):
    """k sweeps from the same start in `precision` and in the plain FP64 GPU form:
    energy difference (kcal/mol and relative), per-factor errors, and the FP64
    form's time per sweep (its first sweep captures the graph and is not timed).
    Before the sweeps, the MTTKRP of each mode in `mttkrp_modes` from the common
    starting factors in both forms: modes a and b run T, W, Y and M (the chain),
    modes i and j the S-build (W_a, W_b, S, P), so their errors locate where the
    split precision loses accuracy.  With normR2 (||R||^2), also the fit of both
    forms after the k sweeps (Eq. cpfit through the residual expansion): their
    difference is the noise floor a |delta fit| stopping test meets in the split
    precision."""
    import torch
    from paper_2503_10380_gb300 import binding
    mixed = binding.CpAls(B, tau, fac, precision=precision, r_chunk=r_chunk)
    M_mixed = {m: mixed.mttkrp(m).cpu().numpy() for m in mttkrp_modes}
    if normR2 is not None:
        mixed.set_normR2(normR2)
    mixed.sweep(k, want_hist=False)
    fit_mixed = mixed.fit() if normR2 is not None else None
    E_mixed, F_mixed = mixed.energy(), _factors_host(mixed)
    mixed.close()
    del mixed
    torch.cuda.empty_cache()
    f64 = binding.CpAls(B, tau, fac, precision="fp64")
    M64 = {m: f64.mttkrp(m).cpu().numpy() for m in mttkrp_modes}
    if normR2 is not None:
        f64.set_normR2(normR2)
    f64.sweep(1, want_hist=False)
    f64_ms = _time_sweeps(f64, k - 1, stream) if k > 1 else None
    fit64 = f64.fit() if normR2 is not None else None
    E64, F64 = f64.energy(), _factors_host(f64)
    f64.close()
    del f64
    torch.cuda.empty_cache()
    d = abs(E_mixed - E64)
    out = {"sweeps": k, "E_cp_mixed": E_mixed, "E_cp_fp64": E64, "dE_kcal_per_mol": d * KCAL,
           "dE_rel": d / abs(E64), "meets_0.1_kcal": d * KCAL <= 0.1,
           "factor_rel_err": factor_errors(F_mixed, F64), "fp64_ms_per_sweep": f64_ms,
           "mttkrp_rel_err_at_start": factor_errors(M_mixed, M64)}
    if normR2 is not None:
        out["fit_mixed"], out["fit_fp64"] = fit_mixed, fit64
        out["fit_abs_diff"] = abs(fit_mixed - fit64)
    if E_exact is not None:
        out["E_exact"] = E_exact
        out["rank_error_kcal_per_mol"] = abs(E64 - E_exact) * KCAL
    return out


def secondary_config(cfg, precision, k_acc, steps, stream, dev, pk):
    """A second configuration in the same run: sweep rate, MTTKRP TFLOP/s, and the
    accuracy of `precision` against the FP64 GPU form after k_acc sweeps."""
    import torch
    from paper_2503_10380_gb300 import binding, inputs
    o, v, X, R = cfg
    B, tau, fac = inputs.make_inputs_torch(o, v, X, R, seed=SEED, device=dev)
    cp = binding.CpAls(B, tau, fac, precision=precision, profile=True)
    rc = cp.autotune()
    cp.sweep(3, want_hist=False)
    ms = _time_sweeps(cp, steps, stream)
    ph = _phases(cp)
    cp.close()
    del cp
    torch.cuda.empty_cache()
    mt_ms = sum(ph[q] for q in MTTKRP_PHASES)
    acc = accuracy_vs_fp64(B, tau, fac, precision, rc, k_acc, stream)
    del B, tau
    torch.cuda.empty_cache()
    tf = alg_flops(o, v, X, R) / (mt_ms / 1e3) / 1e12
    return {"workload": f"cp-als-ppl single instance o={o} v={v} X={X} R={R}", "o": o, "v": v, "X": X, "R": R,
            "r_chunk": rc, "sweeps_per_s": 1000.0 / ms, "ms_per_sweep": ms, "mttkrp_tflops": tf,
            "mttkrp_frac_of_sustained_peak": tf / (pk["tf32_tflops_sustained"] / 3.0), "phase_ms": ph,
            "accuracy": acc,
            "speedup_vs_fp64_gpu": (acc["fp64_ms_per_sweep"] / ms) if acc["fp64_ms_per_sweep"] else None}


def run_ours(args, world, rank, local):
    import numpy as np
    import torch
    from paper_2503_10380_gb300 import binding, inputs
    import __graft_entry__
    if rank == 0:
        __graft_entry__.build()
    if world > 1:
        torch.distributed.barrier()
    binding.lib()
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    stream = torch.cuda.current_stream(dev)

    def barrier():
        if world > 1:
            torch.distributed.barrier()

    pk = measure_peaks(dev, stream)
    o, v, X, R = MAIN_CFG
    B, tau, fac = inputs.make_inputs_torch(o, v, X, R, seed=SEED, device=dev)
    cp = binding.CpAls(B, tau, fac, precision=args.precision, profile=True, r_chunk=args.r_chunk)
    if not args.r_chunk:
        args.r_chunk = cp.autotune()       # the library's own r-chunk autotuner (before the timed region)
    for _ in range(args.warmup):
        cp.sweep(1, want_hist=False)
    torch.cuda.synchronize()

    # ---- timed region: K back-to-back graph-replayed sweeps -------------------
    clocks = ClockSampler(local)
    time.sleep(0.3)
    barrier()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    torch.cuda.nvtx.range_push("timed")
    e0.record(stream)
    cp.sweep(args.steps, want_hist=False)
    e1.record(stream)
    torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()
    barrier()
    ck = clocks.stop()
    ms = reduce_max(e0.elapsed_time(e1), world, dev)
    ms_per_step = ms / args.steps
    value = world * args.steps / (ms / 1000.0)
    launches = int(cp.stats()["kernels_per_sweep"])

    # ---- phase breakdown (CUDA events recorded by the library on its stream) --
    phases = _phases(cp, min(args.steps, 3))
    mttkrp_ms = sum(phases[q] for q in MTTKRP_PHASES)
    solve_ms = sum(phases[q] for q in SOLVE_PHASES)
    flops = alg_flops(o, v, X, R)
    mttkrp_tflops = flops / (mttkrp_ms / 1000.0) / 1e12

    # ---- end to end through the C ABI with host buffers -----------------------
    # one CC-like step: tau copied from pinned host memory, its operand copies
    # rebuilt, E2E_SWEEPS sweeps warm-started from the factors on the device,
    # then the factors and the fit history read back.  B stays resident (the DF
    # integrals do not change between CC iterations).
    tau_h = torch.empty(tau.shape, dtype=tau.dtype, pin_memory=True)
    tau_h.copy_(tau)
    fac_out = torch.empty(cp.fac.numel(), dtype=torch.float64).pin_memory()

    def e2e_step():
        cp.tau.copy_(tau_h, non_blocking=True)
        binding.ppl_cpd_set_tau(cp.h, cp.tau.data_ptr())
        hist = cp.sweep(E2E_SWEEPS, want_hist=True)
        fac_out.copy_(cp.fac, non_blocking=True)
        torch.cuda.current_stream(dev).synchronize()
        return hist

    e2e_step()
    barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(E2E_STEPS):
        e2e_step()
    torch.cuda.synchronize()
    t_e2e = reduce_max(time.perf_counter() - t0, world, dev)
    e2e_value = world * E2E_STEPS * E2E_SWEEPS / t_e2e
    h2d = tau_h.numel() * 8
    d2h = fac_out.numel() * 8 + E2E_SWEEPS * 8
    del tau_h
    # ||R||^2 and E_exact once, from the tensor-core exact contraction
    t0 = time.perf_counter()
    normR2, E_exact, _ = cp.exact_contract(mixed=True)
    t_exact = time.perf_counter() - t0
    cp.close()
    del cp
    torch.cuda.empty_cache()

    # ---- accuracy against the plain FP64 GPU form from the same start ---------
    acc = accuracy_vs_fp64(B, tau, fac, args.precision, args.r_chunk, ACC_SWEEPS_MAIN, stream, E_exact,
                           mttkrp_modes="ai", normR2=normR2)
    del B, tau
    torch.cuda.empty_cache()

    # ---- the other single-instance configurations, in the same run ------------
    secondary = {}
    if not args.no_secondary:
        secondary["o=20 v=200 X=600 R=800"] = secondary_config(CFG1, args.precision, 30, 20, stream, dev, pk)
        secondary["o=40 v=400 X=1200 R=1600"] = secondary_config(CFG2, args.precision, 5, 10, stream, dev, pk)
        # the batch of uneven instances in the precision its configuration names (BF16 split)
        secondary["batch of 64"] = batch_secondary(dev, "bf16x3")

    # ---- CPU baseline: the oracle on the host cores (rank 0, N = 1) -----------
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        hin = host_inputs(MAIN_CFG, dev)
        val, R_s, t_or = oracle_sample(hin, R, 20.0)
        del hin
        cores, how = oracle_cores()
        cpu = {"value": val, "unit": "sweeps/s", "cores": cores, "kind": "oracle",
               "sample": f"2 FP64 oracle sweeps of the o={o} v={v} X={X} instance over its first {R_s} of {R} rank "
                         f"columns ({t_or:.1f} s), scaled by {R}/{R_s}; threads from {how}"}

    peak_tc = pk["tf32_tflops_sustained"] / 3.0
    solve_tflops = fp64_solve_flops(o, v, R) / (solve_ms / 1000.0) / 1e12
    roof_solve = {"bound": "alu", "achieved": solve_tflops, "peak": pk["fp64_tflops"], "unit": "TFLOP/s",
                  "frac": solve_tflops / pk["fp64_tflops"],
                  "traffic": traffic_from_profile("solve_bytes_per_sweep", src_names=("ppl_solve.cu", "ppl_cpd.cu"))
                  if MAIN_CFG == (60, 600, 1800, 2400) else None, "ms_per_sweep": solve_ms,
                  "kernel": "k_solve (FP64 mode updates, cooperative, 4 launches per sweep)",
                  "peak_source": "measured in this run: ppl_probe_fp64_peak (FP64 FMA chains on every SM)",
                  "work": "per sweep 4 (R^3/3 + 4 dim R^2) FP64 flops: Cholesky, two triangular solves, Gram"}
    roof_mttkrp = {"bound": "tensor", "achieved": mttkrp_tflops, "peak": peak_tc, "unit": "TFLOP/s",
                   "frac": mttkrp_tflops / peak_tc,
                   "traffic": traffic_from_profile("mttkrp_bytes_per_sweep") if MAIN_CFG == (60, 600, 1800, 2400) else None,
                   "traffic_unit": "DRAM bytes per sweep (ncu, profiles/mttkrp_tc_cfg4_traffic.json)",
                   "ms_per_sweep": mttkrp_ms,
                   "kernel": "k_tc_gemm and its helpers (all MTTKRP contractions of one sweep)",
                   "peak_source": "measured in this run: sustained TF32 cuBLAS GEMM / 3 (three tf32 MMAs per "
                                  "product); burst TF32 / 3 = %.1f TFLOP/s" % (pk["tf32_tflops"] / 3.0),
                   "work": "per sweep 4 o^2 v^2 R + 16 X v^2 R algorithmic flops"}
    dominant = roof_mttkrp if mttkrp_ms >= solve_ms else roof_solve
    line = {
        "metric": METRIC, "value": value, "unit": "sweeps/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": args.precision,
        "data": "synthetic (seeded; shapes of the paper's molecules)",
        "config": main_config(world),
        "precision": args.precision, "r_chunk": args.r_chunk,
        "mttkrp_tflops": mttkrp_tflops,
        "phase_ms": phases,
        "roofline": dominant,
        "roofline_mttkrp": roof_mttkrp,
        "roofline_solve": roof_solve,
        "peaks_measured": pk,
        "fp64_gpu": {"ms_per_sweep": acc["fp64_ms_per_sweep"],
                     "speedup_mixed_vs_fp64": (acc["fp64_ms_per_sweep"] / ms_per_step)
                     if acc["fp64_ms_per_sweep"] else None},
        "accuracy": acc,
        "exact_contract_s": t_exact,
        "e2e": {"value": e2e_value, "unit": "sweeps/s", "h2d_bytes_per_step": int(h2d),
                "d2h_bytes_per_step": int(d2h),
                "step": f"one warm-started CC-like step: tau H2D from pinned memory, operand rebuild, {E2E_SWEEPS} "
                        f"sweeps, factors + fit history D2H"},
        "secondary": secondary,
        "gpu_launches": launches * args.steps,
        "clocks": {k: ck[k] for k in ("sm_mhz", "sm_max_mhz", "reasons")},
        "clock_samples": ck["samples"],
        "cpu_baseline": cpu,
    }
    if rank == 0:
        print(json.dumps(line), flush=True)


def run_batch(args, world, rank, local):
    """64 uneven instances (o in [4,24], v in [40,240], X = 3v, R in [2v,4v]) swept
    together from one CUDA graph; one step = one sweep of every instance."""
    import numpy as np
    import torch
    from paper_2503_10380_gb300 import binding, inputs
    import __graft_entry__
    if rank == 0:
        __graft_entry__.build()
    if world > 1:
        torch.distributed.barrier()
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    shapes = inputs.batch_shapes(64, seed=SEED)
    data = [inputs.make_inputs_torch(*sh, seed=SEED + k, device=dev) for k, sh in enumerate(shapes)]
    flops = sum(alg_flops(*sh) for sh in shapes)
    probs = []
    for (B, tau, fac) in data:
        cp = binding.CpAls(B, tau, fac, precision=args.precision)
        cp.autotune()
        probs.append(cp)
    batch = binding.Batch(probs, nstreams=8)
    batch.sweep(args.warmup, want_fits=False)
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream(dev)
    clocks = ClockSampler(local)
    time.sleep(0.3)
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    torch.cuda.nvtx.range_push("timed")
    e0.record(stream)
    batch.sweep(args.steps, want_fits=False)
    e1.record(stream)
    torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()
    ck = clocks.stop()
    ms = reduce_max(e0.elapsed_time(e1), world, dev)
    launches = batch.kernels_per_sweep()
    # plain FP64 form of the same batch
    f64 = [binding.CpAls(B, tau, fac, precision="fp64") for (B, tau, fac) in data]
    fb = binding.Batch(f64, nstreams=8)
    fb.sweep(1, want_fits=False)
    torch.cuda.synchronize()
    g0 = torch.cuda.Event(enable_timing=True)
    g1 = torch.cuda.Event(enable_timing=True)
    g0.record(stream)
    fb.sweep(2, want_fits=False)
    g1.record(stream)
    torch.cuda.synchronize()
    f64_ms = g0.elapsed_time(g1) / 2
    fb.close()
    for p in f64:
        p.close()
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        # oracle sweeps over the first instances until ~15 s, scaled by flops to the batch
        from oracle import ppl_oracle as orc
        t_or, fl_or, k = 0.0, 0.0, 0
        while t_or < 15.0 and k < len(shapes):
            B, tau, fac = data[k]
            o = shapes[k][0]
            Bvv = np.ascontiguousarray(B.cpu().numpy()[:, o:, o:])
            t = tau.cpu().numpy()
            t0 = time.perf_counter()
            orc.als_sweep(Bvv, t, fac, np.ones(shapes[k][3]))
            t_or += time.perf_counter() - t0
            fl_or += alg_flops(*shapes[k])
            k += 1
        cores, how = oracle_cores()
        cpu = {"value": (fl_or / flops) / t_or, "unit": "batch sweeps/s", "cores": cores, "kind": "oracle",
               "sample": f"one FP64 oracle sweep of each of the first {k} instances, scaled by flops to all 64; "
                         f"threads from {how}"}
    pk = measure_peaks(dev, torch.cuda.current_stream(dev))
    pk_kind = "measured in this run"
    peak, _ = tensor_peak(pk, args.precision)
    tflops = flops / (ms / args.steps / 1000.0) / 1e12
    value = world * args.steps / (ms / 1000.0)
    line = {
        "metric": METRIC, "value": value, "unit": "batch sweeps/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": args.precision, "data": "synthetic (seeded; shapes of the paper's molecules)",
        "config": {"workload": "cp-als-ppl batch of 64 uneven instances (o 4-24, v 40-240, X = 3v, R 2v-4v), one graph",
                   "instances": 64, "precision": args.precision},
        "sweep_tflops": tflops,
        "roofline": {"bound": "tensor", "achieved": tflops, "peak": peak, "unit": "TFLOP/s", "frac": tflops / peak,
                     "traffic": None, "kernel": "whole batch sweep (MTTKRP flops / sweep time)",
                     "peak_source": f"{pk_kind}"},
        "fp64_gpu": {"ms_per_sweep": f64_ms, "speedup_mixed_vs_fp64": f64_ms / (ms / args.steps)},
        "gpu_launches": int(launches) * args.steps,
        "clocks": {k2: ck[k2] for k2 in ("sm_mhz", "sm_max_mhz", "reasons")},
        "cpu_baseline": cpu,
    }
    batch.close()
    for p in probs:
        p.close()
    if rank == 0:
        print(json.dumps(line), flush=True)


def batch_secondary(dev, precision, steps=3, warmup=3):
    """The 64-instance batch (o in [4,24], v in [40,240], X = 3v, R in [2v,4v]) as a
    secondary field of the main line: batch sweeps/s from CUDA events around
    `steps` graph-replayed batch sweeps, launches per batch sweep and the whole-
    sweep MTTKRP TFLOP/s.  Any failure is reported in the field, never raised."""
    import torch
    from paper_2503_10380_gb300 import binding, inputs
    try:
        shapes = inputs.batch_shapes(64, seed=SEED)
        data = [inputs.make_inputs_torch(*sh, seed=SEED + k, device=dev) for k, sh in enumerate(shapes)]
        flops = sum(alg_flops(*sh) for sh in shapes)
        probs = []
        for (B, tau, fac) in data:
            cp = binding.CpAls(B, tau, fac, precision=precision)
            cp.autotune()
            probs.append(cp)
        batch = binding.Batch(probs, nstreams=8)
        batch.sweep(warmup, want_fits=False)
        stream = torch.cuda.current_stream(dev)
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        batch.sweep(steps, want_fits=False)
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / steps
        out = {"workload": "cp-als-ppl batch of 64 uneven instances (o 4-24, v 40-240, X = 3v, R 2v-4v), one graph",
               "precision": precision, "batch_sweeps_per_s": 1000.0 / ms, "ms_per_batch_sweep": ms,
               "sweep_tflops": flops / (ms / 1000.0) / 1e12, "launches_per_batch_sweep": int(batch.kernels_per_sweep())}
        batch.close()
        for p in probs:
            p.close()
        del data, probs
        torch.cuda.empty_cache()
        return out
    except Exception as exc:   # a secondary field must not take the main line down
        return {"error": f"{type(exc).__name__}: {exc}"}


PREC_CFG, PREC_SWEEPS = (40, 400, 1200, 1600), 20
SEQ_CFG, SEQ_STEPS, SEQ_MAX_SWEEPS, SEQ_EPS = (60, 600, 1800, 2400), 15, 50, 1e-6


def _timed_sweeps(cp, n, stream):
    return _time_sweeps(cp, n, stream)


def run_precision(args, world, rank, local):
    """o=40 v=400 X=1200 R=1600: BF16x3, TF32 and TF32x3 against the plain FP64 GPU form
    from the same start after PREC_SWEEPS sweeps (energy in kcal/mol, relative
    error of every factor), and the sweep rate of each form."""
    import numpy as np
    import torch
    from paper_2503_10380_gb300 import binding, inputs
    import __graft_entry__
    if rank == 0:
        __graft_entry__.build()
    if world > 1:
        torch.distributed.barrier()
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    stream = torch.cuda.current_stream(dev)
    o, v, X, R = PREC_CFG
    B, tau, fac = inputs.make_inputs_torch(o, v, X, R, seed=SEED, device=dev)
    # ||R||^2 and E_exact from the TF32x3 tensor-core exact contraction (relative error ~1e-6)
    cp = binding.CpAls(B, tau, fac, precision="tf32x3")
    normR2, E_exact, _ = cp.exact_contract(mixed=True)
    cp.close()
    del cp
    f64 = binding.CpAls(B, tau, fac, precision="fp64")
    f64.set_normR2(normR2)
    f64.sweep(1, want_hist=False)
    torch.cuda.synchronize()
    f64_ms = _timed_sweeps(f64, PREC_SWEEPS - 1, stream)
    E64, F64, fit64 = f64.energy(), _factors_host(f64), f64.fit()
    f64.close()
    del f64
    torch.cuda.empty_cache()
    variants = {}
    clocks = None
    for prec in ("tf32x3", "bf16x3", "tf32"):
        cp = binding.CpAls(B, tau, fac, precision=prec, profile=True)
        rc_chosen = cp.autotune()
        cp.set_normR2(normR2)
        cp.sweep(PREC_SWEEPS, want_hist=False)
        E, F, fit = cp.energy(), _factors_host(cp), cp.fit()
        cp.sweep(args.warmup, want_hist=False)
        torch.cuda.synchronize()
        ck = ClockSampler(local) if prec == "tf32x3" else None
        ms = _timed_sweeps(cp, args.steps, stream)
        if ck is not None:
            clocks = ck.stop()
        acc = None
        for _ in range(3):
            cp.sweep(1, want_hist=False)
            ph = cp.phase_ms()
            acc = ph if acc is None else {k: acc[k] + ph[k] for k in acc}
        mt_ms = sum(acc[k] for k in ("tau_r", "chain_a", "chain_b", "s_and_p")) / 3
        launches = int(cp.stats()["kernels_per_sweep"])
        cp.close()
        del cp
        variants[prec] = {
            "ms_per_sweep": ms, "sweeps_per_s": 1000.0 / ms,
            "mttkrp_tflops": alg_flops(o, v, X, R) / (mt_ms / 1000.0) / 1e12,
            "speedup_vs_fp64_gpu": f64_ms / ms, "E_cp": E, "fit": fit,
            "dE_kcal_per_mol": abs(E - E64) * KCAL, "dE_rel": abs(E - E64) / abs(E64),
            "factor_rel_err": {m: float(np.linalg.norm(F[m] - F64[m]) / np.linalg.norm(F64[m])) for m in F64},
            "kernels_per_sweep": launches, "r_chunk": rc_chosen,
        }
    ms = reduce_max(variants["tf32x3"]["ms_per_sweep"], world, dev)
    pk = measure_peaks(dev, torch.cuda.current_stream(dev))
    pk_kind = "measured in this run"
    peak, peak_note = tensor_peak(pk, "tf32x3")
    tf = variants["tf32x3"]["mttkrp_tflops"]
    line = {
        "metric": METRIC, "value": world * 1000.0 / ms, "unit": "sweeps/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "tf32x3", "data": "synthetic (seeded; shapes of the paper's molecules)",
        "config": {"workload": f"cp-als-ppl precision study o={o} v={v} X={X} R={R}, {PREC_SWEEPS} sweeps "
                               f"from one start in FP64, BF16x3 and TF32", "o": o, "v": v, "X": X, "R": R,
                   "l2": "inputs larger than L2"},
        "roofline": {"bound": "tensor", "achieved": tf, "peak": peak, "unit": "TFLOP/s", "frac": tf / peak,
                     "traffic": None, "kernel": "all MTTKRP contractions of one sweep (phase events)",
                     "peak_source": f"{pk_kind}: {peak_note}"},
        "fp64_gpu": {"ms_per_sweep": f64_ms, "E_cp": E64, "fit": fit64},
        "variants": variants,
        "E_exact_tf32x3": E_exact, "normR2_tf32x3": normR2,
        "rank_error_kcal_per_mol": abs(E64 - E_exact) * KCAL,
        "gpu_launches": variants["tf32x3"]["kernels_per_sweep"] * args.steps,
        "clocks": {k: clocks[k] for k in ("sm_mhz", "sm_max_mhz", "reasons")} if clocks else None,
        "cpu_baseline": oracle_estimate(o, v, X, R) if rank == 0 and world == 1 and not args.no_cpu_baseline else None,
    }
    if rank == 0:
        print(json.dumps(line), flush=True)


def run_sequence(args, world, rank, local):
    """o=60 v=600 X=1800 R=2400: SEQ_STEPS CC-like steps tau_k = tau_{k-1} + dtau_k,
    each a CPD warm-started from the previous factors on the device and swept
    until |dfit| < SEQ_EPS (at most SEQ_MAX_SWEEPS sweeps); ||R_k||^2 from the
    tensor-core exact contraction at every step."""
    import torch
    from paper_2503_10380_gb300 import binding, inputs
    import __graft_entry__
    if rank == 0:
        __graft_entry__.build()
    if world > 1:
        torch.distributed.barrier()
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    stream = torch.cuda.current_stream(dev)
    o, v, X, R = SEQ_CFG
    B, tau, fac = inputs.make_inputs_torch(o, v, X, R, seed=SEED, device=dev)
    rms0 = float(torch.sqrt(torch.mean(tau * tau)))
    torch.cuda.empty_cache()
    cp = binding.CpAls(B, tau, fac, precision=args.precision, profile=True)
    rc_chosen = cp.autotune()
    clocks = ClockSampler(local)
    steps, t_solve, t_exact, n_sweeps = [], 0.0, 0.0, 0
    for k in range(SEQ_STEPS):
        if k > 0:
            tau += inputs.tau_increment_t(torch, rms0, tuple(tau.shape), k, seed=SEED, device=dev)
            cp.set_tau(tau)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        normR2, E_exact, _ = cp.exact_contract(mixed=True)
        t1 = time.perf_counter()
        sweeps, fits, _ = cp.solve(SEQ_MAX_SWEEPS, "dfit", SEQ_EPS)
        torch.cuda.synchronize()
        t2 = time.perf_counter()
        E = cp.energy()
        t_exact += t1 - t0
        t_solve += t2 - t1
        n_sweeps += sweeps
        steps.append({"k": k, "sweeps": sweeps, "stop": "dfit" if sweeps < SEQ_MAX_SWEEPS else "max_sweeps",
                      "fit": fits[sweeps - 1] if sweeps else None,
                      "dfit_last": abs(fits[sweeps - 1] - fits[sweeps - 2]) if sweeps > 1 else None,
                      "E_cp": E, "E_exact_mixed": E_exact, "solve_s": t2 - t1, "exact_s": t1 - t0})
        if rank == 0:
            print(json.dumps({"progress": steps[-1]}), file=sys.stderr, flush=True)
    ck = clocks.stop()
    acc = None
    for _ in range(3):
        cp.sweep(1, want_hist=False)
        ph = cp.phase_ms()
        acc = ph if acc is None else {kk: acc[kk] + ph[kk] for kk in acc}
    phases = {kk: acc[kk] / 3 for kk in acc}
    mt_ms = phases["tau_r"] + phases["chain_a"] + phases["chain_b"] + phases["s_and_p"]
    ms_sweep = _timed_sweeps(cp, 3, stream)
    launches = int(cp.stats()["kernels_per_sweep"])
    cp.close()
    del cp
    torch.cuda.empty_cache()
    f64 = binding.CpAls(B, tau, fac, precision="fp64")
    f64.sweep(1, want_hist=False)
    torch.cuda.synchronize()
    f64_ms = _timed_sweeps(f64, 1, stream)
    f64.close()
    t_solve = reduce_max(t_solve, world, dev)
    pk = measure_peaks(dev, torch.cuda.current_stream(dev))
    pk_kind = "measured in this run"
    peak, _ = tensor_peak(pk, args.precision)
    tf = alg_flops(o, v, X, R) / (mt_ms / 1000.0) / 1e12
    line = {
        "metric": METRIC, "value": world * n_sweeps / t_solve, "unit": "sweeps/s", "n_gpus": world,
        "steps": SEQ_STEPS, "warmup": 0, "ms_per_step": 1000.0 * t_solve / n_sweeps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": args.precision,
        "data": "synthetic (seeded; shapes of the paper's molecules)",
        "config": {"workload": f"cp-als-ppl warm-started CC-like sequence o={o} v={v} X={X} R={R}, {SEQ_STEPS} steps, "
                               f"|dfit| < {SEQ_EPS} or {SEQ_MAX_SWEEPS} sweeps", "o": o, "v": v, "X": X, "R": R,
                   "l2": "inputs larger than L2 (tau 10.4 GB)"},
        "sweeps_total": n_sweeps, "solve_s": t_solve, "exact_contract_s": t_exact, "r_chunk": rc_chosen,
        "ms_per_sweep_steady": ms_sweep, "phase_ms": phases,
        "roofline": {"bound": "tensor", "achieved": tf, "peak": peak, "unit": "TFLOP/s", "frac": tf / peak,
                     "traffic": None, "kernel": "all MTTKRP contractions of one sweep (phase events)",
                     "peak_source": f"{pk_kind}"},
        "fp64_gpu": {"ms_per_sweep": f64_ms, "speedup_mixed_vs_fp64": f64_ms / ms_sweep},
        "per_step": steps,
        "gpu_launches": launches * n_sweeps,
        "clocks": {kk: ck[kk] for kk in ("sm_mhz", "sm_max_mhz", "reasons")},
        "cpu_baseline": oracle_estimate(o, v, X, R) if rank == 0 and world == 1 and not args.no_cpu_baseline else None,
    }
    if rank == 0:
        print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--precision", choices=["bf16x3", "tf32", "tf32x3"], default=None,
                    help="tensor-core precision of the MTTKRP (default: tf32x3, the split that meets the "
                         "0.1 kcal/mol bar; bf16x3 for --workload batch)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-secondary", action="store_true", help="skip the o=20 and o=40 configurations of the line")
    ap.add_argument("--config", default="", help="o,v,X,R of the single-instance workload (default 60,600,1800,2400)")
    ap.add_argument("--r-chunk", type=int, default=0, help="rank columns per pass of the MTTKRP chain (0 = auto)")
    ap.add_argument("--workload", choices=["single", "batch", "precision", "sequence"], default="single",
                    help="single: o=20 v=200 X=600 R=800 (default); batch: 64 uneven instances; "
                         "precision: o=40 v=400 X=1200 R=1600 in FP64, BF16x3 and TF32; "
                         "sequence: o=60 v=600 X=1800 R=2400, 15 warm-started CC-like steps")
    args = ap.parse_args()
    if args.config:
        set_main_cfg(int(x) for x in args.config.split(","))
    if args.precision is None:
        args.precision = "bf16x3" if args.workload == "batch" else "tf32x3"
    if args.warmup < 3:
        args.warmup = 3
    world, rank, local = dist_setup()
    if world > 1:
        import torch
        backend = "nccl" if torch.cuda.is_available() else "gloo"
        torch.distributed.init_process_group(backend=backend)
    try:
        if args.impl == "reference":
            run_reference(args, world, rank)
        elif args.workload == "batch":
            run_batch(args, world, rank, local)
        elif args.workload == "precision":
            run_precision(args, world, rank, local)
        elif args.workload == "sequence":
            run_sequence(args, world, rank, local)
        else:
            run_ours(args, world, rank, local)
    finally:
        if world > 1:
            import torch
            torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()

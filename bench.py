#!/usr/bin/env python3
"""Benchmark of the matrix-free monolithic multigrid Stokes solver on one GB300 (or N replicas).

Workload (one "step"): three solves of the 3D generalized Stokes system, Q2-Q1 Taylor-Hood on
32^3 hexahedra of the unit cube whose vertices are moved by a smooth seeded field of amplitude
0.1 h (trilinear cells), 5 levels, mu = rho = 1, gamma in {0, 1e2, 1e4}; right-hand side
b = M_v f with a 4-mode Fourier forcing (seed 0); FP64 flexible GMRES(30) right-preconditioned
by one FP32 V-cycle (Chebyshev degrees k_A = k_S = 1, m = 2, Schur diagonal d) to ||b - K x|| <= 1e-8 ||b||,
from x = 0.  Setup (hierarchy, diagonals, Lanczos, coarse inverse) is outside the timed region.

Metric: MDoF/s solved (DoFs per second of time-to-1e-8; the inverse of solve time per MDoF),
with FP64-MG, vmult throughput, roofline of the dominant kernel, end-to-end throughput through
the host-buffer C call, and the CPU oracle baseline reported beside it.

    python bench.py [--steps K] [--warmup W] [--gpus N] [--impl ours|reference]
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "MDoF/s Stokes vmult; solve time/MDoF to 1e-8 residual, FP32-MG vs FP64-MG"
# Smoother: the paper's 3D recommendation, two smoothing steps of the (1, 1) Chebyshev smoother
# (k_A, k_S, m) = (1, 1, 2) with the Schur-complement diagonal D~_S~d = diag(B diag(A)^-1 B^T), the
# diagonal its rate studies use (Sec. 4.3-4.5: highest residual reduction per second in 3D; diag d
# as good as the exact diagonal).  `--smoother-sweep` repeats that study on GB300 in time-to-1e-8.
WL = dict(dim=3, k=2, n=(32, 32, 32), levels=5, amplitude=0.1, seed=0, gammas=(0.0, 1e2, 1e4), rtol=1e-8,
          kA=1, kS=1, m=2, schur_diag="d", restart=30)
WORKLOAD_NAME = ("3D generalized Stokes Q2-Q1, unit cube 32^3 hexes, smooth trilinear vertex perturbation "
                 "0.1h (seed 0), 5 levels, mu=rho=1, gamma in {0,1e2,1e4}, FGMRES(30)+FP32 V-cycle "
                 "(Chebyshev kA=1, kS=1, m=2, Schur diagonal d), rtol 1e-8")
SWEEP = [(3, 3, 2), (1, 1, 2), (2, 1, 2), (1, 2, 2), (2, 2, 1), (1, 1, 1), (3, 2, 1), (2, 2, 2), (0, 0, 4),
         (1, 0, 2), (0, 1, 2)]
L2_FLUSH_BYTES = 256 << 20
FALLBACK_HBM_GBS = 6800.0


def max_over_ranks(x, world, device="cpu"):
    """The largest x over the ranks of the default process group (the slowest replica sets the
    step time); x itself when there is one rank."""
    if world <= 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_throughput(ms_per_step, world, solves, n_dofs):
    """Whole-job MDoF/s: every rank solves the same `solves` systems of `n_dofs` DoFs per step
    (independent replicas, weak scaling), the step lasting ms_per_step on the slowest rank."""
    return world * solves * n_dofs / (ms_per_step / 1e3) / 1e6


def dofs(n, k=2, dim=3):
    nu = dim
    npr = 1
    for a in range(dim):
        nu *= k * n[a] + 1
        npr *= (k - 1) * n[a] + 1
    return nu + npr


def tuning_string(S):
    """The setup's choices of a context as a STOKES_TUNING value (to profile the same configuration:
    timings taken under a profiler choose differently)."""
    j = lambda v: ",".join(str(int(x)) for x in v)
    return (f"s32={j(S.launch_shapes(32))};s64={j(S.launch_shapes(64))};f32={j(S.fused_levels(32))};"
            f"f64={j(S.fused_levels(64))};g32={j(S.geometry_stored(32))};p32={j(S.plane_levels(32))}")


# ---------------------------------------------------------------------------------------------
def perturbed_vertices():
    import workloads as W
    return W.perturbed_vertices(WL["dim"], WL["n"], seed=WL["seed"], amplitude=WL["amplitude"])


def forcing():
    import workloads as W
    return W.fourier_forcing(WL["dim"], WL["k"], WL["n"], seed=WL["seed"]).reshape(-1)


ORACLE_GAMMA = 1e2  # the middle gamma of the workload: the CPU sample solves this one


def oracle_sample(steps=1, warmup=0):
    """CPU oracle on the workload itself: the 32^3 perturbed hierarchy (859,812 DoFs, 5 levels),
    gamma = 1e2, the same smoother and Schur diagonal, FP64 multigrid + FGMRES(30) to 1e-8 from
    x = 0.  Setup (assembly, Lanczos, Schur diagonal, coarse LU) is untimed; each step is one
    solve.  Returns seconds per step."""
    from oracle.assemble import load_vector_nodal
    from oracle.krylov import fgmres
    from oracle.mesh import Hierarchy
    from oracle.mg import Multigrid
    t0 = time.perf_counter()
    H = Hierarchy(3, 2, WL["n"], WL["levels"], perturbed_vertices())
    lev = H.levels[-1]
    mg = Multigrid(H, gamma_rho=ORACLE_GAMMA, kA=WL["kA"], kS=WL["kS"], m=WL["m"], schur_diag=WL["schur_diag"])
    b = load_vector_nodal(lev, mg.ops[-1], forcing())
    setup_s = time.perf_counter() - t0
    times, iters = [], None
    for s in range(warmup + steps):
        t0 = time.perf_counter()
        _, it, _ = fgmres(lambda v: mg.K @ v, mg.precondition, b, rtol=WL["rtol"], restart=WL["restart"])
        dt = time.perf_counter() - t0
        if s >= warmup:
            times.append(dt)
            iters = it
    return {"seconds_per_step": sum(times) / len(times), "dofs": lev.size, "solves_per_step": 1,
            "iterations": iters, "steps": steps, "setup_s": round(setup_s, 2)}


def host_cpu_info():
    """Logical CPUs of this host and its CPU model (from /proc/cpuinfo where present)."""
    model = None
    try:
        with open("/proc/cpuinfo") as fh:
            for line in fh:
                key = line.split(":")[0].strip().lower()
                if key in ("model name", "cpu model", "hardware") and ":" in line:
                    model = line.split(":", 1)[1].strip()
                    break
                if key == "cpu part" and model is None:
                    model = "cpu part " + line.split(":", 1)[1].strip()
    except OSError:
        pass
    import platform
    return {"nproc": os.cpu_count(), "model": model, "machine": platform.machine()}


def _oracle_env(threads):
    t = str(threads)
    return dict(os.environ, OMP_NUM_THREADS=t, OPENBLAS_NUM_THREADS=t, MKL_NUM_THREADS=t)


def run_oracle_subprocess(steps=1, warmup=0, threads=1):
    r = subprocess.run([sys.executable, os.path.abspath(__file__), "--_oracle-sample", str(steps), str(warmup)],
                       capture_output=True, text=True, env=_oracle_env(threads), timeout=3600)
    if r.returncode != 0:
        raise RuntimeError("oracle sample failed:\n" + r.stderr[-2000:])
    return json.loads(r.stdout.strip().splitlines()[-1])


def cpu_table_rows():
    """The CPU-baseline plan's measurements of the oracle (one process, the thread count set by the
    caller's environment): CSR SpMV MDoF/s on the 2D 16^2 cavity mesh, the 32^3 workload mesh and
    the channel [0,4]x[0,1]^2 (Q2, 32^3 cells: the per-DoF rate of the 64^3 channel, whose CSR
    assembly would take minutes), and time-to-solution of the 2D 16^2 problem (FGMRES + one V(3,3)
    cycle, rtol 1e-10) and of the 32^3 workload for each gamma (rtol 1e-8)."""
    import numpy as np
    from oracle.assemble import assemble, load_vector_nodal
    from oracle.krylov import fgmres
    from oracle.mesh import Hierarchy, Level
    from oracle.mg import Multigrid
    import workloads as W
    rows = []

    def spmv_rate(K, reps):
        x = np.random.default_rng(0).uniform(-1, 1, K.shape[0])
        K @ x
        t0 = time.perf_counter()
        for _ in range(reps):
            K @ x
        dt = (time.perf_counter() - t0) / reps
        return K.shape[0] / dt / 1e6

    lev2 = Level(2, 2, (16, 16), W.lattice_vertices(2, (16, 16)))
    rows.append({"row": "spmv", "config": "2D Q2-Q1 16^2", "dofs": lev2.size,
                 "mdof_s": spmv_rate(assemble(lev2)["K"], 2000)})
    lev3 = Level(3, 2, WL["n"], perturbed_vertices())
    rows.append({"row": "spmv", "config": "3D Q2-Q1 32^3 perturbed", "dofs": lev3.size,
                 "mdof_s": spmv_rate(assemble(lev3, 1.0, 1e2)["K"], 20)})
    levc = Level(3, 2, (32, 32, 32), W.lattice_vertices(3, (32, 32, 32), hi=(4.0, 1.0, 1.0)), 0x3F & ~0x2)
    rows.append({"row": "spmv", "config": "3D Q2-Q1 channel 32^3 cells", "dofs": levc.size,
                 "mdof_s": spmv_rate(assemble(levc, 1e-3)["K"], 20)})
    # 2D 16^2, FGMRES + V(3,3) to 1e-10 (manufactured forcing of the 2D case)
    H2 = Hierarchy(2, 2, (16, 16), 4, W.lattice_vertices(2, (16, 16)))
    mg2 = Multigrid(H2, kA=3, kS=3, m=2)
    l2 = H2.levels[-1]
    ax = W.velocity_lattice(2, 2, (16, 16))
    Y, X = np.meshgrid(ax[1], ax[0], indexing="ij")
    f1, f2 = W.mms2d_forcing(X, Y)
    b2 = load_vector_nodal(l2, mg2.ops[-1], np.stack([f1, f2]).reshape(-1))
    t0 = time.perf_counter()
    reps = 20
    for _ in range(reps):
        _, it2, _ = fgmres(lambda v: mg2.K @ v, mg2.precondition, b2, rtol=1e-10)
    rows.append({"row": "solve", "config": "2D Q2-Q1 16^2, FGMRES + V(3,3), rtol 1e-10", "dofs": l2.size,
                 "seconds": (time.perf_counter() - t0) / reps, "iterations": it2})
    H3 = Hierarchy(3, 2, WL["n"], WL["levels"], perturbed_vertices())
    l3 = H3.levels[-1]
    for g in WL["gammas"]:
        mg3 = Multigrid(H3, gamma_rho=g, kA=WL["kA"], kS=WL["kS"], m=WL["m"], schur_diag=WL["schur_diag"])
        b3 = load_vector_nodal(l3, mg3.ops[-1], forcing())
        t0 = time.perf_counter()
        _, it3, _ = fgmres(lambda v: mg3.K @ v, mg3.precondition, b3, rtol=WL["rtol"], restart=WL["restart"])
        rows.append({"row": "solve", "config": f"3D Q2-Q1 32^3 perturbed, gamma {g:g}, FP64-MG FGMRES, rtol 1e-8",
                     "dofs": l3.size, "seconds": time.perf_counter() - t0, "iterations": it3})
    return rows


def run_cpu_table(args):
    """The oracle's CPU-baseline table on this host, with 1 thread and with every logical CPU."""
    info = host_cpu_info()
    print(json.dumps({"host": info}), flush=True)
    for threads in (1, info["nproc"] or 1):
        r = subprocess.run([sys.executable, os.path.abspath(__file__), "--_cpu-table-rows"], capture_output=True,
                           text=True, env=_oracle_env(threads), timeout=3600)
        if r.returncode != 0:
            print(json.dumps({"threads": threads, "error": r.stderr[-1500:]}), flush=True)
            continue
        for row in json.loads(r.stdout.strip().splitlines()[-1]):
            row["threads"] = threads
            print(json.dumps(row), flush=True)


# ---------------------------------------------------------------------------------------------
class ClockSampler:
    """nvidia-smi clock / throttle sampling every 200 ms.  Started before the warm-up steps (so the
    sampler's own start-up is not inside the timed region); mark() and stop() bracket the timed
    region, and only the samples stamped inside it (widened by one period) are reported."""

    def __init__(self, gpu_index):
        import datetime
        self._dt = datetime
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        self.t0 = self.t1 = None
        q = ("timestamp,index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.f = open(self.path, "w")
            self.p = subprocess.Popen(["nvidia-smi", f"--query-gpu={q}", "--format=csv,noheader,nounits",
                                       "-lms", "200", "-i", str(gpu_index)], stdout=self.f,
                                      stderr=subprocess.DEVNULL)
        except Exception:
            self.p = None

    def mark(self):
        self.t0 = self._dt.datetime.now()

    def stop(self):
        self.t1 = self._dt.datetime.now()
        if self.p is None:
            try:
                self.f.close()
                os.unlink(self.path)
            except Exception:
                pass
            return None
        time.sleep(0.25)  # let the sample that covers the end of the region land
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except Exception:
            self.p.kill()
        self.f.close()
        with open(self.path) as fh:
            out = parse_clock_samples(fh.read().splitlines(), self.t0 or self.t1, self.t1)
        os.unlink(self.path)
        return out


def parse_clock_samples(lines, t0, t1):
    """Clock summary of the nvidia-smi CSV lines (timestamp, index, clocks.sm, clocks.max.sm,
    power.draw, reasons.active, hw_slowdown, hw_thermal_slowdown, sw_thermal_slowdown,
    sw_power_cap) stamped within [t0 - 0.2 s, t1 + 0.2 s] (the last two samples when none is):
    median SM clock, max clock, the throttle reasons seen active, the number of samples."""
    import datetime
    names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
    lo = t0 - datetime.timedelta(seconds=0.2)
    hi = t1 + datetime.timedelta(seconds=0.2)
    rows = []
    for line in lines:
        parts = [p.strip() for p in line.split(",")]
        if len(parts) < 10:
            continue
        try:
            ts = datetime.datetime.strptime(parts[0], "%Y/%m/%d %H:%M:%S.%f")
            rows.append((ts, float(parts[2]), float(parts[3]), parts[6:10]))
        except ValueError:
            continue
    inside = [r for r in rows if lo <= r[0] <= hi] or rows[-2:]
    sm, mx, reasons = [], [], set()
    for _, a, b, flags in inside:
        sm.append(a)
        mx.append(b)
        for nm, v in zip(names, flags):
            if v.lower() == "active":
                reasons.add(nm)
    if not sm:
        return None
    return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
            "samples": len(sm)}


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        try:
            return json.load(open(p)), "measured"
        except Exception:
            pass
    return None, "fallback"


def traffic_record(key, kernel_src_sha):
    """DRAM bytes per launch of the kernel `key` ("fp32_a_block", "fp64_operator") from the
    committed ncu summary, or None when the kernel source changed since the counters were taken."""
    p = os.path.join(ROOT, "profiles", "roofline_traffic.json")
    if not os.path.exists(p):
        return None
    try:
        rec = json.load(open(p)).get(key, {})
    except Exception:
        return None
    if rec.get("kernel_source_sha256") != kernel_src_sha:
        return None
    return rec.get("dram_bytes_per_launch_full_size")


def kernel_source_sha():
    h = hashlib.sha256()
    for f in ("apply.cuh", "apply_col.cuh", "apply_cc.cuh", "apply_fx.cuh", "apply_pl.cuh", "common.cuh"):
        h.update(open(os.path.join(ROOT, "paper_2205_15770_gb300", "csrc", f), "rb").read())
    return h.hexdigest()


# Flops per cell of the full operator K x by sum factorisation and algorithmic bytes per DoF, the
# scope table's measurement model (FMA = 2 flops; forward + backward 24 (k+1)^4 per scalar field,
# the pressure sweeps and point terms; trilinear cells add the geometry from the 8 vertices).
FLOPS_PER_CELL_8D = {("trilinear", 2): 12768, ("affine", 2): 6963, ("affine", 3): 21808, ("affine", 4): 53005}
BYTES_PER_DOF_8D = {(32, "trilinear"): 8.5, (32, "affine"): 8.0, (64, "trilinear"): 17.0, (64, "affine"): 16.0}
NOMINAL_BF16_DENSE_TFLOPS = 2250.0  # GB300 dense bf16 tensor rate (nominal)
LANES_PER_SM = {32: 128, 64: 2}     # FP32 / FP64 FMA lanes per SM (FP64 = 1/64 of FP32)
# The fixed-point full operator on a trilinear Q2 cell: multiply-adds of a (component, z plane) thread, counted from its
# products (three each) and sums (one each), times nine threads; and what an SM issues of them, by a probe kernel of
# independent chains.
INT_MADS_PER_CELL = 9 * 1164
INT_MADS_PER_SM_CLOCK = 50
KERNEL_NAMES = {
    "fp32_operator": "full operator K x, FP32, finest level (V-cycle residual and vmult)",
    "fp64_operator": "full operator K x, FP64, finest level (FGMRES operator; stored coefficients)",
    "fp32_a_block": "A block, FP32, finest level (the V-cycle's most frequent application)",
}


def alu_peak_tflops(prec, sm_count, mhz):
    """FMA peak from the unit counts and the clock: SMs x lanes x 2 flops x clock."""
    return sm_count * LANES_PER_SM[prec] * 2 * mhz * 1e6 / 1e12


def roofline_entry(key, prec, blocks, avg_ms, n_cells, n_dofs, sm_count, mhz, fma_tflops, peaks, sha, shape):
    geom = "trilinear"
    e = {"kernel": KERNEL_NAMES[key], "launch_shape": shape, "avg_launch_us": round(avg_ms * 1e3, 2)}
    peak = alu_peak_tflops(prec, sm_count, mhz)
    bf16 = (peaks or {}).get("bf16_tflops")
    nominal = alu_peak_tflops(prec, 152, 2070.0)
    if blocks == 7:
        fl = FLOPS_PER_CELL_8D[(geom, WL["k"])] * n_cells
        by = BYTES_PER_DOF_8D[(prec, geom)] * n_dofs
        ach = fl / (avg_ms / 1e3) / 1e12
        e.update({"bound": "alu", "achieved": round(ach, 4), "peak": round(peak, 4), "unit": "TFLOP/s",
                  "frac": round(ach / peak, 4), "flops_per_launch": fl, "algorithmic_bytes_per_launch": by,
                  "peak_source": f"derived: {sm_count} SMs x {LANES_PER_SM[prec]} FP{prec} lanes x 2 x {mhz:.0f} MHz",
                  "frac_of_measured_fma": round(ach / fma_tflops, 4),
                  "measured_fma_tflops": round(fma_tflops, 3)})
        if prec == 64 and shape == 5:
            # computed in 64-bit fixed point: the rate that could bound it is the integer multiply-adds'; the sum-factorised
            # flops against the FP64 unit, which it does not use, are kept for comparison
            e["fp64_unit_comparison"] = {q: e.pop(q) for q in ("achieved", "peak", "unit", "frac", "peak_source",
                                                               "frac_of_measured_fma", "measured_fma_tflops")}
            mads, ipk = INT_MADS_PER_CELL * n_cells, sm_count * INT_MADS_PER_SM_CLOCK * mhz * 1e6 / 1e12
            ach = mads / (avg_ms / 1e3) / 1e12
            e.update({"bound": "integer multiply-add", "achieved": round(ach, 4), "peak": round(ipk, 4),
                      "unit": "T multiply-adds/s (32 x 32 + 64 bit)", "frac": round(ach / ipk, 4),
                      "int_mads_per_launch": mads,
                      "peak_source": f"measured by a probe: {sm_count} SMs x {INT_MADS_PER_SM_CLOCK} per clock x {mhz:.0f} MHz"})
            bf16 = None
        if bf16:
            dv = bf16 * nominal / NOMINAL_BF16_DENSE_TFLOPS
            e["peak_from_measured_bf16"] = round(dv, 4)
            e["frac_of_peak_from_measured_bf16"] = round(ach / dv, 4)
        hbm = (peaks or {}).get("hbm_gbs", FALLBACK_HBM_GBS)
        e["hbm_frac_algorithmic"] = round(by / (avg_ms / 1e3) / 1e9 / hbm, 4)
    tr = traffic_record(key, sha)
    e["traffic"] = tr
    if tr and blocks == 7:
        e["traffic_over_algorithmic_bytes"] = round(tr / e["algorithmic_bytes_per_launch"], 2)
    share = launch_share(key)
    if share is not None:
        e["launch_list_share"] = share
    return e


def roofline_object(rl, peaks, peaks_src):
    """The kernel with the largest share of the committed launch list leads; the others follow."""
    order = sorted(rl, key=lambda k: -(rl[k].get("launch_list_share") or 0.0))
    lead = next(k for k in order if "frac" in rl[k])
    out = dict(rl[lead])
    out["key"] = lead
    out["others"] = {k: rl[k] for k in order if k != lead}
    out["hbm_peak_gbs"] = (peaks or {}).get("hbm_gbs", FALLBACK_HBM_GBS)
    out["hbm_peak_source"] = peaks_src
    return out


def launch_share(key):
    p = os.path.join(ROOT, "profiles", "roofline_traffic.json")
    try:
        return json.load(open(p)).get(key, {}).get("launch_share")
    except Exception:
        return None


# ---------------------------------------------------------------------------------------------
def run_ours(args):
    import numpy as np
    import torch
    import torch.distributed as dist
    from paper_2205_15770_gb300 import StokesMG

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl")

    def barrier():
        if world > 1:
            dist.barrier(device_ids=[local])

    V = perturbed_vertices()
    N = dofs(WL["n"])
    f = torch.as_tensor(forcing(), device="cuda")
    common = dict(dim=3, n=WL["n"], n_levels=WL["levels"], k=WL["k"], vertices=V, kA=WL["kA"], kS=WL["kS"],
                  schur_diag=WL["schur_diag"],
                  m=WL["m"], restart=WL["restart"])
    t0 = time.perf_counter()
    S32 = [StokesMG(gamma_rho=g, vcycle_fp32=True, **common) for g in WL["gammas"]]
    setup_s = (time.perf_counter() - t0) / len(S32)
    S64 = [StokesMG(gamma_rho=g, vcycle_fp32=False, **common) for g in WL["gammas"]]
    B = [S.mass_rhs(f) for S in S32]
    X = [torch.zeros(N, dtype=torch.float64, device="cuda") for _ in S32]
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")

    def step(solvers, xs):
        its = []
        for S, b, x in zip(solvers, B, xs):
            x.zero_()
            _, it, rel = S.solve(b, x, rtol=WL["rtol"])
            its.append(it)
        return its

    clocks = ClockSampler(local)
    for _ in range(args.warmup):
        step(S32, X)
    torch.cuda.synchronize()
    barrier()
    torch.cuda.synchronize()
    clocks.mark()
    if args.profile_range:
        torch.cuda.profiler.start()
    l0 = sum(S.launch_count for S in S32)
    total_ms = 0.0
    step_ms = []
    iters = None
    for _ in range(args.steps):
        flush.zero_()  # L2 flush (256 MB write) between timed steps, outside the events
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        iters = step(S32, X)
        e1.record()
        e1.synchronize()
        step_ms.append(e0.elapsed_time(e1))
        total_ms += step_ms[-1]
    torch.cuda.synchronize()
    launches = sum(S.launch_count for S in S32) - l0
    if args.profile_range:
        torch.cuda.profiler.stop()
    clk = clocks.stop()
    barrier()
    t_max = max_over_ranks(total_ms, world, device="cuda")
    ms_per_step = t_max / args.steps
    solves = len(WL["gammas"])
    value = replica_throughput(ms_per_step, world, solves, N)

    # --- final residuals of the timed solves (FP64 operator on the GPU) ------------------------
    rels = []
    for S, b, x in zip(S32, B, X):
        r = b - S.vmult(x)
        rels.append(float(torch.linalg.norm(r) / torch.linalg.norm(b)))

    # --- FP64-MG comparison (same solves, FP64 V-cycle) -----------------------------------------
    X64 = [torch.zeros_like(x) for x in X]
    step(S64, X64)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    flush.zero_()
    e0.record()
    it64 = step(S64, X64)
    e1.record()
    e1.synchronize()
    ms64 = e0.elapsed_time(e1)
    diff = max(float(torch.linalg.norm(a - c) / torch.linalg.norm(c)) for a, c in zip(X, X64))

    # --- vmult throughput ----------------------------------------------------------------------
    vm = {}
    for prec, dt in ((32, torch.float32), (64, torch.float64)):
        xv = torch.randn(N, dtype=dt, device="cuda")
        yv = torch.empty_like(xv)
        S = S32[1]
        for _ in range(3):
            S.vmult(xv, yv)
        reps = 50 if prec == 32 else 10
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            S.vmult(xv, yv)
        e1.record()
        e1.synchronize()
        vm[f"fp{prec}"] = N / (e0.elapsed_time(e1) / reps / 1e3) / 1e6

    # --- rooflines on the finest level, in the terms of the scope table's measurement row:
    # flops per cell of the full operator K x (sum factorisation, FMA = 2 flops; trilinear Q2:
    # 12,768) and algorithmic bytes per DoF (x read + y written: FP32 8.5, FP64 17 with the
    # vertices); ALU peaks from the unit counts and the clock, beside the FP32 / FP64 rates derived
    # from the measured bf16 peak by the nominal ratio and the library's FMA probe --------------
    S = S32[1]
    n_cells = WL["n"][0] * WL["n"][1] * WL["n"][2]
    props = torch.cuda.get_device_properties(local)
    max_mhz = clk["sm_max_mhz"] if clk else 2070.0
    from paper_2205_15770_gb300 import fma_peak
    fma = {32: fma_peak(32), 64: fma_peak(64)}
    peaks, peaks_src = measured_peaks()
    sha = kernel_source_sha()
    rl = {}
    for key, prec, blocks, reps in (("fp32_operator", 32, 7, 200), ("fp64_operator", 64, 7, 20),
                                    ("fp32_a_block", 32, 1, 200)):
        S.time_apply(blocks, precision=prec, reps=max(3, reps // 10))
        avg = S.time_apply(blocks, precision=prec, reps=reps)
        rl[key] = roofline_entry(key, prec, blocks, avg, n_cells, N, props.multi_processor_count, max_mhz, fma[prec],
                                 peaks, sha, S.launch_shapes(prec)[-1])

    # --- deterministic mode: colour-class cooperative cell kernels, plain read-modify-write scatter
    deterministic = run_deterministic(S32[1], B[1], common) if not args.no_extras else None

    # --- batched multi-mesh solves (16 unit-cube meshes of uneven size, seeded) -----------------
    batched = run_batched(args) if not args.no_extras else None
    # --- adjoint (32^3 Cartesian, mu = exp(g)): forward + adjoint solve + viscosity gradient ----
    adjoint = run_adjoint() if not args.no_extras else None

    # --- end to end through the host-buffer C call ----------------------------------------------
    bh = [torch.empty(N, dtype=torch.float64).pin_memory() for _ in S32]
    xh = [torch.empty(N, dtype=torch.float64).pin_memory() for _ in S32]
    for t, b in zip(bh, B):
        t.copy_(b.cpu())
    bn = [t.numpy() for t in bh]
    xn = [t.numpy() for t in xh]
    for S, b, x in zip(S32, bn, xn):
        S.solve_host(b, rtol=WL["rtol"], out=x)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        for S, b, x in zip(S32, bn, xn):
            S.solve_host(b, rtol=WL["rtol"], out=x)
    e2e_s = max_over_ranks((time.perf_counter() - t0) / args.steps, world, device="cuda")
    e2e_val = replica_throughput(e2e_s * 1e3, world, solves, N)

    out = {
        "metric": METRIC, "value": round(value, 3), "unit": "MDoF/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(ms_per_step, 3), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
        "config": {"workload": WORKLOAD_NAME, "dofs_per_solve": N, "solves_per_step": solves,
                   "parallelism": f"replicas{world}" if world > 1 else "single",
                   "l2": "flushed by a 256 MB write before every timed step"},
        "step_ms": [round(t, 3) for t in step_ms],
        "iterations_fp32_mg": iters, "final_rel_residual": rels,
        "solve_ms": {"fp32_mg_per_solve": round(ms_per_step / solves, 3), "fp64_mg_per_solve": round(ms64 / solves, 3)},
        "solve_s_per_mdof": {"fp32_mg": ms_per_step / solves / 1e3 / (N / 1e6),
                             "fp64_mg": ms64 / solves / 1e3 / (N / 1e6)},
        "iterations_fp64_mg": it64, "fp32_vs_fp64_mg_solution_rel_diff": diff,
        "vmult_mdof_s": {k2: round(v, 1) for k2, v in vm.items()},
        "setup_s_per_context": round(setup_s, 3),
        "roofline": roofline_object(rl, peaks, peaks_src),
        "e2e": {"value": round(e2e_val, 3), "unit": "MDoF/s", "h2d_bytes_per_step": solves * N * 8,
                "d2h_bytes_per_step": solves * N * 8},
        "gpu_launches": int(launches),
        "clocks": clk,
        "launch_shapes_fp32": S32[0].launch_shapes(32),
        "fp64_geometry_stored": S32[0].geometry_stored(64),
        "fp32_geometry_stored": S32[0].geometry_stored(32),
        "fused_smoothing_levels": {"fp32": S32[0].fused_levels(32), "fp64": S32[0].fused_levels(64)},
        "tuning": tuning_string(S32[0]),
        "batched": batched,
        "adjoint": adjoint,
        "deterministic": deterministic,
    }
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        try:
            o = run_oracle_subprocess(1, 0, threads=1)
            out["cpu_baseline"] = {"value": round(o["dofs"] / o["seconds_per_step"] / 1e6, 4),
                                   "unit": "MDoF/s", "cores": 1, "kind": "oracle",
                                   "sample": ("one FP64-MG FGMRES(30) solve to 1e-8 of the same 32^3 workload "
                                              f"(859,812 DoFs, 5 levels) at gamma {ORACLE_GAMMA:g}, same smoother "
                                              "and Schur diagonal, numpy/scipy, 1 thread; setup untimed"),
                                   "iterations": o["iterations"], "same_config": True, "host": host_cpu_info()}
        except Exception as e:  # report, do not hide
            out["cpu_baseline"] = {"value": None, "error": str(e)[-300:]}
    if rank == 0:
        print(json.dumps(out))
    for S in S32 + S64:
        S.close()
    if world > 1:
        dist.destroy_process_group()


def run_deterministic(S_atomic, b, common):
    """The workload's gamma = 1e2 solve and vmults in deterministic mode (owner-computes; the colour-class
    form beside it) against the default (atomic) context: time per FP32-MG solve, FP32 / FP64 vmult, and
    whether two solves repeat bitwise."""
    import torch
    from paper_2205_15770_gb300 import StokesMG
    kw = dict(common)
    S = StokesMG(gamma_rho=1e2, vcycle_fp32=True, deterministic=1, **kw)

    def t_solve(Sx, reps=3):
        x = torch.zeros_like(b)
        Sx.solve(b, x, rtol=WL["rtol"])
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            x.zero_()
            _, it, _ = Sx.solve(b, x, rtol=WL["rtol"])
        e1.record()
        e1.synchronize()
        return e0.elapsed_time(e1) / reps, it, x.clone()

    def t_vmult(Sx, dt, reps):
        xv = torch.randn(b.numel(), dtype=dt, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
        yv = torch.empty_like(xv)
        Sx.vmult(xv, yv)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            Sx.vmult(xv, yv)
        e1.record()
        e1.synchronize()
        return e0.elapsed_time(e1) / reps * 1e3

    ms_det, it_det, x1 = t_solve(S)
    _, _, x2 = t_solve(S, reps=1)
    ms_atomic, it_atomic, _ = t_solve(S_atomic)
    out = {"solve_ms": round(ms_det, 3), "iterations": it_det, "atomic_solve_ms": round(ms_atomic, 3),
           "atomic_iterations": it_atomic, "solves_repeat_bitwise": bool(torch.equal(x1, x2))}
    for prec, dt, reps in ((32, torch.float32, 50), (64, torch.float64, 10)):
        out[f"vmult_fp{prec}_us"] = round(t_vmult(S, dt, reps), 2)
        out[f"atomic_vmult_fp{prec}_us"] = round(t_vmult(S_atomic, dt, reps), 2)
    S.close()
    S2 = StokesMG(gamma_rho=1e2, vcycle_fp32=True, deterministic=2, **kw)
    ms_col, it_col, _ = t_solve(S2, reps=1)
    out["colour_classes"] = {"solve_ms": round(ms_col, 3), "iterations": it_col,
                             "vmult_fp32_us": round(t_vmult(S2, torch.float32, 20), 2)}
    S2.close()
    return out


def run_batched(args):
    """16 independent Q2-Q1 solves on unit-cube meshes of 8^3..40^3 cells (seeded sizes, gamma in
    {0, 1e3}, 4-mode Fourier forcing): one batched solve (one graph launch per FGMRES iteration
    for all members) against the same members solved one after another."""
    import torch
    import workloads as W
    from paper_2205_15770_gb300 import StokesBatch
    recipe = W.batch_meshes(16, seed=0)
    members = [dict(dim=3, n=(r["n"],) * 3, n_levels=r["levels"], gamma_rho=r["gamma"]) for r in recipe]
    Bt = StokesBatch(members, kA=WL["kA"], kS=WL["kS"], m=WL["m"], schur_diag=WL["schur_diag"], restart=WL["restart"])
    bs = []
    for r, mv in zip(recipe, Bt.members):
        f = torch.as_tensor(W.fourier_forcing(3, 2, (r["n"],) * 3, seed=r["forcing_seed"]).reshape(-1), device="cuda")
        bs.append(mv.mass_rhs(f))
    xs = [torch.zeros_like(b) for b in bs]
    dofs_total = sum(int(b.numel()) for b in bs)
    for _ in range(2):
        for x in xs:
            x.zero_()
        Bt.solve(bs, xs, rtol=WL["rtol"])
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    reps = 3
    e0.record()
    for _ in range(reps):
        for x in xs:
            x.zero_()
        _, its, rels = Bt.solve(bs, xs, rtol=WL["rtol"])
    e1.record()
    e1.synchronize()
    batch_ms = e0.elapsed_time(e1) / reps
    e0.record()
    for _ in range(reps):
        for mv, b, x in zip(Bt.members, bs, xs):
            x.zero_()
            mv.solve(b, x, rtol=WL["rtol"])
    e1.record()
    e1.synchronize()
    seq_ms = e0.elapsed_time(e1) / reps
    Bt.close()
    # the same batch in the persistent work-queue form (one kernel runs every member's FP32 cycle
    # of an iteration, krylov_mode 2)
    prev = os.environ.get("STOKES_BATCH_QUEUE")
    os.environ["STOKES_BATCH_QUEUE"] = "1"
    try:
        Bq = StokesBatch(members, kA=WL["kA"], kS=WL["kS"], m=WL["m"], schur_diag=WL["schur_diag"],
                         restart=WL["restart"])
        for _ in range(2):
            for x in xs:
                x.zero_()
            Bq.solve(bs, xs, rtol=WL["rtol"])
        torch.cuda.synchronize()
        e0.record()
        for _ in range(reps):
            for x in xs:
                x.zero_()
            _, its_q, rels_q = Bq.solve(bs, xs, rtol=WL["rtol"])
        e1.record()
        e1.synchronize()
        queue_ms = e0.elapsed_time(e1) / reps
        queue_mode = Bq.krylov_mode
        Bq.close()
    finally:
        if prev is None:
            os.environ.pop("STOKES_BATCH_QUEUE", None)
        else:
            os.environ["STOKES_BATCH_QUEUE"] = prev
    return {"meshes": len(members), "sizes": [r["n"] for r in recipe], "gammas": [r["gamma"] for r in recipe],
            "dofs_total": dofs_total, "batch_ms": round(batch_ms, 3), "sequential_ms": round(seq_ms, 3),
            "speedup_vs_sequential": round(seq_ms / batch_ms, 3),
            "batch_mdof_s": round(dofs_total / (batch_ms / 1e3) / 1e6, 3), "iterations": its,
            "max_rel_residual": max(rels),
            "work_queue": {"krylov_mode": queue_mode, "batch_ms": round(queue_ms, 3),
                           "speedup_vs_sequential": round(seq_ms / queue_ms, 3), "iterations": its_q,
                           "max_rel_residual": max(rels_q)}}


def run_adjoint():
    """Forward + adjoint FP64-MG solves and the per-cell viscosity gradient on 32^3 Cartesian hexes,
    mu_c = exp(g_c) (seeded Gaussian field, correlation length 0.2), J = 0.5 ||u - u_obs||^2."""
    import numpy as np
    import torch
    import workloads as W
    from paper_2205_15770_gb300 import StokesMG, stokes_solve_fn
    n = 32
    mu = np.exp(W.gaussian_field_cells(n, seed=0)).reshape(-1)
    mu_obs = np.exp(W.gaussian_field_cells(n, seed=1)).reshape(-1)
    f = torch.as_tensor(W.fourier_forcing(3, 2, (n,) * 3, seed=0).reshape(-1), device="cuda")
    S = StokesMG(dim=3, n=(n,) * 3, n_levels=5, k=2, vcycle_fp32=False, kA=WL["kA"], kS=WL["kS"], m=WL["m"],
                 schur_diag=WL["schur_diag"])
    u_obs = stokes_solve_fn(S, torch.as_tensor(mu_obs, device="cuda"), f, 1e-10).detach()
    nu = S.sizes()[0]
    S.set_viscosity(mu)
    b = S.mass_rhs(f)
    x, _, _ = S.solve(b, rtol=1e-10)
    torch.cuda.synchronize()
    e = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
    e[0].record()
    x, it_f, _ = S.solve(b, rtol=1e-10)
    e[1].record()
    gx = torch.zeros_like(x)
    gx[:nu] = x[:nu] - u_obs[:nu]
    lam, it_a, _ = S.solve(gx, rtol=1e-10)
    e[2].record()
    gmu = S.cell_grad(x, lam)
    gf = S.mass(lam[:nu].contiguous(), full_rows=True)
    e[3].record()
    e[3].synchronize()
    S.close()
    return {"mesh": "32^3 Cartesian, Q2-Q1, FP64 MG, rtol 1e-10", "forward_ms": round(e[0].elapsed_time(e[1]), 3),
            "adjoint_ms": round(e[1].elapsed_time(e[2]), 3), "gradients_ms": round(e[2].elapsed_time(e[3]), 3),
            "iterations": [it_f, it_a], "max_abs_dJ_dmu": float(gmu.abs().max()),
            "max_abs_dJ_df": float(gf.abs().max())}


def run_smoother_sweep(args):
    """Time-to-1e-8 of the workload's three FP32-MG solves for each (k_A, k_S, m) in SWEEP, with the
    Schur-complement diagonals d and loc."""
    import torch
    from paper_2205_15770_gb300 import StokesMG
    V = perturbed_vertices()
    f = torch.as_tensor(forcing(), device="cuda")
    for sd, (kA, kS, m) in [(sd, c) for sd in ("d", "loc") for c in SWEEP]:
        tot, its = 0.0, []
        for g in WL["gammas"]:
            S = StokesMG(dim=3, n=WL["n"], n_levels=WL["levels"], k=WL["k"], vertices=V, gamma_rho=g, kA=kA, kS=kS,
                         m=m, schur_diag=sd)
            b = S.mass_rhs(f)
            x = torch.zeros_like(b)
            for _ in range(2):
                x.zero_()
                S.solve(b, x, rtol=WL["rtol"], maxit=100)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(3):
                x.zero_()
                _, it, _ = S.solve(b, x, rtol=WL["rtol"], maxit=100)
            e1.record()
            e1.synchronize()
            tot += e0.elapsed_time(e1) / 3
            its.append(it)
            S.close()
        print(json.dumps({"schur_diag": sd, "kA": kA, "kS": kS, "m": m, "ms_per_solve": round(tot / len(WL["gammas"]), 3),
                          "iterations": its}), flush=True)


def cavity_lid(S, dim, n):
    """Dirichlet vector of the lid-driven cavity: u = (1, 0[, 0]) on the top face (y = 1 in 2D,
    z = 1 in 3D) without its edges, 0 on the other walls (Sec. 4.3 / 4.5)."""
    import numpy as np
    import torch
    N = 2 * n + 1
    nv = N ** dim
    uD = np.zeros(S.size())
    idx = np.arange(nv)
    gx = idx % N
    top = (idx // (N ** (dim - 1))) == N - 1
    inner = (gx > 0) & (gx < N - 1)
    if dim == 3:
        gy = (idx // N) % N
        inner &= (gy > 0) & (gy < N - 1)
    uD[:nv][top & inner] = 1.0
    return torch.as_tensor(uD, device="cuda")


def run_paper_sweep(args):
    """The paper's rate study on the GPU (Sec. 4.1 protocol, Sec. 4.3.3 / 4.5 settings): stationary
    FP64 multigrid from x = 0 on the lid-driven cavity, 2D Q2-Q1 128^2 (148,739 DoFs, 7 levels) and
    3D Q2-Q1 16^3 (112,724 DoFs, 4 levels), mu = 1, f = 0, local Schur diagonal; for every
    (k_A, k_S) in {0..3}^2, m in {1, 2} and V / W cycles: q = (r^j / r^{j-3})^(1/3) after at most 15
    cycles or a 1e-10 reduction, T_iter (ms per cycle) and T(0.1) = T_iter log(0.1) / log(q)."""
    import math
    import torch
    from paper_2205_15770_gb300 import StokesMG
    cases = [(2, 128, 7), (3, 16, 4)]
    for dim, n, levels in cases:
        for cyc in ("V", "W"):
            for m in (1, 2):
                for kA in range(4):
                    for kS in range(4):
                        S = StokesMG(dim=dim, n=(n,) * dim, n_levels=levels, k=2, kA=kA, kS=kS, m=m, cycle=cyc,
                                     vcycle_fp32=False)
                        uD = cavity_lid(S, dim, n)
                        b = S.lift_rhs(uD, torch.zeros_like(uD))
                        x = torch.zeros_like(b)
                        S.mg_iterate(b, x.zero_(), max_iter=2, reduction=1e-10, allow_divergence=True)
                        torch.cuda.synchronize()
                        t0 = time.perf_counter()
                        _, it, hist, q = S.mg_iterate(b, x.zero_(), max_iter=15, reduction=1e-10,
                                                      allow_divergence=True)
                        torch.cuda.synchronize()
                        t_iter = (time.perf_counter() - t0) / max(it, 1) * 1e3
                        ok = bool(hist) and 0 < q < 1
                        t01 = t_iter * math.log(0.1) / math.log(q) if ok else None
                        print(json.dumps({"dim": dim, "dofs": S.size(), "cycle": cyc, "m": m, "kA": kA, "kS": kS,
                                          "iterations": it, "q": round(q, 4) if ok else None,
                                          "converged": bool(hist) and hist[-1] <= 1e-10 * hist[0],
                                          "T_iter_ms": round(t_iter, 3),
                                          "T_0.1_ms": round(t01, 3) if t01 else None}), flush=True)
                        S.close()


def run_schur_sweep(args):
    """The paper's comparison of Schur-complement diagonals on its two 2D problems: the laser beam
    (Sec. 4.2: unit square, mu = 0.0022, u_D = 0, Gaussian force c1 exp(-c2 |x - x0|^2) in y at
    x0 = (0.75, 0.75)) and the driven cavity (Sec. 4.3.2), both Q2-Q1 on 16^2 (2,467 DoFs, 4 levels),
    stationary FP64 W-cycle multigrid from x = 0; Jacobi (k_A = k_S = 0) and Chebyshev degree 3;
    smoothing steps m in {1, 2, 4, 8, 16}; D_S~ in {loc, p, d, exact}: rate q = (r^j / r^{j-3})^(1/3)."""
    import torch
    import workloads as W
    from paper_2205_15770_gb300 import StokesMG
    dim, n, levels = 2, 16, 4
    for problem in ("laser", "cavity"):
        for kdeg in (0, 3):
            for diag in ("loc", "p", "d", "exact"):
                for m in (1, 2, 4, 8, 16):
                    mu = 0.0022 if problem == "laser" else 1.0
                    S = StokesMG(dim=dim, n=(n,) * dim, n_levels=levels, k=2, mu=mu, kA=kdeg, kS=kdeg, m=m,
                                 cycle="W", schur_diag=diag, vcycle_fp32=False)
                    if problem == "laser":
                        f = torch.as_tensor(W.laser_beam_forcing((n, n)).reshape(-1), device="cuda")
                        b = S.mass_rhs(f)
                    else:
                        uD = cavity_lid(S, dim, n)
                        b = S.lift_rhs(uD, torch.zeros_like(uD))
                    _, it, hist, q = S.mg_iterate(b, torch.zeros_like(b), max_iter=15, reduction=1e-10,
                                                  allow_divergence=True)
                    ok = bool(hist) and 0 < q < 1
                    print(json.dumps({"problem": problem, "dofs": S.size(), "k": kdeg, "diag": diag, "m": m,
                                      "iterations": it, "q": round(q, 4) if ok else None}), flush=True)
                    S.close()


def run_variants(args):
    """The next-steps rows on the 32^3 workload (same mesh, forcing and gamma = 1e2): FP32-MG FGMRES
    solves to 1e-8 (ms per solve, iterations) and FP32 / FP64 vmult throughput for
      laplacian:  the benchmark's form (reference line),
      sym:        mu eps(u):eps(v) + gamma rho u.v with per-cell mu = exp(g1), rho = exp(g2 / 2)
                  (g1, g2 seeded Gaussian fields, correlation length 0.2, sample std 1),
      stabilised: C = 1e-2 M_p + 1e-1 sum_tau h_tau^2 K_p,tau."""
    import numpy as np
    import torch
    import workloads as W
    from paper_2205_15770_gb300 import StokesMG
    V = perturbed_vertices()
    n = WL["n"][0]
    mu = np.exp(W.gaussian_field_cells(n, seed=0)).reshape(-1)
    rho = np.exp(0.5 * W.gaussian_field_cells(n, seed=1)).reshape(-1)
    variants = {"laplacian": {}, "sym": dict(sym_grad=True, mu_cell=mu, rho_cell=rho),
                "stabilised": dict(c_mass=1e-2, c_grad=1e-1)}
    f = torch.as_tensor(forcing(), device="cuda")
    ev = lambda: torch.cuda.Event(enable_timing=True)
    for name, kw in variants.items():
        S = StokesMG(dim=3, n=WL["n"], n_levels=WL["levels"], k=WL["k"], vertices=V, gamma_rho=1e2, kA=WL["kA"],
                     kS=WL["kS"], m=WL["m"], schur_diag=WL["schur_diag"], **kw)
        b = S.mass_rhs(f)
        x = torch.zeros_like(b)
        for _ in range(2):
            S.solve(b, x.zero_(), rtol=WL["rtol"])
        torch.cuda.synchronize()
        e0, e1 = ev(), ev()
        e0.record()
        for _ in range(5):
            _, its, rel = S.solve(b, x.zero_(), rtol=WL["rtol"])
        e1.record()
        e1.synchronize()
        row = {"variant": name, "dofs": S.size(), "solve_ms": round(e0.elapsed_time(e1) / 5, 3), "iterations": its,
               "final_rel_residual": rel, "fused_levels_fp32": S.fused_levels(32)}
        for dt in (torch.float32, torch.float64):
            xv = torch.randn(S.size(), dtype=dt, device="cuda")
            yv = torch.empty_like(xv)
            for _ in range(3):
                S.vmult(xv, yv)
            torch.cuda.synchronize()
            reps = 20 if dt == torch.float32 else 5
            e0.record()
            for _ in range(reps):
                S.vmult(xv, yv)
            e1.record()
            e1.synchronize()
            row[f"vmult_{str(dt)[-7:]}_mdof_s"] = round(S.size() / (e0.elapsed_time(e1) / reps / 1e3) / 1e6, 1)
        print(json.dumps(row), flush=True)
        S.close()


def run_mesh_sweep(args):
    """Mesh independence of the benchmark's solver: the same perturbed unit-cube workload (0.1 h
    perturbation of each mesh, seed 0, Q2-Q1, coarsest mesh 2^3) on n = 8..128 cells per direction,
    FP32-MG FGMRES to 1e-8 for gamma = 0 and 1e2: iterations and solve time per n."""
    import torch
    import workloads as W
    from paper_2205_15770_gb300 import StokesMG
    for n in (8, 16, 32, 64, 128):
        nl = n.bit_length() - 1  # n = 2^(nl) -> levels down to 2^3
        V = W.perturbed_vertices(3, (n, n, n), seed=WL["seed"], amplitude=WL["amplitude"])
        f = torch.as_tensor(W.fourier_forcing(3, WL["k"], (n, n, n), seed=WL["seed"]).reshape(-1), device="cuda")
        row = {"n": n, "levels": nl, "iterations": [], "solve_ms": []}
        for g in (0.0, 1e2):
            S = StokesMG(dim=3, n=(n, n, n), n_levels=nl, k=WL["k"], vertices=V, gamma_rho=g, kA=WL["kA"],
                         kS=WL["kS"], m=WL["m"], schur_diag=WL["schur_diag"], restart=WL["restart"])
            row["dofs"] = S.size()
            b = S.mass_rhs(f)
            x = torch.zeros_like(b)
            S.solve(b, x, rtol=WL["rtol"])
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            reps = 3
            e0.record()
            for _ in range(reps):
                x.zero_()
                _, its, rel = S.solve(b, x, rtol=WL["rtol"])
            e1.record()
            e1.synchronize()
            row["iterations"].append(its)
            row["solve_ms"].append(round(e0.elapsed_time(e1) / reps, 3))
            S.close()
            del S
            torch.cuda.empty_cache()
        row["mdof_s"] = round(row["dofs"] / (min(row["solve_ms"]) / 1e3) / 1e6, 2)
        print(json.dumps(row), flush=True)


def run_channel(args):
    """Q_k-Q_{k-1} channel [0,4] x [0,1]^2 on 64^3 cells (aspect 4:1:1), parabolic inflow
    u = 16 y(1-y) z(1-z) on x = 0, no-slip walls, do-nothing outflow at x = 4, mu = 1e-3, 6 levels.
    For k = 2, 3, 4: vmult throughput (FP32 / FP64, MDoF/s) through stokes_vmult, the full-operator
    cell kernel's duration, and its HBM fraction for the algorithmic bytes (x read once, y written
    once); for k = 3 one FP32-MG FGMRES solve of the lifted problem to 1e-8."""
    import torch
    from paper_2205_15770_gb300 import StokesMG
    peaks, src = measured_peaks()
    hbm = (peaks or {}).get("hbm_gbs", FALLBACK_HBM_GBS)
    props = torch.cuda.get_device_properties(0)
    pk = {prec: alu_peak_tflops(prec, props.multi_processor_count, 2070.0) for prec in (32, 64)}
    out = {"workload": "channel [0,4]x[0,1]^2, 64^3 hexes, mu 1e-3, inflow 16y(1-y)z(1-z), do-nothing outflow",
           "hbm_peak_gbs": hbm, "hbm_peak_source": src, "fp32_peak_tflops": round(pk[32], 2),
           "fp64_peak_tflops": round(pk[64], 3),
           "flops_model": "full operator K x per affine cell: k=2 6,963, k=3 21,808, k=4 53,005 flops",
           "k": {}}
    # k = 2, 3, 4 on 64^3 cells, and the Q2 size sweep's 128^3 point (53.1M DoFs, 7 levels)
    for n, k in ((64, 2), (64, 3), (64, 4), (128, 2)):
        nl = 6 if n == 64 else 7
        S = StokesMG(dim=3, n=(n, n, n), n_levels=nl, k=k, mu=1e-3, hi=(4.0, 1.0, 1.0), dirichlet_faces=0x3D,
                     kA=WL["kA"], kS=WL["kS"], m=WL["m"], schur_diag=WL["schur_diag"])
        N = S.size()
        row = {"dofs": N, "cells": n ** 3}
        for prec, dt in ((32, torch.float32), (64, torch.float64)):
            x = torch.randn(N, dtype=dt, device="cuda")
            y = torch.empty_like(x)
            for _ in range(2):
                S.vmult(x, y)
            reps = 20 if prec == 32 else 4
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(reps):
                S.vmult(x, y)
            e1.record()
            e1.synchronize()
            ms = e0.elapsed_time(e1) / reps
            kern = S.time_apply(7, precision=prec, reps=reps)
            bytes_alg = BYTES_PER_DOF_8D[(prec, "affine")] * N
            tflops = FLOPS_PER_CELL_8D[("affine", k)] * n ** 3 / (kern / 1e3) / 1e12
            row[f"fp{prec}"] = {"vmult_ms": round(ms, 3), "mdof_s": round(N / (ms / 1e3) / 1e6, 1),
                                "kernel_ms": round(kern, 3), "launch_shape": S.launch_shapes(prec)[-1],
                                "hbm_frac_of_kernel": round(bytes_alg / (kern / 1e3) / 1e9 / hbm, 4),
                                "tflops": round(tflops, 3), "alu_frac": round(tflops / pk[prec], 4)}
        if k == 3:
            nodes = S.velocity_nodes()
            nu, _ = S.sizes()
            nv = nu // 3
            uD = torch.zeros(N, dtype=torch.float64, device="cuda")
            inflow = nodes[:, 0] == 0.0
            yy, zz = nodes[:, 1], nodes[:, 2]
            uD[:nv] = torch.where(inflow, 16 * yy * (1 - yy) * zz * (1 - zz), torch.zeros_like(yy))
            b = S.lift_rhs(uD, torch.zeros_like(uD))
            xs = torch.zeros_like(b)
            S.solve(b, xs, rtol=WL["rtol"])
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            xs.zero_()
            e0.record()
            _, its, rel = S.solve(b, xs, rtol=WL["rtol"])
            e1.record()
            e1.synchronize()
            ms = e0.elapsed_time(e1)
            row["solve"] = {"ms": round(ms, 2), "iterations": its, "rel_residual": rel,
                            "mdof_s": round(N / (ms / 1e3) / 1e6, 2),
                            "max_u": float((xs[:nv] + uD[:nv]).max())}
        if n == 64:
            out["k"][k] = row
        else:
            out["q2_128cubed"] = row
        S.close()
        del S
        torch.cuda.empty_cache()
    print(json.dumps(out))


def run_channel_smoothers(args):
    """The Q3 channel solve of run_channel (64^3 cells of aspect 4:1:1, lifted inflow, rtol 1e-8,
    FP32 V-cycle in FP64 FGMRES(30), Schur diagonal d) for several smoothers (k_A, k_S, m): FGMRES
    iterations and ms per solve.  The paper's best settings for its channel benchmark (Schafer-Turek,
    Sec. 4.4) use higher Chebyshev degrees than the cube's (1, 1, 2)."""
    import torch
    from paper_2205_15770_gb300 import StokesMG
    n, k, nl = 64, 3, 6
    for kA, kS, m in ((1, 1, 2), (2, 1, 2), (3, 1, 2), (2, 2, 2), (3, 2, 2), (3, 3, 2)):
        S = StokesMG(dim=3, n=(n, n, n), n_levels=nl, k=k, mu=1e-3, hi=(4.0, 1.0, 1.0), dirichlet_faces=0x3D,
                     kA=kA, kS=kS, m=m, schur_diag="d")
        N = S.size()
        nodes = S.velocity_nodes()
        nu, _ = S.sizes()
        nv = nu // 3
        uD = torch.zeros(N, dtype=torch.float64, device="cuda")
        inflow = nodes[:, 0] == 0.0
        yy, zz = nodes[:, 1], nodes[:, 2]
        uD[:nv] = torch.where(inflow, 16 * yy * (1 - yy) * zz * (1 - zz), torch.zeros_like(yy))
        b = S.lift_rhs(uD, torch.zeros_like(uD))
        xs = torch.zeros_like(b)
        S.solve(b, xs, rtol=WL["rtol"])
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        xs.zero_()
        e0.record()
        _, its, rel = S.solve(b, xs, rtol=WL["rtol"])
        e1.record()
        e1.synchronize()
        print(json.dumps({"kA": kA, "kS": kS, "m": m, "schur_diag": "d", "dofs": N, "iterations": its,
                          "ms_per_solve": round(e0.elapsed_time(e1), 2), "rel_residual": rel}), flush=True)
        S.close()
        del S
        torch.cuda.empty_cache()


def run_level_times(args):
    """Where a V-cycle's time goes: the FP32 V-cycle of the workload's family (perturbed unit cube,
    gamma 1e2, the bench smoother) on 4^3 .. 32^3 cells (coarsest 2^3), each timed over 50 cycles
    (CUDA events, captured cycle graphs), and on the 32^3 hierarchy the cell kernel's duration per
    level, block set (A, B^T, B, A + B^T, full) and launch shape (stokes_time_apply, 200 launches)."""
    import torch
    import workloads as W
    from paper_2205_15770_gb300 import StokesMG
    for n in (4, 8, 16, 32):
        nl = {4: 2, 8: 3, 16: 4, 32: 5}[n]
        V = W.perturbed_vertices(3, (n,) * 3, seed=WL["seed"], amplitude=WL["amplitude"])
        S = StokesMG(dim=3, n=(n,) * 3, n_levels=nl, k=2, vertices=V, gamma_rho=1e2,
                     kA=WL["kA"], kS=WL["kS"], m=WL["m"], schur_diag=WL["schur_diag"])
        f = torch.as_tensor(W.fourier_forcing(3, 2, (n,) * 3, seed=WL["seed"]).reshape(-1), device="cuda")
        b = S.mass_rhs(f).float()
        x = torch.zeros_like(b)
        for _ in range(5):
            x.zero_()
            S.vcycle(b, x)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(50):
            x.zero_()
            S.vcycle(b, x)
        e1.record()
        e1.synchronize()
        row = {"n": n, "levels": nl, "vcycle_fp32_ms": round(e0.elapsed_time(e1) / 50, 4),
               "launch_shapes_fp32": S.launch_shapes(32), "fused_smoothing_levels": S.fused_levels(32),
               "fp32_geometry_stored": S.geometry_stored(32)}
        if n == 32:
            apply_us = {}
            for l in range(1, nl):
                for sh in sorted({S.launch_shapes(32)[l], 5}):
                    S.set_launch_shape(l, sh, precision=32)
                    apply_us[f"level{l}_shape{sh}"] = {
                        name: round(S.time_apply(blk, level=l, precision=32, reps=200) * 1e3, 2)
                        for name, blk in (("A", 1), ("BT", 2), ("B", 4), ("A+BT", 3), ("full", 7))}
            row["apply_us"] = apply_us
        print(json.dumps(row), flush=True)
        S.close()


def run_kernel_only(args):
    """Set up one context of the workload (gamma = 1e2) and launch one cell kernel of the finest
    level a few times inside a cudaProfilerStart/Stop range, for ncu: the FP32 A-block apply
    (--kernel-precision 32) or the FP64 full operator of the FGMRES loop (64)."""
    import torch
    from paper_2205_15770_gb300 import StokesMG
    torch.cuda.set_device(0)
    os.environ.setdefault("STOKES_NO_AUTOTUNE", "1")
    if args.kernel_case == "channel-q2-128":  # the channel's Q2 point at 128^3 Cartesian cells (53.1M DoFs)
        nl, cells = 7, 128 ** 3
        S = StokesMG(dim=3, n=(128, 128, 128), n_levels=nl, k=2, mu=1e-3, hi=(4.0, 1.0, 1.0), dirichlet_faces=0x3D,
                     kA=WL["kA"], kS=WL["kS"], m=WL["m"], schur_diag=WL["schur_diag"])
    else:
        nl, cells = WL["levels"], WL["n"][0] * WL["n"][1] * WL["n"][2]
        S = StokesMG(dim=3, n=WL["n"], n_levels=nl, k=WL["k"], vertices=perturbed_vertices(), gamma_rho=1e2,
                     kA=WL["kA"], kS=WL["kS"], m=WL["m"], schur_diag=WL["schur_diag"])
    prec = args.kernel_precision
    mode = args.kernel_mode if args.kernel_mode else (1 if prec == 32 else 7)
    # the finest level's launch shape is pinned and nothing is timed (a profiler changes the setup's timings): shape 5,
    # the plane kernels of k = 2
    shape = args.kernel_shape if args.kernel_shape else 5
    S.set_launch_shape(nl - 1, shape, precision=prec)
    S.time_apply(mode, precision=prec, reps=3)
    torch.cuda.synchronize()
    torch.cuda.profiler.start()
    ms = S.time_apply(mode, precision=prec, reps=3)
    torch.cuda.profiler.stop()
    print(json.dumps({"kernel": f"cell kernel, blocks {mode}, FP{prec}, launch shape {S.launch_shapes(prec)[-1]}"
                                f"{', plane form' if shape == 5 and S.plane_levels(prec)[-1] else ''}",
                      "avg_launch_us": ms * 1e3, "cells": cells}))
    S.close()


def run_reference(args):
    """The oracle as the reference arm: each step one FP64-MG FGMRES solve of the 32^3 workload at
    gamma = 1e2 (the CPU program is bounded to one untimed warm-up solve at most)."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    warm = min(args.warmup, 1)
    o = run_oracle_subprocess(args.steps, warm, threads=1)
    value = o["dofs"] / o["seconds_per_step"] / 1e6
    sample = (f"each step: one FP64-MG FGMRES(30) solve to 1e-8 of the 32^3 workload at gamma {ORACLE_GAMMA:g} "
              "(859,812 DoFs, 5 levels), numpy/scipy, 1 thread; setup untimed")
    out = {
        "impl": "reference", "metric": METRIC, "value": round(value, 4), "unit": "MDoF/s",
        "n_gpus": int(os.environ.get("WORLD_SIZE", "1")), "steps": args.steps, "warmup": warm,
        "ms_per_step": round(o["seconds_per_step"] * 1e3, 1), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD_NAME, "dofs_per_solve": o["dofs"], "solves_per_step": 1,
                   "parallelism": "single"},
        "cpu_baseline": {"value": round(value, 4), "unit": "MDoF/s", "cores": 1, "kind": "oracle", "sample": sample,
                         "host": host_cpu_info()},
        "e2e": {"value": round(value, 4), "unit": "MDoF/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "iterations": o["iterations"],
    }
    print(json.dumps(out))


def main():
    ap = argparse.ArgumentParser(description=__doc__.split("\n")[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=("ours", "reference"), default="ours")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true", help="skip the batched and adjoint measurements")
    ap.add_argument("--mesh-sweep", action="store_true",
                    help="the workload on 8^3..128^3 cells: FGMRES iterations and solve time per mesh size")
    ap.add_argument("--variants", action="store_true",
                    help="32^3 workload in the symmetric-gradient form and with a stabilisation block: solve, vmult")
    ap.add_argument("--schur-sweep", action="store_true",
                    help="2D laser beam and cavity 16^2: rates q for the Schur diagonals loc/p/d/exact, k = 0, 3, m = 1..16")
    ap.add_argument("--profile-range", action="store_true",
                    help="bracket the timed steps by cudaProfilerStart/Stop (for ncu --profile-from-start off)")
    ap.add_argument("--channel", action="store_true",
                    help="64^3 channel (Q2..Q4): vmult throughput, HBM fraction, Q3 solve of the lifted problem")
    ap.add_argument("--level-times", action="store_true",
                    help="FP32 V-cycle time on 4^3..32^3 and the cell kernel's duration per level and block set")
    ap.add_argument("--channel-smoothers", action="store_true",
                    help="Q3 channel solve for several smoother settings (k_A, k_S, m)")
    ap.add_argument("--paper-sweep", action="store_true",
                    help="the paper's (k_A, k_S, m) rate study on the lid-driven cavities (stationary FP64 MG)")
    ap.add_argument("--smoother-sweep", action="store_true",
                    help="time-to-1e-8 of the workload for a list of (k_A, k_S, m); prints one JSON line each")
    ap.add_argument("--kernel-precision", type=int, choices=(32, 64), default=32,
                    help="with --kernel-only: the FP32 A block (32) or the FP64 full operator (64)")
    ap.add_argument("--kernel-mode", type=int, default=0,
                    help="with --kernel-only: the block bit set (1 A, 2 B^T, 4 B, 7 full; default 1 / 7 by precision)")
    ap.add_argument("--kernel-shape", type=int, default=0,
                    help="with --kernel-only: the finest level's launch shape (default 5)")
    ap.add_argument("--kernel-case", choices=("workload", "channel-q2-128"), default="workload",
                    help="--kernel-only: the 32^3 workload, or the channel's Q2 point at 128^3 cells")
    ap.add_argument("--kernel-only", action="store_true",
                    help="only launch the dominant kernel inside a profiler range (for ncu --set full)")
    ap.add_argument("--cpu-table", action="store_true",
                    help="the oracle's CPU-baseline table on this host (SpMV rates, solve times; 1 and all threads)")
    ap.add_argument("--_oracle-sample", nargs=2, type=int, default=None, dest="oracle_sample")
    ap.add_argument("--_cpu-table-rows", action="store_true", dest="cpu_table_rows")
    args = ap.parse_args()
    if args.oracle_sample is not None:
        print(json.dumps(oracle_sample(*args.oracle_sample)))
        return
    if args.cpu_table_rows:
        print(json.dumps(cpu_table_rows()))
        return
    if args.cpu_table:
        run_cpu_table(args)
        return
    if args.warmup < 3 and args.impl == "ours":
        ap.error("--warmup must be >= 3")
    if args.channel:
        run_channel(args)
    elif args.channel_smoothers:
        run_channel_smoothers(args)
    elif args.level_times:
        run_level_times(args)
    elif args.paper_sweep:
        run_paper_sweep(args)
    elif args.smoother_sweep:
        run_smoother_sweep(args)
    elif args.schur_sweep:
        run_schur_sweep(args)
    elif args.variants:
        run_variants(args)
    elif args.mesh_sweep:
        run_mesh_sweep(args)
    elif args.kernel_only:
        run_kernel_only(args)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()

#!/usr/bin/env python3
"""Newton solves/s of the MAS-PCG linear solve on the 64^3 stiffness sweep.

Workload (synthetic, seeded): a 64^3-vertex tet cube (262,144 vertices,
786,432 DOF, 1,250,235 tets split 5 per cell), stable Neo-Hookean Hessian
with E in {1e5, 1e7, 1e9} Pa, nu = 0.4, lumped mass / dt^2 (rho = 1000,
dt = 0.01), 200k PSD contact blocks between vertices closer than 2h; 8 N(0,1)
right-hand sides; 3-level MAS with 32-node domains; PCG to 1e-6 relative
residual.  It stands in for the paper's FEM scenes, which are not available.

One step = one Newton solve of each of the three systems: hash-key assembly
of its 13.4M triplets, device MAS build, and 8-RHS PCG (supplement Eq. 1:
T = T_ga + T_pa + N_pcg T_pcg).  The level-0 partition is computed once per
mesh before timing, as the paper runs METIS once before the simulation.
`value` counts Newton solves (one system, all its right-hand sides) per
second with inputs resident in HBM; `e2e` repeats the step through the
same public API with the triplets and right-hand sides copied from pinned
host memory every step and the solutions copied back.
"""

import argparse
from concurrent.futures import ThreadPoolExecutor
import json
import os
import statistics
import subprocess
import sys
import tempfile
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

FP64_FMA_PER_CLK_PER_SM = 2  # GB300: derived from the nominal 1.25 TFLOP/s FP64 at 2.07 GHz, 152 SMs
TOL = 1e-6
# The headline metric as named for this workload: `value` is the FP64 path's
# Newton solves/s; the mixed-precision forms are under forms.mixed_precision
# and the SpMV's HBM GB/s under roofline.hbm_gbs / kernels.spmv_hbm_gbs.
METRIC = "Newton solves/s to 1e-6 rel. residual (FP64 vs mixed MAS-PCG); SpMV HBM GB/s"


# what brief() leaves out beside lists and long texts
DETAILS = {"phase_ms", "phase_ms_one_step", "phase_ms_one_solve", "launches_one_step", "kernels", "roofline", "host",
           "clocks"}


def brief(form):
    """A form's record without its tables, lists and long texts, numbers to five digits."""
    out = {}
    for k, v in form.items():
        if isinstance(v, dict) and k not in DETAILS:
            v = brief(v)
            if v:
                out[k] = v
        elif isinstance(v, bool) or (isinstance(v, str) and (len(v) <= 60 or k == "error")):
            out[k] = v
        elif hasattr(v, "item") or isinstance(v, (int, float)):
            v = v.item() if hasattr(v, "item") else v
            out[k] = float(f"{v:.5g}") if isinstance(v, float) else v
    return out


def _json_scalar(o):
    """numpy scalars in the output line as plain numbers."""
    if hasattr(o, "item"):
        return o.item()
    raise TypeError(f"not serialisable: {type(o).__name__}")


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=3)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", default="ours", choices=["ours", "reference"])
    p.add_argument("--grid", type=int, default=64, help="vertices per cube edge (64 = the named workload)")
    p.add_argument("--nrhs", type=int, default=8)
    p.add_argument("--sweep", default="1e5,1e7,1e9",
                   help="Young's moduli of the step's systems (the named workload: 1e5,1e7,1e9; a single value "
                        "keeps profiling runs small)")
    p.add_argument("--precision", default="fp64", choices=["fp64", "fp32", "bf16"],
                   help="preconditioner storage of the main path (FP64 PCG throughout)")
    p.add_argument("--spmv", default="ff", choices=["row", "srbk", "ff"],
                   help="row: FP64 row gather; srbk: the paper's SRBK; ff: row gather in float-float on the FP32 units")
    p.add_argument("--e2e-steps", type=int, default=2)
    p.add_argument("--mixed-steps", type=int, default=3, help="timed steps of the mixed-precision form")
    p.add_argument("--no-lanes", dest="lanes", action="store_false",
                   help="solve the systems of a step one after another on one stream")
    p.add_argument("--streams", type=int, default=0,
                   help="with lanes: library contexts / streams working the queue (0 = one per system of a step)")
    p.add_argument("--step-sync", dest="queue", action="store_false",
                   help="with lanes: wait for all systems of a step before the next step starts, instead of one "
                        "queue over the timed steps' solves")
    p.add_argument("--no-autotune", dest="autotune", action="store_false",
                   help="keep the default launch shapes instead of tuning them first")
    p.add_argument("--batch-steps", type=int, default=2, help="timed steps of the batched form (64 uneven systems)")
    p.add_argument("--cloth", type=int, default=512,
                   help="vertices per edge of the stiff-cloth precision case (0 = skip)")
    p.add_argument("--set-tune", action="append", default=[], metavar="NAME=VALUE",
                   help="force a launch shape after tuning (names as in config.launch_shapes), e.g. "
                        "spmv_lanes=2; repeatable")
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--partition-steps", type=int, default=1,
                   help="timed solves per variant of the partition / level comparison (0 = skip)")
    p.add_argument("--no-config1", dest="config1", action="store_false",
                   help="skip the plain FP64 solve of the 16^3 cube (forms.plain16)")
    p.add_argument("--no-abd", dest="abd", action="store_false",
                   help="skip the differentiation form on the 100^3 + 2,000-body coupled scene")
    p.add_argument("--abd-steps", type=int, default=2, help="timed steps of the coupled-scene form")
    p.add_argument("--no-newton", dest="newton", action="store_false",
                   help="skip the Newton loop on the elastic cube (forms.newton)")
    p.add_argument("--element-probe", type=int, default=0, metavar="GRID",
                   help="instead of the solve benchmark: build the Newton form's elastic cube at GRID^3, assemble "
                        "its Hessian once and refill it --refills times (a short run for ncu captures)")
    p.add_argument("--refills", type=int, default=3)
    p.add_argument("--cloth-probe", type=int, default=0, metavar="N",
                   help="only the cloth element-Hessian kernels on an N x N sheet, --refills times (for captures)")
    p.add_argument("--micro", action="store_true",
                   help="instead of the solve benchmark: the paper's reduction and SpMV microbenchmarks")
    p.add_argument("--oracle-sample", default=None, help=argparse.SUPPRESS)  # worker mode
    return p.parse_args()


# --------------------------------------------------------------------------- oracle sample
def host_info():
    """Host cores and CPU model of the machine the oracle runs on."""
    model = None
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=20).stdout
        for ln in out.splitlines():
            if ln.lower().startswith("model name"):
                model = ln.split(":", 1)[1].strip()
                break
    except Exception:  # noqa: BLE001
        pass
    return {"nproc": os.cpu_count(), "cpu_model": model}


_ORACLE_SHARED = {}  # set before the pool forks: the children inherit the operators, nothing is pickled


def _oracle_pcg_iters(job):
    """Worker: `iters` oracle PCG iterations on RHS j (forked from the sample
    process, which never touches a GPU)."""
    j, iters = job
    from oracle import pcg

    A, M, bs = _ORACLE_SHARED["A"], _ORACLE_SHARED["M"], _ORACLE_SHARED["b"]
    t0 = time.perf_counter()
    pcg.pcg(A, M, bs[j], fixed_iters=iters)
    return time.perf_counter() - t0


def oracle_sample(spec):
    """Time the oracle on bounded samples of the workload (run in a fresh
    process with one BLAS thread per process and no GPU).  Input generation
    and the once-per-mesh partition are not timed.  Phases per sample:
    `phases` lists which of "ga" (assembly), "pa" (MAS build) and "pcg" run.
    PCG: `iters` iterations on one RHS (t_iter), and, with procs > 1, `iters`
    iterations on each of `procs` RHS in as many concurrent processes
    (t_iter_par: wall time per iteration, all procs RHS advancing).  Prints
    one JSON object: the samples and the host."""
    from oracle import assembly, mas, partition, pcg
    from synth.workloads import rhs, stiffness_sweep

    systems = stiffness_sweep(Es=tuple(spec["Es"]), n=spec["grid"])
    V = systems[0].n_vertices
    mp, _ = partition.map_remap(partition.recursive_bisection(systems[0].X, 32), 32)  # pre-simulation
    procs = int(spec.get("procs", 1))
    bs = rhs(3 * V, max(procs, 1))
    phases = spec.get("phases", ["ga", "pa", "pcg"])
    cache = {}
    out = []
    for q in range(spec["samples"]):
        si = q % len(systems)
        sys_ = systems[si]
        ph = phases[q % len(phases)] if spec.get("cycle") else None
        rec = {"E": sys_.params["E"], "V": V}
        if ph in (None, "ga") or si not in cache:
            t0 = time.perf_counter()
            rid, cid, au = assembly.assemble(sys_.rows, sys_.cols, sys_.blocks)
            rec["t_ga"] = time.perf_counter() - t0
            cache[si] = {"asm": (rid, cid, au)}
        rid, cid, au = cache[si]["asm"]
        if ph in (None, "pa") or "M" not in cache[si]:
            t0 = time.perf_counter()
            M = mas.build_mas(mp, 32, 3, sys_.adj_ptr, sys_.adj, sys_.contacts, rid, cid, au)
            A = pcg.SymmetricMatrix(V, rid, cid, au)
            rec["t_pa"] = time.perf_counter() - t0
            cache[si].update(M=M, A=A)
        M, A = cache[si]["M"], cache[si]["A"]
        if ph in (None, "pcg"):
            k = spec["iters"]
            t0 = time.perf_counter()
            pcg.pcg(A, M, bs[0], fixed_iters=k)
            rec["t_iter"] = (time.perf_counter() - t0) / k
            rec["k"] = k
            if procs > 1:
                import multiprocessing as mpc

                # fork: the children inherit A, M and b; no GPU exists in this process
                _ORACLE_SHARED.update(A=A, M=M, b=bs)
                with mpc.get_context("fork").Pool(procs) as pool:
                    t0 = time.perf_counter()
                    pool.map(_oracle_pcg_iters, [(j, k) for j in range(procs)], chunksize=1)
                    rec["t_iter_par"] = (time.perf_counter() - t0) / k
                rec["procs"] = procs
        out.append(rec)
    print(json.dumps({"samples": out, "host": host_info()}))


def oracle_full_plain16(spec):
    """Worker: the oracle's complete Newton solve of the 16^3 plain system
    (assembly, 2-level MAS build, 4-RHS PCG to 1e-6), `reps` times, single
    thread; prints per-phase seconds and iteration counts (JSON)."""
    from oracle import assembly, mas, partition, pcg
    from synth.workloads import plain_small, rhs

    s_ = plain_small()
    V = s_.n_vertices
    mp, _ = partition.map_remap(partition.recursive_bisection(s_.X, 32), 32)
    b = rhs(3 * V, 4)
    out = []
    for _ in range(spec["reps"]):
        t0 = time.perf_counter()
        rid, cid, au = assembly.assemble(s_.rows, s_.cols, s_.blocks)
        t1 = time.perf_counter()
        M = mas.build_mas(mp, 32, 2, s_.adj_ptr, s_.adj, s_.contacts, rid, cid, au)
        A = pcg.SymmetricMatrix(V, rid, cid, au)
        t2 = time.perf_counter()
        _, it, _ = pcg.pcg(A, M, b, tol=1e-6)
        t3 = time.perf_counter()
        out.append({"t_ga": t1 - t0, "t_pa": t2 - t1, "t_pcg": t3 - t2, "iters": [int(v) for v in it]})
    print(json.dumps({"samples": out, "host": host_info()}))


def oracle_elastic_sample(spec):
    """Worker: the oracle's element Hessians (PSD projection by a numeric 9x9
    eigendecomposition, pullback, triplets with masses: elastic.system_triplets)
    and its energy and gradient on the first `tets` tets of the elastic scene,
    single thread; prints seconds (JSON)."""
    from oracle import elastic
    from synth.workloads import make_elastic_scene

    s_ = make_elastic_scene(spec["grid"], n_springs=0, omega=10.0, seed=spec["seed"])
    tets = s_.tets[: spec["tets"]]
    t0 = time.perf_counter()
    elastic.system_triplets(s_.X, s_.x, tets, spec["E"], spec["nu"], spec["rho"], spec["dt"])
    t1 = time.perf_counter()
    elastic.energy_and_gradient(s_.X, s_.x, tets, spec["E"], spec["nu"])
    t2 = time.perf_counter()
    print(json.dumps({"tets": int(len(tets)), "t_hessian": t1 - t0, "t_energy_gradient": t2 - t1,
                      "host": host_info()}))


def oracle_abd_sample(spec):
    """Worker: the oracle's complete differentiated solve (two-level ABD
    assembly, 3-level MAS build, forward PCG to 1e-6, adjoint PCG to 1e-6 for
    L = ||x - x_t||^2, dL/dH on the stored blocks) of a scene of the coupled
    recipe at spec["n"]^3 vertices, single thread; prints per-phase seconds,
    iteration counts and sizes (JSON)."""
    import numpy as np

    from oracle import adjoint, assembly, mas, partition, pcg
    from synth.abd import make_abd_scene

    n = spec["n"]
    frac = n ** 3 / 1e6
    s_ = make_abd_scene(n=n, n_bodies=max(4, round(2000 * frac)), n_contacts=round(500_000 * frac), seed=1005)
    mp, _ = partition.map_remap(partition.recursive_bisection(s_.X, 32), 32)
    rng = np.random.default_rng(2005)
    b = rng.normal(size=(1, 3 * s_.n_red))
    xt = rng.normal(size=(1, 3 * s_.n_red))
    t0 = time.perf_counter()
    rid, cid, au = assembly.assemble_abd(s_.rows, s_.cols, s_.blocks, s_.body_of_node, s_.xbar, s_.n_fem)
    t1 = time.perf_counter()
    M = mas.build_mas(mp, 32, 3, s_.adj_ptr, s_.adj, s_.contacts, rid, cid, au)
    A = pcg.SymmetricMatrix(s_.n_red, rid, cid, au)
    t2 = time.perf_counter()
    x, it, _ = pcg.pcg(A, M, b, tol=1e-6)
    t3 = time.perf_counter()
    lam, it_a, _ = pcg.pcg(A, M, 2.0 * (x - xt), tol=1e-6)
    adjoint.block_gradients(rid, cid, x.reshape(1, -1, 3), lam.reshape(1, -1, 3))
    t4 = time.perf_counter()
    print(json.dumps({"t_ga": t1 - t0, "t_pa": t2 - t1, "t_fwd": t3 - t2, "t_adj": t4 - t3,
                      "iters": [int(it[0]), int(it_a[0])], "inputs": int(s_.rows.size), "rows": int(s_.n_red),
                      "stored": int(rid.size), "host": host_info()}))


def run_oracle_sample(grid, Es, samples, iters=20, procs=1, cycle=False):
    env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1",
               CUDA_VISIBLE_DEVICES="")
    spec = json.dumps({"grid": grid, "Es": list(Es), "samples": samples, "iters": iters, "procs": procs,
                       "cycle": cycle})
    r = subprocess.run([sys.executable, os.path.abspath(__file__), "--oracle-sample", spec], env=env,
                       capture_output=True, text=True, timeout=3600)
    if r.returncode != 0:
        raise RuntimeError(r.stderr[-2000:])
    return json.loads(r.stdout.strip().splitlines()[-1])


def oracle_rates(t_ga, t_pa, t_iter, t_iter_par, iters):
    """Newton solves/s of the oracle for per-RHS PCG iteration counts `iters`:
    single thread T = T_ga + T_pa + sum_k iters_k T_iter (supplement Eq. 1);
    with the RHS in concurrent processes T = T_ga + T_pa + max_k iters_k
    T_iter_par (assembly and build stay single-threaded, as the oracle is)."""
    t1 = t_ga + t_pa + sum(iters) * t_iter
    tp = t_ga + t_pa + max(iters) * t_iter_par if t_iter_par else None
    return 1.0 / t1, (1.0 / tp if tp else None), t1, tp


# --------------------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        with open(self.path) as f:
            lines = f.readlines()
        os.unlink(self.path)
        return self.summarise(lines)

    @staticmethod
    def summarise(lines):
        """Median SM clock, maximum SM clock and the throttle reasons seen in
        nvidia-smi CSV lines of FIELDS (no header, no units); None if none parse."""
        rows = []
        for line in lines:
            parts = [x.strip() for x in line.split(",")]
            if len(parts) >= 9:
                rows.append(parts)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower().startswith("active")})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# --------------------------------------------------------------------------- workload on the GPU
def autotune_current(B, ctx):
    from paper_2411_06224_gb300 import autotune

    return autotune.current(ctx)


def make_workload(grid, nrhs, rank, Es=(1e5, 1e7, 1e9)):
    import numpy as np

    from synth.workloads import rhs, stiffness_sweep

    systems = stiffness_sweep(Es=tuple(Es), n=grid, seed=1002 + rank)
    b = rhs(3 * systems[0].n_vertices, nrhs, seed0=2000 + 100 * rank)
    return systems, np.ascontiguousarray(b)


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    return json.load(open(path)) if os.path.exists(path) else {}


def recorded_traffic(kernel, workload, table="dram_traffic.md"):
    """DRAM bytes per launch of `kernel` on `workload` as recorded from an ncu
    capture in profiles/dram_traffic.md (or the first value column of another
    table of the same layout), if the kernel's source file still has the hash
    recorded with it (else None: the kernel changed since)."""
    import hashlib

    path = os.path.join(ROOT, "profiles", table)
    if not os.path.exists(path):
        return None
    for ln in open(path):
        cells = [c.strip() for c in ln.strip().strip("|").split("|")]
        if len(cells) < 5 or cells[0] != kernel or cells[1] != workload:
            continue
        src = os.path.join(ROOT, cells[2])
        if not os.path.exists(src):
            return None
        if hashlib.sha256(open(src, "rb").read()).hexdigest()[:16] != cells[3]:
            return None
        return float(cells[4])
    return None


def kernel_lines(B, ctx, dev, clk, spmv, prec, nrhs, N, V, nnzb, ndom, mp, live, alone, workload=None):
    """Roofline lines of the level-0 MAS apply and the SpMV: algorithmic bytes
    (or operations) per launch over the mean CUDA-event launch time, `live`
    (launches, ms per class) inside the timed region and `alone` from a
    sequential per-class step."""
    import numpy as np
    import torch

    launches, kms = live
    launches_1, ms_1 = alone
    props = torch.cuda.get_device_properties(dev)
    sms = props.multi_processor_count
    sm_mhz_max = (clk or {}).get("sm_max_mhz") or 2070.0
    fp64_peak_tflops = sms * FP64_FMA_PER_CLK_PER_SM * 2 * sm_mhz_max * 1e6 / 1e12
    hbm = measured_peaks().get("hbm_gbs", 6800.0)
    ld = 3 * N
    n_dom0 = ndom
    real0 = np.bincount(mp // N, minlength=n_dom0)
    apply_flops = 2.0 * float(np.sum((3 * real0) ** 2)) * nrhs
    # the method's bytes: each inverse's packed lower triangle, read once per apply
    inv_bytes = (8 if prec == B.GS_PREC_FP64 else 4) * n_dom0 * ld * (ld + 1) // 2
    apply_bytes = inv_bytes + 2 * 8 * 3 * V * nrhs
    n_off = nnzb - V
    spmv_flops = nrhs * (18.0 * V + 36.0 * n_off)
    spmv_bytes = 76.0 * nnzb + 4.0 * (V + 1) + 2 * 8 * 3 * V * nrhs
    t_apply = kms[B.GS_K_MAS_APPLY_L0] / 1e3 / max(launches[B.GS_K_MAS_APPLY_L0], 1)
    t_spmv = kms[B.GS_K_SPMV] / 1e3 / max(launches[B.GS_K_SPMV], 1)
    t_apply_iso = ms_1[B.GS_K_MAS_APPLY_L0] / 1e3 / max(launches_1[B.GS_K_MAS_APPLY_L0], 1)
    t_spmv_iso = ms_1[B.GS_K_SPMV] / 1e3 / max(launches_1[B.GS_K_SPMV], 1)
    traffic_key = f"{workload},{nrhs}rhs" if workload else None

    def fp64_line(flops, nbytes, tsec, traffic):
        return {"bound": "alu", "achieved": flops / tsec / 1e12, "peak": fp64_peak_tflops, "unit": "TFLOP/s",
                "frac": flops / tsec / 1e12 / fp64_peak_tflops, "traffic": traffic,
                "hbm_gbs": nbytes / tsec / 1e9, "hbm_frac": nbytes / tsec / 1e9 / hbm,
                "flops_per_launch": flops, "bytes_per_launch": nbytes, "avg_launch_ms": tsec * 1e3}

    tune_tc = B.gs_tune_get(ctx, B.GS_TUNE_F64_TC)
    f64tc = (prec == B.GS_PREC_FP64 and nrhs <= 8 and ld % 16 == 0 and tune_tc in (1, 2, 3, 4))
    if f64tc:
        if tune_tc == 3:
            # the block lower triangle of every level-0 inverse as 8 base-128
            # digit bytes per entry (64 B per 8x8 core block) streams from HBM
            # once per apply, plus r read and z written (FP64)
            nb = ld // 8
            dig_bytes = 8 * 64 * (nb * (nb + 1) // 2) * n_dom0
            kname = "k_f64sym"
            kdesc = ("k_f64sym (level-0 MAS apply in FP64 accuracy from the symmetric inverses' block lower "
                     "triangles as base-128 digit bytes, expanded to BF16 in shared memory, on tcgen05, "
                     "+ prolongation)")
        else:
            # the 7 digit bytes per entry of every level-0 inverse
            dig_bytes = 7 * n_dom0 * ld * ld
            kname = "k_level0_f64tc"
            kdesc = ("k_level0_f64tc (level-0 MAS apply in FP64 accuracy from digit bytes by exact F16 digit "
                     "splitting on tcgen05, + prolongation)")
        tc_bytes = dig_bytes + 2 * 8 * 3 * V * nrhs
        traffic = recorded_traffic(kname, traffic_key) if traffic_key else None
        apply_line = {"bound": "hbm", "achieved": tc_bytes / t_apply / 1e9, "peak": hbm, "unit": "GB/s",
                      "frac": tc_bytes / t_apply / 1e9 / hbm, "traffic": traffic,
                      "method_bytes_frac": apply_bytes / t_apply / 1e9 / hbm,
                      "fp64_equivalent_tflops": apply_flops / t_apply / 1e12,
                      "fp64_equivalent_frac_of_fp64_peak": apply_flops / t_apply / 1e12 / fp64_peak_tflops,
                      "flops_per_launch": apply_flops, "bytes_per_launch": tc_bytes,
                      "method_bytes_per_launch": apply_bytes, "avg_launch_ms": t_apply * 1e3,
                      "kernel": kdesc}
        apply_iso_ach = tc_bytes / t_apply_iso / 1e9
    elif prec == B.GS_PREC_FP32 and nrhs <= 8:
        # FP32 inverses streamed as packed lower triangles (k_level0_f32)
        apply_line = {"bound": "hbm", "achieved": apply_bytes / t_apply / 1e9, "peak": hbm, "unit": "GB/s",
                      "frac": apply_bytes / t_apply / 1e9 / hbm, "traffic": None,
                      "flops_per_launch": apply_flops, "bytes_per_launch": apply_bytes,
                      "avg_launch_ms": t_apply * 1e3,
                      "kernel": "k_level0_f32 (level-0 MAS apply from packed FP32 lower triangles, + prolongation)"}
        apply_iso_ach = apply_bytes / t_apply_iso / 1e9
    else:
        apply_line = fp64_line(apply_flops, apply_bytes, t_apply, None)
        apply_line["kernel"] = (f"k_domain_product<double,{B.gs_tune_get(ctx, B.GS_TUNE_APPLY_RHS)},1> "
                                "(level-0 MAS apply + prolongation)")
        apply_iso_ach = apply_flops / t_apply_iso / 1e12
    apply_line["isolated"] = {"avg_launch_ms": t_apply_iso * 1e3, "achieved": apply_iso_ach,
                              "frac": apply_iso_ach / apply_line["peak"]}
    spmv_ws = spmv in ("row", "ff") and B.gs_tune_get(ctx, B.GS_TUNE_SPMV_WS) == 1
    if spmv == "ff":
        # float-float on the FP32 units: 12 FP32 instructions per term (exact
        # product, two-sum, small parts), 9 terms per block use and RHS, one use
        # per diagonal block and two per off-diagonal block
        ff_inst = nrhs * 9 * 12.0 * (V + 2.0 * n_off)
        fp32_peak = sms * 128 * sm_mhz_max * 1e6 / 1e12  # T FP32 instructions/s
        kname = "k_pcg_spmv" if nrhs <= 8 else ("k_spmv_ff_ws" if spmv_ws else "k_spmv_ff_row")
        spmv_line = {"bound": "alu", "achieved": ff_inst / t_spmv / 1e12, "peak": fp32_peak,
                     "unit": "T FP32 instructions/s", "frac": ff_inst / t_spmv / 1e12 / fp32_peak,
                     "traffic": (recorded_traffic(kname, traffic_key if kname == "k_pcg_spmv" else
                                                  f"{traffic_key},ff_rhs{B.gs_tune_get(ctx, B.GS_TUNE_SPMV_FF_RHS)}")
                                 if traffic_key else None),
                     "hbm_gbs": spmv_bytes / t_spmv / 1e9, "hbm_frac": spmv_bytes / t_spmv / 1e9 / hbm,
                     "fp64_equivalent_tflops": spmv_flops / t_spmv / 1e12,
                     "fp64_equivalent_frac_of_fp64_peak": spmv_flops / t_spmv / 1e12 / fp64_peak_tflops,
                     "instructions_per_launch": ff_inst, "flops_per_launch": spmv_flops,
                     "bytes_per_launch": spmv_bytes, "avg_launch_ms": t_spmv * 1e3, "kernel": kname}
        spmv_line["isolated"] = {"avg_launch_ms": t_spmv_iso * 1e3, "achieved": ff_inst / t_spmv_iso / 1e12,
                                 "frac": ff_inst / t_spmv_iso / 1e12 / fp32_peak,
                                 "hbm_frac": spmv_bytes / t_spmv_iso / 1e9 / hbm}
    else:
        kname = ("k_pcg_spmv" if nrhs <= 8 and spmv != "srbk" else
                 "k_spmv_row_ws" if spmv_ws else f"k_spmv_{spmv}")
        spmv_line = fp64_line(spmv_flops, spmv_bytes, t_spmv,
                              recorded_traffic(kname, traffic_key) if traffic_key else None)
        spmv_line["kernel"] = kname
        spmv_line["isolated"] = {"avg_launch_ms": t_spmv_iso * 1e3, "achieved": spmv_flops / t_spmv_iso / 1e12,
                                 "frac": spmv_flops / t_spmv_iso / 1e12 / fp64_peak_tflops}
    return apply_line, spmv_line


def config1_form(args, B, dev, variant, clk):
    """The plain FP64 solve on the 16^3 cube (4,096 vertices, 2,000 random
    contacts, E = 1e5, 4 RHS, 2-level MAS with 32-node domains, tol 1e-6):
    Newton solves/s through the whole path on one stream, the kernels'
    roofline lines, and the oracle's complete solve timed on the host."""
    import numpy as np
    import torch

    from synth.workloads import plain_small, rhs

    s_ = plain_small()
    V, N, L, K = s_.n_vertices, 32, 2, 4
    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device=dev)
    mp, nd = B.gs_partition(s_.X, N)
    d = dict(rows=t(s_.rows, torch.int32), cols=t(s_.cols, torch.int32),
             blocks=t(s_.blocks.reshape(-1, 3, 3), torch.float64), map=t(mp, torch.int32),
             adj_ptr=t(s_.adj_ptr, torch.int32), adj=t(s_.adj, torch.int32), contacts=t(s_.contacts, torch.int32))
    b = t(rhs(3 * V, K), torch.float64)
    x = torch.zeros_like(b)
    ctx = B.gs_create(dev.index or 0, torch.cuda.current_stream())

    def solve():
        mat = B.gs_assemble(ctx, V, d["rows"], d["cols"], d["blocks"])
        mas = B.gs_build_mas(ctx, mat, d["map"], nd, d["adj_ptr"], d["adj"], d["contacts"], domain_size=N,
                             max_levels=L)
        it, _, _ = B.gs_pcg_solve(ctx, mat, mas, b, x, nrhs=K, tol=TOL, max_iter=20000, variant=variant)
        info = B.gs_mat_info(mat)[1]
        B.gs_mas_destroy(mas)
        B.gs_mat_destroy(mat)
        return it, info

    try:
        for _ in range(max(args.warmup, 3)):
            it, nnzb = solve()
        B.gs_profile_begin(ctx, range(B.GS_K_COUNT))
        solve()
        alone = B.gs_profile_end(ctx)
        steps = 20
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        B.gs_profile_begin(ctx, [B.GS_K_MAS_APPLY_L0, B.GS_K_SPMV])
        e0.record()
        for _ in range(steps):
            it, _ = solve()
        e1.record()
        torch.cuda.synchronize()
        live = B.gs_profile_end(ctx)
        sec = e0.elapsed_time(e1) / 1e3
        apply_line, spmv_line = kernel_lines(B, ctx, dev, clk, "ff" if variant == B.GS_SPMV_ROW_FF else "row",
                                             B.GS_PREC_FP64, K, N, V, nnzb, nd, mp, live, alone)
        dominant = apply_line if live[1][B.GS_K_MAS_APPLY_L0] >= live[1][B.GS_K_SPMV] else spmv_line
        out = {"workload": "tet cube 16^3 (4096 vertices), E=1e5, 2000 random contacts, 4 RHS, 2-level MAS N=32, "
                           "PCG tol 1e-6, one stream", "value": steps / sec, "unit": "Newton solves/s",
                "ms_per_solve": sec / steps * 1e3, "steps": steps, "pcg_iterations": [int(v) for v in it],
                "roofline": dominant, "kernels": {"mas_apply_l0": apply_line, "spmv": spmv_line},
                "phase_ms_one_solve": {B.K_NAMES[k]: float(alone[1][k]) for k in range(B.GS_K_COUNT)}}
    finally:
        B.gs_destroy(ctx)
    if not args.no_cpu_baseline:
        try:
            env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1",
                       CUDA_VISIBLE_DEVICES="")
            r = subprocess.run([sys.executable, os.path.abspath(__file__), "--oracle-sample",
                                json.dumps({"kind": "plain16", "reps": 3})], env=env, capture_output=True, text=True,
                               timeout=1800)
            res = json.loads(r.stdout.strip().splitlines()[-1])
            smp = res["samples"][-1]
            tot = smp["t_ga"] + smp["t_pa"] + smp["t_pcg"]
            out["cpu_baseline"] = {
                "value": 1.0 / tot, "unit": "Newton solves/s", "cores": 1, "kind": "oracle",
                "sample": (f"the FP64 numpy/scipy oracle's complete solve of this system on one host core "
                           f"({res['host']['cpu_model']}): assembly {smp['t_ga']:.3f} s, 2-level MAS build "
                           f"{smp['t_pa']:.3f} s, PCG {smp['t_pcg']:.3f} s (iterations {smp['iters']}); last of 3"),
                "host": res["host"]}
        except Exception as e:  # noqa: BLE001
            out["cpu_baseline"] = {"value": None, "error": str(e)[:300]}
    return out


def abd_form(args, B, dev, clk):
    """The differentiation form on the coupled scene: the 100^3 tet cube
    (1M vertices, E = 1e6) with 2,000 affine bodies and 500k contact pairs
    (51M full-space input triplets).  One step = two-level hash assembly
    (gs_assemble_abd), MAS build with FP32 inverses (N = 32, 3 levels; the
    partition once per mesh), forward PCG to 1e-6 (FP64 PCG and reductions,
    float-float SpMV), the adjoint solve for L = ||x - x_t||^2 to 1e-6 and
    dL/dH on the stored blocks (gs_adjoint), inputs resident in HBM, one
    stream.  `value`: differentiated solves (forward + adjoint) per second."""
    import numpy as np
    import torch

    from synth.abd import make_abd_scene

    t_gen = time.time()
    # the bodies, contacts and graph on the host; the FEM part's stable
    # Neo-Hookean element blocks and masses (same positions, same recipe)
    # from the library's element kernel, untimed input generation
    s_ = make_abd_scene(fem_blocks=False)
    N, L = 32, 3
    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device=dev)
    ctx = B.gs_create(dev.index or 0, torch.cuda.current_stream())
    p_ = s_.params
    fem = B.gs_fem_create(ctx, t(s_.X[: s_.n_fem], torch.float64), t(s_.fem_tets, torch.int32), p_["E"], 0.4,
                          p_["rho"], p_["dt"])
    n_fem_trip = 10 * s_.fem_tets.shape[0] + s_.n_fem
    rf, cf, bf = B.gs_fem_triplets(ctx, fem, t(s_.fem_x, torch.float64), n_fem_trip)
    B.gs_fem_destroy(fem)
    rows = torch.cat([rf, t(s_.rows, torch.int32)])
    cols = torch.cat([cf, t(s_.cols, torch.int32)])
    blocks = torch.cat([bf, t(s_.blocks, torch.float64)])
    del rf, cf, bf
    # emission order of a parallel element loop: one seeded shuffle of all inputs
    perm = torch.randperm(rows.numel(), generator=torch.Generator(device=dev).manual_seed(1005 + 7919), device=dev)
    rows, cols, blocks = rows[perm].contiguous(), cols[perm].contiguous(), blocks[perm].contiguous()
    del perm
    torch.cuda.synchronize()
    t_gen = time.time() - t_gen
    mp, nd = B.gs_partition(s_.X, N)
    d = dict(rows=rows, cols=cols, blocks=blocks,
             body=t(s_.body_of_node, torch.int32), xbar=t(s_.xbar, torch.float64), map=t(mp, torch.int32),
             adj_ptr=t(s_.adj_ptr, torch.int32), adj=t(s_.adj, torch.int32), contacts=t(s_.contacts, torch.int32))
    n_inputs = int(rows.numel())
    n = s_.n_red
    rng = np.random.default_rng(2005)
    b = t(rng.normal(size=(1, 3 * n)), torch.float64)
    xt = t(rng.normal(size=(1, 3 * n)), torch.float64)
    x = torch.zeros_like(b)
    g = torch.empty_like(b)
    variant = B.GS_SPMV_ROW_FF
    buf = {}

    def step():
        mat = B.gs_assemble_abd(ctx, s_.n_nodes, s_.n_fem, s_.n_bodies, d["body"], d["xbar"], d["rows"], d["cols"],
                                d["blocks"])
        M = B.gs_build_mas(ctx, mat, d["map"], nd, d["adj_ptr"], d["adj"], d["contacts"], domain_size=N,
                           max_levels=L, precision=B.GS_PREC_FP32)
        nnzb = B.gs_mat_info(mat)[1]
        if "dLdH" not in buf or buf["dLdH"].shape[0] != nnzb:
            buf["dLdH"] = torch.empty((nnzb, 3, 3), dtype=torch.float64, device=dev)
        x.zero_()
        it, _, _ = B.gs_pcg_solve(ctx, mat, M, b, x, nrhs=1, tol=TOL, max_iter=20000, variant=variant)
        torch.sub(x, xt, out=g).mul_(2.0)  # dL/dx of the caller's loss
        lam, it_a = B.gs_adjoint(ctx, mat, M, x, g, nrhs=1, tol=TOL, dLdH=buf["dLdH"])
        B.gs_mas_destroy(M)
        B.gs_mat_destroy(mat)
        return [int(it[0]), int(it_a[0])], nnzb

    try:
        for _ in range(max(args.warmup, 3)):
            its, nnzb = step()
        B.gs_profile_begin(ctx, range(B.GS_K_COUNT))
        step()
        alone = B.gs_profile_end(ctx)
        steps = max(args.abd_steps, 1)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        B.gs_profile_begin(ctx, [B.GS_K_MAS_APPLY_L0, B.GS_K_SPMV])
        e0.record()
        for _ in range(steps):
            its, _ = step()
        e1.record()
        torch.cuda.synchronize()
        live = B.gs_profile_end(ctx)
        sec = e0.elapsed_time(e1) / 1e3
        apply_line, spmv_line = kernel_lines(B, ctx, dev, clk, "ff", B.GS_PREC_FP32, 1, N, n, nnzb, nd, mp, live,
                                             alone)
        dominant = apply_line if live[1][B.GS_K_MAS_APPLY_L0] >= live[1][B.GS_K_SPMV] else spmv_line
        out = {"workload": "tet cube 100^3 (1M vertices, E=1e6) + 2000 affine bodies + 500k contact pairs, "
                           "two-level ABD assembly, 3-level MAS N=32 with FP32 inverses, forward PCG + adjoint "
                           "(L = ||x - x_t||^2) to 1e-6, dL/dH on the pattern, one stream",
               "value": steps / sec, "unit": "differentiated solves/s (forward + adjoint)",
               "ms_per_step": sec / steps * 1e3, "steps": steps, "pcg_iterations": {"forward": its[0],
                                                                                 "adjoint": its[1]},
               "reduced_rows": n, "stored_blocks": nnzb, "input_triplets": n_inputs,
               "input_generation_s": t_gen, "roofline": dominant,
               "kernels": {"mas_apply_l0": apply_line, "spmv": spmv_line},
               "phase_ms_one_step": {B.K_NAMES[k]: float(alone[1][k]) for k in range(B.GS_K_COUNT)}}
    finally:
        B.gs_destroy(ctx)
    if not args.no_cpu_baseline:
        try:
            env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1",
                       CUDA_VISIBLE_DEVICES="")
            r = subprocess.run([sys.executable, os.path.abspath(__file__), "--oracle-sample",
                                json.dumps({"kind": "abd", "n": 32})], env=env, capture_output=True, text=True,
                               timeout=1800)
            res = json.loads(r.stdout.strip().splitlines()[-1])
            # per-unit rates of the sample applied to the full scene: assembly per
            # input triplet, build per reduced row, PCG per stored block and iteration
            t_ga = res["t_ga"] * n_inputs / res["inputs"]
            t_pa = res["t_pa"] * n / res["rows"]
            per_it = (res["t_fwd"] + res["t_adj"]) / sum(res["iters"]) * nnzb / res["stored"]
            tot = t_ga + t_pa + per_it * sum(its)
            out["cpu_baseline"] = {
                "value": 1.0 / tot, "unit": "differentiated solves/s (forward + adjoint)", "cores": 1,
                "kind": "oracle",
                "sample": (f"the FP64 numpy/scipy oracle's complete differentiated solve on one host core "
                           f"({res['host']['cpu_model']}) of the same recipe at 32^3 vertices "
                           f"({res['rows']} reduced rows, {res['stored']} stored blocks): assembly "
                           f"{res['t_ga']:.2f} s, MAS build {res['t_pa']:.2f} s, forward + adjoint PCG "
                           f"{res['t_fwd'] + res['t_adj']:.2f} s ({res['iters']} iterations); scaled to this scene "
                           f"per input triplet, reduced row and stored block x iteration (the GPU's counts)"),
                "sample_rate": 1.0 / (res["t_ga"] + res["t_pa"] + res["t_fwd"] + res["t_adj"]),
                "host": res["host"]}
        except Exception as e:  # noqa: BLE001
            out["cpu_baseline"] = {"value": None, "error": str(e)[:300]}
    return out


# FP64 operations per element of the cloth kernels, counted from their source
# (FMA = 2; square roots and divisions as 1): triangle = F (24), two
# directions (norm, coefficients, strain limit, 6 entries of the symmetric
# block: 57 each), the shear scale and cross block (14), H_01 + H_01^T (6),
# 3 symmetric vertex blocks (3 weight products, 6 entries of 5: 33 each) and
# 3 others (4 weight products, 9 entries of 7: 67 each); hinge = edge vectors,
# normals, norms, projections and gradients (94), 2 k_b g (13) and 10 blocks
# of 9 products
CLOTH_FLOP_TRI = 24 + 2 * 57 + 14 + 6 + 3 * 33 + 3 * 67
CLOTH_FLOP_HINGE = 94 + 13 + 10 * 9
# FP64 instructions (DFMA + DMUL + DADD, per thread) per element as the
# hardware counters show them for k_cloth_membrane and k_cloth_bending on the
# 512^2 sheet (square roots and divisions expand into several FP64
# instructions; the source count above takes them as one).  The FP64 pipe is
# the bound: it issues FP64_FMA_PER_CLK_PER_SM thread instructions per clock
# per SM whatever the instruction.
CLOTH_FP64_INST_TRI = 300.0
CLOTH_FP64_INST_HINGE = 181.0


def cloth_element_line(args, B, dev, stream, clk):
    """Device cloth element Hessians (gs_cloth_triplets) on the bench's sheet:
    elements per second, the FP64 roofline of the launch sequence, and the
    oracle's per-element rate on a 48 x 48 sample of the same recipe."""
    import numpy as np
    import torch

    from synth.cloth import hinges, sheet

    n = args.cloth
    X, tris = sheet(n)
    hg = hinges(tris)
    rng = np.random.default_rng(1003)
    h = 1.0 / (n - 1)
    sh = rng.uniform(0.0, 0.1)
    x = X @ np.array([[1.02, sh, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]]).T + rng.normal(0.0, 0.01 * h, X.shape)
    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device=dev)
    ctx = B.gs_create(dev.index or 0, stream)
    try:
        c = B.gs_cloth_create(ctx, t(X, torch.float64), t(tris, torch.int32), t(hg, torch.int32), 1e8, 0.05e6, 1e-3,
                              200.0, 0.01)
        xd = t(x, torch.float64)
        nt = B.gs_cloth_info(c)
        rows = torch.empty(nt, dtype=torch.int32, device=dev)
        cols = torch.empty(nt, dtype=torch.int32, device=dev)
        blocks = torch.empty((nt, 3, 3), dtype=torch.float64, device=dev)
        call = lambda: B.lib().gs_cloth_triplets(ctx, c, ctypes_ptr(xd), ctypes_ptr(rows), ctypes_ptr(cols),
                                                 ctypes_ptr(blocks))
        for _ in range(3):
            call()
        reps = 10
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            call()
        e1.record(stream)
        torch.cuda.synchronize()
        sec = e0.elapsed_time(e1) / 1e3 / reps
        B.gs_cloth_destroy(c)
    finally:
        B.gs_destroy(ctx)
    T, H, V = len(tris), len(hg), X.shape[0]
    props = torch.cuda.get_device_properties(dev)
    sm_mhz = (clk or {}).get("sm_max_mhz") or 2070.0
    inst_peak = props.multi_processor_count * FP64_FMA_PER_CLK_PER_SM * sm_mhz * 1e6 / 1e9  # G instr/s
    inst = CLOTH_FP64_INST_TRI * T + CLOTH_FP64_INST_HINGE * H
    tm, tb = (recorded_traffic(k, f"cloth{n}") for k in ("k_cloth_membrane", "k_cloth_bending"))
    traffic = tm + tb if tm is not None and tb is not None else None
    flops = CLOTH_FLOP_TRI * T + CLOTH_FLOP_HINGE * H
    nbytes = T * (3 * 24 + 48 + 8 + 12 + 6 * 80) + H * (4 * 24 + 16 + 8 + 10 * 80) + V * (8 + 80)
    out = {"workload": f"cloth {n}x{n}: {T} triangles, {H} hinges, {V} vertices -> {nt} triplets",
           "value": (T + H) / sec, "unit": "elements/s (triangles + hinges)", "ms_per_launch_sequence": sec * 1e3,
           "roofline": {"bound": "alu", "achieved": inst / sec / 1e9, "peak": inst_peak,
                        "unit": "G FP64 instr/s", "frac": inst / sec / 1e9 / inst_peak, "traffic": traffic,
                        "traffic_kernels": "k_cloth_membrane + k_cloth_bending (the mass-block kernel not captured)",
                        "fp64_instr_per_launch": inst, "source_flops_per_launch": flops,
                        "source_tflops": flops / sec / 1e12, "bytes_per_launch": nbytes,
                        "hbm_gbs": nbytes / sec / 1e9,
                        "kernel": "k_cloth_membrane + k_cloth_bending + k_cloth_mass_blocks (FP64 pipe)"}}
    if not args.no_cpu_baseline:
        from oracle import cloth as ocloth

        Xs, ts = sheet(48)
        hs = hinges(ts)
        xs = Xs @ np.array([[1.02, sh, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]]).T
        t0 = time.perf_counter()
        ocloth.cloth_triplets(Xs, xs, ts, hs, 1e8, 0.05e6, 1e-3, 200.0, 0.01)
        dt_ = time.perf_counter() - t0
        out["cpu_baseline"] = {"value": (len(ts) + len(hs)) / dt_, "unit": "elements/s (triangles + hinges)",
                               "cores": 1, "kind": "oracle",
                               "sample": f"oracle.cloth.cloth_triplets on a 48x48 sheet of the same recipe "
                                         f"({len(ts)} triangles, {len(hs)} hinges), numpy, one process"}
    return out


def ctypes_ptr(tensor):
    import ctypes

    return ctypes.c_void_p(tensor.data_ptr())


def element_probe(args):
    """The Newton form's elastic cube at --element-probe vertices per edge:
    body created (element keys sorted), springs set, Hessian assembled at the
    start positions, then refilled --refills times; prints the counts."""
    import numpy as np
    import torch

    from paper_2411_06224_gb300.build import build
    from synth.workloads import make_elastic_scene

    build()
    from paper_2411_06224_gb300 import binding as B

    n = args.element_probe
    s_ = make_elastic_scene(n, n_springs=max(1, 200_000 * n ** 3 // 64 ** 3), omega=10.0, seed=3000 + n)
    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    ctx = B.gs_create(0)
    f = B.gs_fem_create(ctx, t(s_.X, torch.float64), t(s_.tets, torch.int32), 1e5, 0.4, 1000.0, 0.01)
    B.gs_fem_set_springs(ctx, f, t(s_.pairs, torch.int32), t(s_.K, torch.float64), t(s_.rest, torch.float64))
    x0 = t(s_.x, torch.float64)
    m = B.gs_fem_assemble(ctx, f, x0)
    for _ in range(args.refills):
        B.gs_fem_refill(ctx, f, x0, m)
    torch.cuda.synchronize()
    print(json.dumps({"tets": int(len(s_.tets)), "vertices": s_.n_vertices, "stored_blocks": B.gs_fem_info(f)[0],
                      "refills": args.refills}))
    B.gs_mat_destroy(m)
    B.gs_fem_destroy(f)
    B.gs_destroy(ctx)


def cloth_probe(args):
    """The stiff-cloth sheet of the precision form at --cloth-probe vertices per
    edge: rest data once, then the element Hessians --refills times; prints
    the counts."""
    import numpy as np
    import torch

    from paper_2411_06224_gb300.build import build
    from synth.cloth import hinges, sheet

    build()
    from paper_2411_06224_gb300 import binding as B

    n = args.cloth_probe
    X, tris = sheet(n)
    hg = hinges(tris)
    rng = np.random.default_rng(1003)
    h = 1.0 / (n - 1)
    sh = rng.uniform(0.0, 0.1)
    x = X @ np.array([[1.02, sh, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]]).T + rng.normal(0.0, 0.01 * h, X.shape)
    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    stream = torch.cuda.Stream()
    ctx = B.gs_create(0, stream)
    c = B.gs_cloth_create(ctx, t(X, torch.float64), t(tris, torch.int32), t(hg, torch.int32), 1e8, 0.05e6, 1e-3,
                          200.0, 0.01)
    xd = t(x, torch.float64)
    B.gs_cloth_triplets(ctx, c, xd)
    nt = B.gs_cloth_info(c)
    rows = torch.empty(nt, dtype=torch.int32, device="cuda")
    cols = torch.empty(nt, dtype=torch.int32, device="cuda")
    blocks = torch.empty((nt, 3, 3), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.refills):
        B.lib().gs_cloth_triplets(ctx, c, ctypes_ptr(xd), ctypes_ptr(rows), ctypes_ptr(cols), ctypes_ptr(blocks))
    e1.record(stream)
    torch.cuda.synchronize()
    print(json.dumps({"triangles": int(len(tris)), "hinges": int(len(hg)), "triplets": nt,
                      "launch_sequences": args.refills,
                      "ms_per_launch_sequence": e0.elapsed_time(e1) / max(args.refills, 1)}))
    B.gs_cloth_destroy(c)
    B.gs_destroy(ctx)


def newton_form(args, B, dev, clk):
    """Newton's method on the implicit-Euler step of the tet cube (stable
    Neo-Hookean, E = 1e5, nu = 0.4, rho = 1000, dt = 0.01; springs on random
    vertex pairs standing in for contacts): element Hessians on the device,
    values reduced through the pattern sorted once, MAS built at the first
    step and refreshed after, MAS-PCG to 1e-6 per step, Armijo backtracking.
    Also: the numeric assembly (no sort) against re-sorting every step, and
    the element-Hessian kernel's roofline line."""
    import numpy as np
    import torch

    from synth.workloads import make_elastic_scene

    E_, NU, RHO, DT = 1e5, 0.4, 1000.0, 0.01
    n_springs = max(1, 200_000 * args.grid ** 3 // 64 ** 3)
    seed = 3000 + args.grid
    s_ = make_elastic_scene(args.grid, E=E_, n_springs=n_springs, omega=10.0, seed=seed)
    V, T = s_.n_vertices, len(s_.tets)
    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device=dev)
    X, tets, x0, xt = t(s_.X, torch.float64), t(s_.tets, torch.int32), t(s_.x, torch.float64), t(s_.xt, torch.float64)
    pairs, K, rest = t(s_.pairs, torch.int32), t(s_.K, torch.float64), t(s_.rest, torch.float64)
    ptr, adj = t(s_.adj_ptr, torch.int32), t(s_.adj, torch.int32)
    stream = torch.cuda.current_stream()
    ctx = B.gs_create(dev.index or 0, stream)
    ev = lambda: torch.cuda.Event(enable_timing=True)
    out = {"workload": f"tet cube {args.grid}^3 ({V} vertices, {T} tets), SNH E=1e5 nu=0.4, rho=1000, dt=0.01, "
                       f"{n_springs} springs k n n^T (k 1e2-1e4) on random vertex pairs, rotation 10 rad/s per axis; "
                       "Newton tol |d|_inf <= 1e-3 dt, PCG tol 1e-6, FP64 MAS N=32, 3 levels, float-float SpMV"}
    f = None
    try:
        torch.cuda.synchronize()
        a, b_ = ev(), ev()
        a.record(stream)
        f = B.gs_fem_create(ctx, X, tets, E_, NU, RHO, DT)
        B.gs_fem_set_springs(ctx, f, pairs, K, rest)
        b_.record(stream)
        torch.cuda.synchronize()
        U, Ue, _, _ = B.gs_fem_info(f)
        out["symbolic_ms"] = a.elapsed_time(b_)
        out["stored_blocks"], out["element_stored_blocks"] = U, Ue
        # numeric assembly through the fixed pattern vs a full re-sort of the same triplets
        m = B.gs_fem_assemble(ctx, f, x0)
        reps = 5
        for _ in range(2):
            B.gs_fem_refill(ctx, f, x0, m)
        torch.cuda.synchronize()
        B.gs_profile_begin(ctx, [B.GS_K_ELEMENT, B.GS_K_ASSEMBLE])
        a.record(stream)
        for _ in range(reps):
            B.gs_fem_refill(ctx, f, x0, m)
        b_.record(stream)
        torch.cuda.synchronize()
        launches, kms = B.gs_profile_end(ctx)
        ms_refill = a.elapsed_time(b_) / reps
        n_in = 10 * T + V + 3 * n_springs
        r, c, bl = B.gs_fem_triplets(ctx, f, x0, n_in)
        m2 = B.gs_assemble(ctx, V, r, c, bl)
        B.gs_mat_destroy(m2)
        torch.cuda.synchronize()
        a.record(stream)
        for _ in range(reps):
            r, c, bl = B.gs_fem_triplets(ctx, f, x0, n_in)
            m2 = B.gs_assemble(ctx, V, r, c, bl)
            B.gs_mat_destroy(m2)
        b_.record(stream)
        torch.cuda.synchronize()
        ms_resort = a.elapsed_time(b_) / reps
        del r, c, bl
        B.gs_mat_destroy(m)
        n_el = int(max(launches[B.GS_K_ELEMENT] // reps, 1))
        t_hess = kms[B.GS_K_ELEMENT] / 1e3 / reps  # both kernels of one refill
        props = torch.cuda.get_device_properties(dev)
        sm_mhz_max = (clk or {}).get("sm_max_mhz") or 2070.0
        fp64_peak = props.multi_processor_count * FP64_FMA_PER_CLK_PER_SM * 2 * sm_mhz_max * 1e6 / 1e12
        hbm = measured_peaks().get("hbm_gbs", 6800.0)
        # algorithmic bytes per tet: 4 x 24 B of x gathered, 96 B w, 8 B vol, 16 B tets read; 10 x 72 B written
        el_bytes = T * (96 + 96 + 8 + 16 + 720) + V * 80
        wl = f"tet{args.grid}"
        flops = recorded_traffic("k_element_hessians", wl, table="fp64_ops.md")
        line = {"bound": "alu", "unit": "TFLOP/s", "peak": fp64_peak,
                "achieved": flops / t_hess / 1e12 if flops else None,
                "frac": flops / t_hess / 1e12 / fp64_peak if flops else None,
                "traffic": recorded_traffic("k_element_hessians", wl),
                "flops_per_launch": flops, "bytes_per_launch": el_bytes,
                "hbm_gbs": el_bytes / t_hess / 1e9, "hbm_frac": el_bytes / t_hess / 1e9 / hbm,
                "avg_launch_ms": t_hess * 1e3, "tets_per_s": T / t_hess, "launches_per_refill": n_el,
                "kernel": "k_element_hessians (SNH, analytic-eigensystem PSD projection, pullback; FP64) + k_mass_blocks",
                "flops_source": "FP64 operations per launch (2 per DFMA) from an ncu capture, profiles/fp64_ops.md"}
        out["kernels"] = {"element_hessians": line}
        out["assembly"] = {"ms_numeric_refill": ms_refill, "ms_resort_every_step": ms_resort,
                           "speedup": ms_resort / ms_refill,
                           "ms_refill_element_kernels": kms[B.GS_K_ELEMENT] / reps,
                           "ms_refill_reduction": kms[B.GS_K_ASSEMBLE] / reps,
                           "resort": "gs_fem_triplets (same element kernel, triplets copied out) + gs_assemble "
                                     "(inputs counted and scattered by row, rows sorted, row reduction)"}
        # the Newton loop
        def newton_run():
            x = x0.clone()
            st, en, status = B.gs_fem_newton(ctx, f, xt, x, ptr, adj, tol=1e-3, max_newton=50, pcg_tol=TOL,
                                             pcg_max_iter=20000, spmv_variant=B.GS_SPMV_ROW_FF, domain_size=32,
                                             max_levels=3, raise_on_maxiter=False)
            return st, en, status

        newton_run()  # warm-up
        torch.cuda.synchronize()
        a.record(stream)
        st, en, status = newton_run()
        b_.record(stream)
        torch.cuda.synchronize()
        sec = a.elapsed_time(b_) / 1e3
        out.update({"value": 1.0 / sec, "unit": "Newton solves/s (complete implicit steps)",
                    "ms_per_solve": sec * 1e3, "newton_steps": st["iterations"],
                    "newton_steps_per_s": st["iterations"] / sec, "converged": st["converged"],
                    "status": int(status), "pcg_iterations_total": st["pcg_iterations"],
                    "line_search_halvings": st["halvings"], "energy": [float(e) for e in en],
                    "phase_ms": st["ms"]})
    finally:
        if f is not None:
            B.gs_fem_destroy(f)
        B.gs_destroy(ctx)
    if not args.no_cpu_baseline:
        try:
            k = min(T, 20000)
            env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1",
                       CUDA_VISIBLE_DEVICES="")
            spec = {"kind": "elastic", "grid": args.grid, "seed": seed, "tets": k, "E": E_, "nu": NU, "rho": RHO,
                    "dt": DT}
            r_ = subprocess.run([sys.executable, os.path.abspath(__file__), "--oracle-sample", json.dumps(spec)],
                                env=env, capture_output=True, text=True, timeout=1800)
            res = json.loads(r_.stdout.strip().splitlines()[-1])
            rate = res["tets"] / res["t_hessian"]
            out["kernels"]["element_hessians"]["cpu_baseline"] = {
                "value": rate, "unit": "element Hessians/s", "cores": 1, "kind": "oracle",
                "sample": (f"oracle elastic.system_triplets on the first {res['tets']} tets of this scene, one host "
                           f"core ({res['host']['cpu_model']}): {res['t_hessian']:.2f} s; energy and gradient "
                           f"{res['t_energy_gradient']:.2f} s"),
                "device_ratio": (T / t_hess) / rate}
        except Exception as e:  # noqa: BLE001
            out["kernels"]["element_hessians"]["cpu_baseline"] = {"value": None, "error": str(e)[:300]}
    return out


def main():
    args = parse()
    if args.oracle_sample:
        spec = json.loads(args.oracle_sample)
        if spec.get("kind") == "plain16":
            oracle_full_plain16(spec)
        elif spec.get("kind") == "elastic":
            oracle_elastic_sample(spec)
        elif spec.get("kind") == "abd":
            oracle_abd_sample(spec)
        else:
            oracle_sample(spec)
        return
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        return reference_arm(args, rank, world)
    if args.micro:
        return micro(args)
    if args.element_probe:
        return element_probe(args)
    if args.cloth_probe:
        return cloth_probe(args)

    import numpy as np
    import torch
    import torch.distributed as dist

    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl")
    from paper_2411_06224_gb300.build import build

    build()
    from paper_2411_06224_gb300 import binding as B

    dev = torch.device("cuda", local)
    systems, b_host = make_workload(args.grid, args.nrhs, rank, Es=[float(e) for e in args.sweep.split(",")])
    V = systems[0].n_vertices
    N, L = 32, 3
    prec = {"fp64": B.GS_PREC_FP64, "fp32": B.GS_PREC_FP32, "bf16": B.GS_PREC_BF16}[args.precision]
    variant = {"row": B.GS_SPMV_ROW, "srbk": B.GS_SPMV_SRBK, "ff": B.GS_SPMV_ROW_FF}[args.spmv]
    mp, ndom = B.gs_partition(systems[0].X, N)  # once per mesh, before timing
    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device=dev)
    shared = dict(map=t(mp, torch.int32), adj_ptr=t(systems[0].adj_ptr, torch.int32), adj=t(systems[0].adj, torch.int32),
                  contacts=t(systems[0].contacts, torch.int32))
    dsys = [dict(rows=t(s.rows, torch.int32), cols=t(s.cols, torch.int32), blocks=t(s.blocks.reshape(-1, 3, 3), torch.float64),
                 E=s.params["E"]) for s in systems]
    b = t(b_host, torch.float64)
    x = torch.zeros_like(b)
    stream = torch.cuda.current_stream()
    ctx = B.gs_create(local, stream)

    def solve_one(rows, cols, blocks, bb, xx, c=None):
        c = c or ctx
        mat = B.gs_assemble(c, V, rows, cols, blocks)
        mas = B.gs_build_mas(c, mat, shared["map"], ndom, shared["adj_ptr"], shared["adj"], shared["contacts"],
                             domain_size=N, max_levels=L, precision=prec)
        it, rel, _ = B.gs_pcg_solve(c, mat, mas, bb, xx, nrhs=args.nrhs, tol=TOL, max_iter=20000, variant=variant)
        info = (B.gs_mat_info(mat)[1], B.gs_mas_info(mas))
        B.gs_mas_destroy(mas)
        B.gs_mat_destroy(mat)
        return it, rel, info

    # The systems of a step are independent Newton solves.  With --lanes (the
    # default) each runs on its own library context and CUDA stream, driven by
    # its own host thread, so the FP64-pipe-bound SpMV of one system overlaps
    # the HBM- and tensor-bound MAS apply of another.
    n_lanes = (args.streams if args.streams > 0 and args.queue else len(dsys)) if args.lanes else 1
    multi = n_lanes > 1  # one lane is the main context on the main stream
    lane_streams = [torch.cuda.Stream(device=dev) for _ in range(n_lanes)] if multi else [stream]
    lane_ctx = [B.gs_create(local, s_) for s_ in lane_streams] if multi else [ctx]
    # solution buffers per lane and system: two steps' solves of one system
    # may run at once on two lanes
    lane_xs = [[torch.zeros_like(b) for _ in dsys] for _ in range(n_lanes)] if multi else [[x] * len(dsys)]
    last_lane = {}  # system -> lane of its latest finished solve
    pool = ThreadPoolExecutor(max_workers=n_lanes)

    def fork():
        ev = torch.cuda.Event()
        ev.record(stream)
        for s_ in lane_streams:
            s_.wait_event(ev)

    def join():
        for s_ in lane_streams:
            ev = torch.cuda.Event()
            ev.record(s_)
            stream.wait_event(ev)

    def lane_run(i, fn):
        torch.cuda.set_device(local)
        with torch.cuda.stream(lane_streams[i]):
            return fn(i)

    def step():
        if n_lanes == 1:
            return [solve_one(s["rows"], s["cols"], s["blocks"], b, x) for s in dsys]
        fork()
        futs = [pool.submit(lane_run, i, lambda i, s=s: solve_one(s["rows"], s["cols"], s["blocks"], b, lane_xs[i][i],
                                                                   lane_ctx[i]))
                for i, s in enumerate(dsys)]
        out = [f.result() for f in futs]
        join()
        for i in range(len(dsys)):
            last_lane[i] = i
        return out

    def queue(n_steps, order, job):
        """The solves of n_steps steps as one queue over the lanes: each lane's
        thread takes the next solve as soon as its previous one is done, so no
        lane idles while a step's slowest system finishes.  order: the systems
        of a step, longest first.  job(lane, system) -> result."""
        jobs = [si for _ in range(n_steps) for si in order]
        nxt = iter(range(len(jobs)))
        lock = threading.Lock()
        out = {}

        def worker(i):
            while True:
                with lock:
                    j = next(nxt, None)
                if j is None:
                    return
                r = job(i, jobs[j])
                with lock:
                    out[jobs[j]] = r
                    last_lane[jobs[j]] = i

        fork()
        futs = [pool.submit(lane_run, i, worker) for i in range(n_lanes)]
        [f.result() for f in futs]
        join()
        return [out[si] for si in range(len(dsys))]

    def solve_job(i, si):
        s = dsys[si]
        return solve_one(s["rows"], s["cols"], s["blocks"], b, lane_xs[i][si], lane_ctx[i])

    def profile_begin(classes):
        for c in lane_ctx:
            B.gs_profile_begin(c, classes)

    def profile_end():
        tot_l, tot_ms = None, None
        for c in lane_ctx:
            l_, m_ = B.gs_profile_end(c)
            tot_l = l_ if tot_l is None else tot_l + l_
            tot_ms = m_ if tot_ms is None else tot_ms + m_
        return tot_l, tot_ms

    def barrier():
        if world > 1:
            dist.barrier()

    # launch shapes: the autotuner times each candidate on the stiffest system
    # (outside the timed region) and leaves the fastest set in the context
    tuned = None
    if args.autotune:
        from paper_2411_06224_gb300 import autotune

        s = dsys[-1]
        mat = B.gs_assemble(ctx, V, s["rows"], s["cols"], s["blocks"])
        mas = B.gs_build_mas(ctx, mat, shared["map"], ndom, shared["adj_ptr"], shared["adj"], shared["contacts"],
                             domain_size=N, max_levels=L, precision=prec)
        res = autotune.tune(ctx, mat, mas, nrhs=args.nrhs, reps=5, mixed=args.mixed_steps > 0,
                            fp64=prec == B.GS_PREC_FP64,
                            spmv_variant=variant if variant != B.GS_SPMV_SRBK else B.GS_SPMV_ROW)
        B.gs_mas_destroy(mas)
        if args.mixed_steps > 0 and args.nrhs <= 8:  # BF16 level-0 product: tensor cores or FP32 cores
            mas = B.gs_build_mas(ctx, mat, shared["map"], ndom, shared["adj_ptr"], shared["adj"], shared["contacts"],
                                 domain_size=N, max_levels=L, precision=B.GS_PREC_BF16)
            xr = torch.randn((args.nrhs, 3 * V), dtype=torch.float64, device=dev)
            yr = torch.empty_like(xr)
            res[autotune.NAMES[B.GS_TUNE_BF16_TC]] = autotune.sweep(
                ctx, B.GS_TUNE_BF16_TC, B.GS_K_MAS_APPLY_L0, lambda: B.gs_mas_apply(ctx, mas, xr, yr, nrhs=args.nrhs),
                reps=5)
            B.gs_mas_destroy(mas)
        tuned = {k: {"best": v[0], "ms_per_launch": {str(c): round(m, 4) for c, m in v[1].items()}}
                 for k, v in res.items()}
        B.gs_mat_destroy(mat)
        for c in lane_ctx:  # every lane uses the tuned shapes
            for prm in autotune.CANDIDATES:
                B.gs_tune_set(c, prm, B.gs_tune_get(ctx, prm))
    if args.set_tune:  # forced shapes, on every context
        from paper_2411_06224_gb300 import autotune

        by_name = {v: k for k, v in autotune.NAMES.items()}
        for item in args.set_tune:
            name, value = item.split("=")
            for c in {id(c): c for c in [ctx] + lane_ctx}.values():
                B.gs_tune_set(c, by_name[name], int(value))

    # warm-up
    for _ in range(args.warmup):  # with the queue its own lanes, so --streams may differ from the systems
        warm = queue(1, list(range(len(dsys))), solve_job) if (n_lanes > 1 and args.queue) else step()
    iters = [[int(v) for v in o[0]] for o in warm]
    # the queue takes a step's systems longest first (by the warm-up's iterations)
    order = sorted(range(len(dsys)), key=lambda si: -max(iters[si]))
    use_queue = n_lanes > 1 and args.queue
    nnzb = warm[0][2][0]
    mas_levels = warm[0][2][1]
    # per-class breakdown of one step, the systems one after another on the
    # main context (isolated kernel times; outside the timed region)
    B.gs_profile_begin(ctx, range(B.GS_K_COUNT))
    for s in dsys:
        solve_one(s["rows"], s["cols"], s["blocks"], b, x)
    launches_1, ms_1 = B.gs_profile_end(ctx)

    # timed region: the dominant kernels are bracketed by CUDA events on the library's stream
    timed_classes = [B.GS_K_MAS_APPLY_L0, B.GS_K_SPMV]
    clocks = ClockSampler(local)
    barrier()
    torch.cuda.synchronize()
    clocks.start()
    profile_begin(timed_classes)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    w0 = time.perf_counter()
    e0.record(stream)
    if use_queue:
        res = queue(args.steps, order, solve_job)
    else:
        for _ in range(args.steps):
            res = step()
    e1.record(stream)
    torch.cuda.synchronize()
    wall = time.perf_counter() - w0
    launches, kms = profile_end()
    barrier()
    clk = clocks.stop()
    from paper_2411_06224_gb300 import replicas

    # independent replicas: every rank solved its own systems; the slowest rank sets the time
    value, elapsed = replicas.throughput(len(dsys) * args.steps, e0.elapsed_time(e1) / 1e3, dev)

    # true residuals of the last step (checked on the device through the library's SpMV)
    true_rel = []
    if n_lanes > 1:
        x.copy_(lane_xs[last_lane[len(dsys) - 1]][len(dsys) - 1])
    Ax = torch.empty_like(x)
    for s in dsys[-1:]:
        mat = B.gs_assemble(ctx, V, s["rows"], s["cols"], s["blocks"])
        B.gs_spmv(ctx, mat, x, Ax, nrhs=args.nrhs, variant=B.GS_SPMV_ROW)
        true_rel = ((b - Ax).norm(dim=1) / b.norm(dim=1)).tolist()
        B.gs_mat_destroy(mat)

    # end-to-end through the public API with host buffers
    e2e = None
    if args.e2e_steps > 0:
        hsys = [dict(rows=torch.as_tensor(s.rows).pin_memory(), cols=torch.as_tensor(s.cols).pin_memory(),
                     blocks=torch.as_tensor(np.ascontiguousarray(s.blocks.reshape(-1, 3, 3))).pin_memory())
                for s in systems]
        hb = torch.as_tensor(b_host).pin_memory()
        hx = torch.empty_like(hb).pin_memory()
        h2d = sum(h["rows"].nbytes + h["cols"].nbytes + h["blocks"].nbytes + hb.nbytes for h in hsys)
        d2h = hx.nbytes * len(hsys)
        barrier()
        torch.cuda.synchronize()
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        hxs = [[torch.empty_like(hb).pin_memory() for _ in hsys] for _ in range(n_lanes)]

        def e2e_one(i, si, c):  # lane i, system si
            h = hsys[si]
            rows = h["rows"].to(dev, non_blocking=True)
            cols = h["cols"].to(dev, non_blocking=True)
            blocks = h["blocks"].to(dev, non_blocking=True)
            bb = hb.to(dev, non_blocking=True)
            xx = torch.empty_like(bb)
            solve_one(rows, cols, blocks, bb, xx, c)
            hxs[i][si].copy_(xx, non_blocking=True)
            torch.cuda.current_stream().synchronize()  # the host holds the answer

        f0.record(stream)
        if use_queue:
            queue(args.e2e_steps, order, lambda i, si: e2e_one(i, si, lane_ctx[i]))
        else:
            for _ in range(args.e2e_steps):
                if n_lanes == 1:
                    for si in range(len(hsys)):
                        e2e_one(0, si, ctx)
                else:
                    fork()
                    futs = [pool.submit(lane_run, i, lambda i: e2e_one(i, i, lane_ctx[i])) for i in range(len(hsys))]
                    [f.result() for f in futs]
                    join()
        f1.record(stream)
        torch.cuda.synchronize()
        e2e_rate, el = replicas.throughput(len(hsys) * args.e2e_steps, f0.elapsed_time(f1) / 1e3, dev)
        e2e = {"value": e2e_rate, "unit": "Newton solves/s",
               "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h)}

    # the mixed-precision forms on the same workload and right-hand sides:
    #   f64_pcg_f32_mas   FP64 PCG, MAS inverses stored and applied in FP32
    #   f64_pcg_bf16_mas  FP64 PCG, BF16 level-0 inverse Cholesky factors on the tensor cores
    #   f32_inner_pcg     FP32 PCG (FP32 SpMV + FP32 MAS) with FP64 reliable updates
    mixed = None
    if args.mixed_steps > 0 and args.nrhs <= 8:
        x_fp64 = x.clone()  # FP64 solution of the last system (last timed step)
        variants = [("f64_pcg_f32_mas", B.GS_PREC_FP32, False), ("f64_pcg_bf16_mas", B.GS_PREC_BF16, False),
                    ("f32_inner_pcg", B.GS_PREC_FP32, True)]
        mixed = {}
        def run_variant(vprec, inner32):
            def mixed_one(s):
                mat = B.gs_assemble(ctx, V, s["rows"], s["cols"], s["blocks"])
                mas = B.gs_build_mas(ctx, mat, shared["map"], ndom, shared["adj_ptr"], shared["adj"],
                                     shared["contacts"], domain_size=N, max_levels=L, precision=vprec)
                try:
                    if inner32:
                        it, rel, outer, _ = B.gs_pcg_solve_mixed(ctx, mat, mas, b, x, nrhs=args.nrhs, tol=TOL,
                                                                 max_iter=20000)
                    else:
                        it, rel, _ = B.gs_pcg_solve(ctx, mat, mas, b, x, nrhs=args.nrhs, tol=TOL, max_iter=20000,
                                                    variant=variant)
                        outer = None
                finally:
                    B.gs_mas_destroy(mas)
                    B.gs_mat_destroy(mat)
                return [int(v) for v in it], [float(v) for v in rel], outer

            mixed_one(dsys[0])  # warm-up
            B.gs_profile_begin(ctx, range(B.GS_K_COUNT))  # per-class times of one step, outside the timed region
            for s in dsys:
                mixed_one(s)
            m_launch, m_ms = B.gs_profile_end(ctx)
            barrier()
            torch.cuda.synchronize()
            g0 = torch.cuda.Event(enable_timing=True)
            g1 = torch.cuda.Event(enable_timing=True)
            g0.record(stream)
            mres = []
            for _ in range(args.mixed_steps):
                mres = [mixed_one(s) for s in dsys]
            g1.record(stream)
            torch.cuda.synchronize()
            mrate, mel = replicas.throughput(len(dsys) * args.mixed_steps, g0.elapsed_time(g1) / 1e3, dev)
            # true residuals of the last system, recomputed in FP64 through the library's SpMV
            s = dsys[-1]
            mat = B.gs_assemble(ctx, V, s["rows"], s["cols"], s["blocks"])
            B.gs_spmv(ctx, mat, x, Ax, nrhs=args.nrhs, variant=B.GS_SPMV_ROW)
            B.gs_mat_destroy(mat)
            return {
                "value": mrate, "unit": "Newton solves/s", "ms_per_step": mel / args.mixed_steps * 1e3,
                "steps": args.mixed_steps,
                "iterations": [r[0] for r in mres], "outer_steps": [r[2] for r in mres],
                "true_rel_residual_last_system": ((b - Ax).norm(dim=1) / b.norm(dim=1)).tolist(),
                # both solves stop on the 1e-6 residual test; their distance (last system)
                "rel_error_vs_fp64_max": float(((x - x_fp64).norm(dim=1) / x_fp64.norm(dim=1)).max()),
                "phase_ms_one_step": {B.K_NAMES[k]: round(float(m_ms[k]), 2) for k in range(B.GS_K_COUNT)},
                "launches_one_step": {B.K_NAMES[k]: int(m_launch[k]) for k in range(B.GS_K_COUNT)},
            }

        for name, vprec, inner32 in variants:
            try:
                mixed[name] = run_variant(vprec, inner32)
            except B.GsError as e:  # a form that fails is reported; the main measurement stands
                mixed[name] = {"error": str(e)[:300]}

    # the precision forms on a stiff cloth sheet (the paper's strain-limited cloth:
    # cubic strain limiting with E = 1e8, 512 x 512 vertices, 4 RHS): FP64 PCG
    # with the FP64 / FP32 / BF16 preconditioner, time per solve and the
    # distance of each answer from the FP64 one
    cloth = None
    if args.cloth > 0:
        from synth.cloth import make_cloth_system

        cs = make_cloth_system(args.cloth, seed=1003 + rank)
        Vc, nrc = cs.n_vertices, 4
        cmap, cnd = B.gs_partition(cs.X, N)
        cd = dict(rows=t(cs.rows, torch.int32), cols=t(cs.cols, torch.int32),
                  blocks=t(cs.blocks.reshape(-1, 3, 3), torch.float64), map=t(cmap, torch.int32),
                  adj_ptr=t(cs.adj_ptr, torch.int32), adj=t(cs.adj, torch.int32))
        cb = t(np.stack([np.random.default_rng(2000 + k).normal(size=3 * Vc) for k in range(nrc)]), torch.float64)
        cloth = {"workload": f"cloth {args.cloth}x{args.cloth} ({Vc} vertices, {cs.rows.size} triplets), strain "
                             f"limiting E=1e8, {nrc} RHS, 3-level MAS N=32, FP64 PCG tol 1e-6"}
        xc64 = None
        for name, cprec in (("fp64", B.GS_PREC_FP64), ("fp32", B.GS_PREC_FP32), ("bf16", B.GS_PREC_BF16)):
            def csolve():
                mat = B.gs_assemble(ctx, Vc, cd["rows"], cd["cols"], cd["blocks"])
                mas = B.gs_build_mas(ctx, mat, cd["map"], cnd, cd["adj_ptr"], cd["adj"], None, domain_size=N,
                                     max_levels=L, precision=cprec)
                xc = torch.zeros_like(cb)
                try:
                    it, _, _ = B.gs_pcg_solve(ctx, mat, mas, cb, xc, nrhs=nrc, tol=TOL, max_iter=20000)
                    Ac = torch.empty_like(xc)
                    B.gs_spmv(ctx, mat, xc, Ac, nrhs=nrc)
                    true = ((cb - Ac).norm(dim=1) / cb.norm(dim=1)).max().item()
                finally:
                    B.gs_mas_destroy(mas)
                    B.gs_mat_destroy(mat)
                return it, true, xc

            try:
                csolve()  # warm-up
                torch.cuda.synchronize()
                c0 = torch.cuda.Event(enable_timing=True)
                c1 = torch.cuda.Event(enable_timing=True)
                c0.record(stream)
                it, true, xc = csolve()
                c1.record(stream)
                torch.cuda.synchronize()
                row = {"ms_per_solve": c0.elapsed_time(c1), "iterations": [int(v) for v in it],
                       "true_rel_residual_max": true}
                if name == "fp64":
                    xc64 = xc
                else:
                    row["rel_error_vs_fp64_max"] = float(((xc - xc64).norm(dim=1) / xc64.norm(dim=1)).max())
                cloth[name] = row
            except B.GsError as e:
                cloth[name] = {"error": str(e)[:300]}
        try:
            cloth["element_hessians"] = cloth_element_line(args, B, dev, stream, clk)
        except B.GsError as e:
            cloth["element_hessians"] = {"error": str(e)[:300]}

    # the batched form: 64 independent uneven tet cubes (1k-50k vertices, E 1e5-1e9,
    # contacts on 5% of the vertices), one RHS each, solved as one block-diagonal
    # batch with one PCG recurrence per system and the loop in one CUDA graph;
    # compared with solving the same systems one after another on the plain path
    batched = None
    if args.batch_steps > 0:
        from synth.workloads import uneven_batch

        bt = uneven_batch(64, seed=1004 + rank)
        Vb = bt.n_vertices
        bmap, bnd = B.gs_partition_batch(bt.X, bt.node_off, N)  # once per mesh set, before timing
        bd = dict(rows=t(bt.rows, torch.int32), cols=t(bt.cols, torch.int32),
                  blocks=t(bt.blocks.reshape(-1, 3, 3), torch.float64), map=t(bmap, torch.int32),
                  adj_ptr=t(bt.adj_ptr, torch.int32), adj=t(bt.adj, torch.int32), contacts=t(bt.contacts, torch.int32))
        bb = t(rhs_batch := np.random.default_rng(3000 + rank).normal(size=3 * Vb), torch.float64)
        bx = torch.zeros_like(bb)

        def batch_solve(prec_b):
            mat = B.gs_assemble(ctx, Vb, bd["rows"], bd["cols"], bd["blocks"])
            mas = B.gs_build_mas(ctx, mat, bd["map"], bnd, bd["adj_ptr"], bd["adj"], bd["contacts"],
                                 domain_size=N, max_levels=L, precision=prec_b)
            it, rel, _ = B.gs_pcg_solve_batch(ctx, mat, mas, bt.node_off, bb, bx, tol=TOL, max_iter=20000,
                                              use_graph=True)
            B.gs_mas_destroy(mas)
            B.gs_mat_destroy(mat)
            return it, rel

        def timed(fn, steps):
            fn()  # warm-up
            torch.cuda.synchronize()
            q0 = torch.cuda.Event(enable_timing=True)
            q1 = torch.cuda.Event(enable_timing=True)
            q0.record(stream)
            out = None
            for _ in range(steps):
                out = fn()
            q1.record(stream)
            torch.cuda.synchronize()
            return q0.elapsed_time(q1) / 1e3 / steps, out

        tb64, (it64, rel64) = timed(lambda: batch_solve(B.GS_PREC_FP64), args.batch_steps)
        tb32, (it32, rel32) = timed(lambda: batch_solve(B.GS_PREC_FP32), args.batch_steps)
        # the same 64 systems one at a time on the plain path
        seq = []
        for si, sysb in enumerate(bt.systems):
            Vs = sysb.n_vertices
            mps, nds = B.gs_partition(sysb.X, N)
            seq.append((Vs, t(sysb.rows, torch.int32), t(sysb.cols, torch.int32),
                        t(sysb.blocks.reshape(-1, 3, 3), torch.float64), t(mps, torch.int32), nds,
                        t(sysb.adj_ptr, torch.int32), t(sysb.adj, torch.int32), t(sysb.contacts, torch.int32),
                        t(rhs_batch[3 * bt.node_off[si]:3 * bt.node_off[si + 1]], torch.float64)))

        def sequential():
            for (Vs, r_, c_, bl_, mp_, nd_, ap_, aj_, ct_, b_) in seq:
                mat = B.gs_assemble(ctx, Vs, r_, c_, bl_)
                mas = B.gs_build_mas(ctx, mat, mp_, nd_, ap_, aj_, ct_, domain_size=N, max_levels=L)
                xs = torch.empty_like(b_)
                B.gs_pcg_solve(ctx, mat, mas, b_, xs, nrhs=1, tol=TOL, max_iter=20000)
                B.gs_mas_destroy(mas)
                B.gs_mat_destroy(mat)

        tseq, _ = timed(sequential, 1)
        batched = {
            "workload": "64 tet cubes, vertices log-uniform 1k-50k (%d total), E log-uniform 1e5-1e9, contacts on 5%% of "
                        "vertices, 1 RHS each, 3-level MAS N=32, tol 1e-6" % Vb,
            "fp64": {"value": 64 / tb64, "unit": "Newton solves/s", "ms_per_batch": tb64 * 1e3,
                     "max_iterations": int(max(it64)), "true_rel_residual_max": float(max(rel64))},
            "fp32_preconditioner": {"value": 64 / tb32, "unit": "Newton solves/s", "ms_per_batch": tb32 * 1e3,
                                    "max_iterations": int(max(it32))},
            "sequential_plain_fp64": {"value": 64 / tseq, "unit": "Newton solves/s", "ms_for_64": tseq * 1e3},
            "graph": "whole PCG loop = one CUDA graph launch (conditional WHILE node)",
        }

    # level-0 partitions and level counts compared (the paper's Table MAS:
    # connectivity-enhanced MAS against the Morton-order MAS of Wu et al.,
    # and block-Jacobi), on the stiffest sweep system and on a scene of
    # separate bodies interleaved in one box; the partition runs on the
    # device inside the timed build
    partitions = None
    if args.partition_steps > 0:
        from synth.workloads import uneven_batch

        def compare(rows_, cols_, blocks_, Vn, Xd, ptr_d, adj_d, con_d, bb, nr, variants):
            out = {}
            for name, rule, levels in variants:
                xx = torch.zeros_like(bb)

                def run():
                    b0 = torch.cuda.Event(enable_timing=True)
                    b1 = torch.cuda.Event(enable_timing=True)
                    b2 = torch.cuda.Event(enable_timing=True)
                    b0.record(stream)
                    mat = B.gs_assemble(ctx, Vn, rows_, cols_, blocks_)
                    mas = B.gs_build_mas_mesh(ctx, mat, Xd, ptr_d, adj_d, con_d, domain_size=N, max_levels=levels,
                                              part_rule=rule)
                    b1.record(stream)
                    it, _, _ = B.gs_pcg_solve(ctx, mat, mas, bb, xx, nrhs=nr, tol=TOL, max_iter=20000,
                                              variant=variant)
                    b2.record(stream)
                    torch.cuda.synchronize()
                    nl = B.gs_mas_info(mas)
                    B.gs_mas_destroy(mas)
                    B.gs_mat_destroy(mat)
                    return it, b0.elapsed_time(b1), b1.elapsed_time(b2), nl

                run()  # warm-up
                it, t_build, t_pcg = None, 0.0, 0.0
                for _ in range(args.partition_steps):
                    it, tb, tp, nl = run()
                    t_build += tb / args.partition_steps
                    t_pcg += tp / args.partition_steps
                out[name] = {"pcg_iterations": [int(v) for v in it], "levels": nl[1],
                             "ms_assembly_and_build": t_build, "ms_pcg": t_pcg,
                             "solves_per_s": 1e3 / (t_build + t_pcg)}
            return out

        variants = [("ce_mas_rcb", B.GS_PART_RCB, L), ("mas_morton", B.GS_PART_MORTON, L),
                    ("block_jacobi", B.GS_PART_RCB, 1)]
        sx = systems[-1]
        Xs = t(sx.X, torch.float64)
        partitions = {"sweep_E1e9": {
            "workload": f"{args.grid}^3 sweep system E=1e9, {args.nrhs} RHS, N=32, tol 1e-6",
            **compare(dsys[-1]["rows"], dsys[-1]["cols"], dsys[-1]["blocks"], V, Xs, shared["adj_ptr"],
                      shared["adj"], shared["contacts"], b, args.nrhs, variants)}}
        bt = uneven_batch(24, seed=1006 + rank)
        Vb = bt.n_vertices
        rb = t(np.random.default_rng(3100).normal(size=(1, 3 * Vb)), torch.float64)
        partitions["interleaved_bodies"] = {
            "workload": f"24 tet cubes (1k-50k vertices, {Vb} total, E 1e5-1e9) in the same unit box as one "
                        "system, 1 RHS, N=32, tol 1e-6",
            **compare(t(bt.rows, torch.int32), t(bt.cols, torch.int32), t(bt.blocks.reshape(-1, 3, 3), torch.float64),
                      Vb, t(bt.X, torch.float64), t(bt.adj_ptr, torch.int32), t(bt.adj, torch.int32),
                      t(bt.contacts, torch.int32), rb, 1,
                      [("ce_mas_rcb_components", B.GS_PART_RCB_COMPONENTS, L), ("ce_mas_rcb", B.GS_PART_RCB, L),
                       ("mas_morton", B.GS_PART_MORTON, L), ("block_jacobi", B.GS_PART_RCB_COMPONENTS, 1)])}

    # the plain FP64 solve on the 16^3 cube
    plain16 = None
    if args.config1:
        try:
            plain16 = config1_form(args, B, dev, variant, clk)
        except B.GsError as e:
            plain16 = {"error": str(e)[:300]}

    # Newton's method with device element Hessians and the fixed pattern
    newton_f = None
    if args.newton:
        try:
            newton_f = newton_form(args, B, dev, clk)
        except B.GsError as e:
            newton_f = {"error": str(e)[:300]}

    # the differentiation form on the coupled FEM + affine-body scene
    abd_f = None
    if args.abd:
        try:
            abd_f = abd_form(args, B, dev, clk)
        except B.GsError as e:
            abd_f = {"error": str(e)[:300]}

    # roofline of the dominant kernel class
    apply_line, spmv_line = kernel_lines(B, ctx, dev, clk, args.spmv, prec, args.nrhs, N, V, nnzb, ndom, mp,
                                         (launches, kms), (launches_1, ms_1),
                                         workload="tet64" if args.grid == 64 else None)
    for ln in (apply_line, spmv_line):
        ln["concurrent_streams"] = n_lanes
    # dominant by the per-class device time of one step with the systems one
    # after another (the order of the ncu launch list's shares); with three
    # streams overlapping, each launch's event time also holds the other
    # streams' kernels, and the SpMV's stretches the most
    dominant = apply_line if ms_1[B.GS_K_MAS_APPLY_L0] >= ms_1[B.GS_K_SPMV] else spmv_line
    dominant = dict(dominant, dominant_by="device time per class in one step, systems one after another")
    mine = int(sum(launches[k] for k in range(B.GS_K_COUNT) if k != B.GS_K_LIBPRIM))

    line = {
        "metric": METRIC,
        "value": value,
        "unit": "Newton solves/s",
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": elapsed / args.steps * 1e3,
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f64" if prec == B.GS_PREC_FP64 else f"f64+{args.precision}-precond",
        "data": "synthetic",
        "config": {
            "workload": f"tet cube {args.grid}^3 stiffness sweep E=1e5,1e7,1e9; {len(systems[0].contacts)} contacts; "
                        f"{args.nrhs} RHS; 3-level MAS N=32; PCG tol 1e-6",
            "vertices": V, "dof": 3 * V, "triplets_per_system": int(systems[0].rows.size), "stored_blocks": int(nnzb),
            "mas_levels": mas_levels[1], "nrhs": args.nrhs, "spmv": args.spmv, "precision": args.precision,
            "pcg_iterations": iters, "true_rel_residual_last_system": true_rel,
            "l2": "inputs larger than L2 (1.07 GB of triplets and 0.6 GB of level-0 inverses per system vs 129 MB L2); no flush",
            "parallelism": f"independent systems per GPU x{world}",
            "schedule": (f"one queue over the timed steps' {len(dsys)} x steps solves on {n_lanes} streams, "
                         "each step's systems longest first" if use_queue else
                         (f"{n_lanes} streams, one system each, synchronised per step" if n_lanes > 1
                          else "one stream, systems one after another")),
            "launch_shapes": autotune_current(B, ctx),
            "autotune": tuned,
        },
        "roofline": dominant,
        "kernels": {"mas_apply_l0": apply_line, "spmv": spmv_line,
                    "spmv_hbm_gbs": spmv_line["hbm_gbs"]},
        "phase_ms_one_step": {B.K_NAMES[k]: float(ms_1[k]) for k in range(B.GS_K_COUNT)},
        "launches_one_step": {B.K_NAMES[k]: int(launches_1[k]) for k in range(B.GS_K_COUNT)},
        "e2e": e2e,
        "forms": {"mixed_precision": mixed, "batched": batched, "precision_cloth": cloth, "plain16": plain16,
                  "partitions": partitions, "newton": newton_f, "differentiation_abd": abd_f},
        "clocks": clk,
        "gpu_launches": mine,
        "libprim_calls": int(launches[B.GS_K_LIBPRIM]),
        "wall_s": wall,
    }
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        try:
            res = run_oracle_sample(args.grid, [1e5], 1, iters=20, procs=args.nrhs)
            smp, host = res["samples"][0], res["host"]
            T1 = Tp = 0.0
            for its in iters:  # the step's systems, with the GPU run's per-RHS counts
                _, _, t1, tp = oracle_rates(smp["t_ga"], smp["t_pa"], smp["t_iter"], smp.get("t_iter_par"), its)
                T1 += t1
                Tp += tp if tp else t1
            rate1, ratep = len(iters) / T1, len(iters) / Tp
            line["cpu_baseline"] = {
                "value": ratep, "unit": "Newton solves/s", "cores": smp.get("procs", 1), "kind": "oracle",
                "sample": (f"FP64 numpy/scipy oracle on the host ({host['nproc']} cores, {host['cpu_model']}), one BLAS "
                           f"thread per process, E=1e5 system of the {args.grid}^3 sweep: full assembly "
                           f"({smp['t_ga']:.2f} s), full 3-level MAS build ({smp['t_pa']:.2f} s), {smp['k']} PCG "
                           f"iterations on 1 RHS ({smp['t_iter']:.3f} s each) and on {smp.get('procs', 1)} RHS in as "
                           f"many concurrent processes ({smp.get('t_iter_par', 0):.3f} s per iteration); a step's "
                           f"three solves timed with the GPU run's per-RHS iteration counts, RHS in parallel "
                           f"(assembly and build single-threaded)"),
                "single_thread": {"value": rate1, "cores": 1},
                "phases_s": {"assembly": smp["t_ga"], "mas_build": smp["t_pa"], "pcg_iteration_1rhs": smp["t_iter"],
                             "pcg_iteration_parallel": smp.get("t_iter_par")},
                "host": host,
            }
        except Exception as e:  # noqa: BLE001
            line["cpu_baseline"] = {"value": None, "error": str(e)[:300]}
    B.gs_destroy(ctx)
    if rank == 0:
        # the forms' whole records (16 KB) go to stderr: a line that long is cut by what reads it
        print("forms: " + json.dumps(line["forms"], default=_json_scalar), file=sys.stderr, flush=True)
        line["forms"] = brief(line["forms"])
        print(json.dumps(line, default=_json_scalar), flush=True)
    if world > 1:
        dist.destroy_process_group()


def micro(args):
    """The paper's microbenchmarks, one JSON line.

    reduce: 2^24 3x3 blocks with sorted keys, every key repeated 2^d times;
      the paper's FastHashReduction against the CUB library's ReduceByKey on
      the same sorted input (both gather nothing; inputs resident in HBM).
    spmv: random symmetric patterns, 2^18 block rows with about b blocks per
      full row (diagonal plus (b-1)/2 random upper blocks per row); the
      paper's symmetric storage with atomic scatter (SRBK), the row-gather
      over the same storage, and the cuSPARSE library's BSR SpMV on the full
      matrix; one right-hand side."""
    import numpy as np
    import torch

    from paper_2411_06224_gb300.build import build

    build()
    from paper_2411_06224_gb300 import binding as B

    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    ctx = B.gs_create(0, torch.cuda.current_stream())
    gen = torch.Generator(device=dev).manual_seed(1007)
    out = {"metric": "microbenchmarks", "config": {"workload": "paper reduction / SpMV microbenchmarks"}}
    nb = 1 << 24
    blocks = torch.randn((nb, 3, 3), dtype=torch.float64, device=dev, generator=gen)
    red = []
    for d in (0, 1, 2, 4, 7, 10, 13, 16):
        keys = torch.arange(nb, device=dev, dtype=torch.int64) >> d
        row = {"dup": 1 << d}
        for method, name in ((0, "fast_hash_reduction"), (1, "cub_reduce_by_key")):
            times = []
            for _ in range(4):
                o, ms = B.gs_micro_segment_reduce(ctx, keys, blocks, method)
                times.append(ms)
            t_ms = float(np.median(times[1:]))
            u = o.shape[0]
            row[name] = {"ms": t_ms, "gbs": (nb * 80 + u * 72) / t_ms / 1e6}
        row["speedup"] = row["cub_reduce_by_key"]["ms"] / row["fast_hash_reduction"]["ms"]
        red.append(row)
        del keys
    del blocks
    out["reduce_16M_blocks"] = red
    n = 1 << 18
    sp = []
    for bpr in (1, 2, 4, 8, 16, 32, 64):
        m = (bpr - 1) / 2.0
        k_off = int(round(m * n))
        r_off = torch.randint(0, n - 1, (k_off,), device=dev, generator=gen)
        span = (n - 1 - r_off).to(torch.float64)
        c_off = r_off + 1 + (torch.rand(k_off, device=dev, generator=gen, dtype=torch.float64) * span).long()
        rows = torch.cat([torch.arange(n, device=dev), r_off]).int()
        cols = torch.cat([torch.arange(n, device=dev), c_off]).int()
        vals = torch.randn((rows.numel(), 3, 3), dtype=torch.float64, device=dev, generator=gen)
        mat = B.gs_assemble(ctx, n, rows, cols, vals)
        _, nnzb = B.gs_mat_info(mat)
        x = torch.randn((1, 3 * n), dtype=torch.float64, device=dev, generator=gen)
        y = torch.empty_like(x)
        row = {"blocks_per_full_row": bpr, "upper_blocks": int(nnzb)}
        for variant, name in ((B.GS_SPMV_SRBK, "srbk_symmetric"), (B.GS_SPMV_ROW, "row_gather_symmetric")):
            B.gs_spmv(ctx, mat, x, y, nrhs=1, variant=variant)
            B.gs_profile_begin(ctx, [B.GS_K_SPMV])
            for _ in range(10):
                B.gs_spmv(ctx, mat, x, y, nrhs=1, variant=variant)
            launches, kms = B.gs_profile_end(ctx)
            row[name] = {"ms": float(kms[B.GS_K_SPMV] / max(launches[B.GS_K_SPMV], 1))}
        rid, cid, au = B.gs_mat_export(ctx, mat)
        off = rid != cid
        fr = torch.cat([rid, cid[off]]).long()
        fc = torch.cat([cid, rid[off]]).long()
        fa = torch.cat([au, au[off].transpose(1, 2)])
        order = torch.argsort(fr * n + fc)
        fr, fc, fa = fr[order], fc[order], fa[order].contiguous()
        ptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
        ptr[1:] = torch.cumsum(torch.bincount(fr, minlength=n), 0)
        yf = torch.empty(3 * n, dtype=torch.float64, device=dev)
        B.gs_micro_bsr_spmv_cusparse(ctx, n, ptr.int(), fc.int(), fa, x[0].contiguous(), yf, reps=2)
        ms = B.gs_micro_bsr_spmv_cusparse(ctx, n, ptr.int(), fc.int(), fa, x[0].contiguous(), yf, reps=10)
        row["cusparse_bsr_full"] = {"ms": ms, "full_blocks": int(fc.numel())}
        row["max_rel_diff_vs_row_gather"] = float((yf - y[0]).abs().max() / y[0].abs().max())
        for name in ("srbk_symmetric", "row_gather_symmetric", "cusparse_bsr_full"):
            # algorithmic bytes of the symmetric storage: 76 B per stored block + 48 B per row
            row[name]["gbs_symmetric_bytes"] = (nnzb * 76 + n * 48) / row[name]["ms"] / 1e6
            row[name]["gflops"] = (2 * 9 * (2 * nnzb - n)) / row[name]["ms"] / 1e6
        sp.append(row)
        B.gs_mat_destroy(mat)
    out["spmv_random_2p18_rows"] = sp
    B.gs_destroy(ctx)
    print(json.dumps(out), flush=True)


def reference_arm(args, rank, world):
    """The oracle timed on the host cores (rank 0 only), same metric and workload.

    A step is one bounded phase sample of the workload, cycling through
    assembly, MAS build and PCG (20 iterations on 1 RHS, then on every RHS in
    as many concurrent processes); `value` combines the timed steps' mean
    phase times with the oracle's own per-RHS iteration counts of the three
    systems (supplement Eq. 1), RHS in parallel.  `ms_per_step` is the wall
    time of a step."""
    if rank != 0:
        return
    import json as _json

    golden = os.path.join(ROOT, "tests", "golden", "sweep64_pcg_iterations.json")
    its = None
    if args.grid == 64 and os.path.exists(golden):
        its = list(_json.load(open(golden))["iterations"].values())
    n_contacts = max(1, 200_000 * args.grid ** 3 // 64 ** 3)
    Es = [float(e) for e in args.sweep.split(",")]
    # at least one sample of each of the cycle's three phases, however few steps are asked for
    res = run_oracle_sample(args.grid, Es, max(args.warmup + args.steps, 3), iters=20, procs=args.nrhs,
                            cycle=True)
    allv, host = res["samples"], res["host"]
    vals = allv[args.warmup:args.warmup + args.steps] or allv[-1:]
    mean = lambda key: statistics.mean([v[key] for v in vals if v.get(key) is not None] or
                                      [v[key] for v in allv if v.get(key) is not None])
    t_ga, t_pa, t_it, t_par = mean("t_ga"), mean("t_pa"), mean("t_iter"), mean("t_iter_par")
    if its is None:
        its = [[150] * args.nrhs] * len(Es)
    T1 = sum(oracle_rates(t_ga, t_pa, t_it, t_par, v)[2] for v in its)
    Tp = sum(oracle_rates(t_ga, t_pa, t_it, t_par, v)[3] for v in its)
    value = len(its) / Tp
    step_wall = []
    for v in vals:
        w = v.get("t_ga", 0.0) if "k" not in v else 0.0
        w += v.get("t_pa", 0.0) if "k" not in v else 0.0
        if "k" in v:
            w = v["k"] * (v["t_iter"] + v.get("t_iter_par", 0.0))
        step_wall.append(w)
    line = {
        "impl": "reference",
        "metric": METRIC,
        "value": value,
        "unit": "Newton solves/s",
        "n_gpus": world,
        "steps": len(vals),
        "warmup": args.warmup,
        "ms_per_step": 1e3 * statistics.mean(step_wall),
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": f"tet cube {args.grid}^3 stiffness sweep E={args.sweep}; {n_contacts} contacts; "
                               f"{args.nrhs} RHS; 3-level MAS N=32; PCG tol 1e-6",
                   "step": "one phase sample of the workload (assembly, MAS build, or 20 PCG iterations on 1 RHS "
                           f"and on {args.nrhs} RHS in concurrent processes), cycling"},
        "cpu_baseline": {"value": value, "unit": "Newton solves/s", "cores": args.nrhs, "kind": "oracle",
                         "sample": (f"FP64 numpy/scipy oracle on {host['nproc']} host cores ({host['cpu_model']}), one "
                                    f"BLAS thread per process: mean phase times assembly {t_ga:.2f} s, MAS build "
                                    f"{t_pa:.2f} s, PCG iteration {t_it:.3f} s (1 RHS) / {t_par:.3f} s ({args.nrhs} RHS "
                                    f"in parallel processes); solves timed with the oracle's own per-RHS iteration "
                                    + ("counts (tests/golden/sweep64_pcg_iterations.json)" if args.grid == 64
                                       else "counts assumed 150 per RHS")),
                         "single_thread": {"value": len(its) / T1, "cores": 1},
                         "host": host},
        "e2e": {"value": value, "unit": "Newton solves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line, default=_json_scalar))


if __name__ == "__main__":
    main()

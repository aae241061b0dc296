#!/usr/bin/env python
"""Throughput of the per-time-step path (Algorithm 2) on the 3D hybrid workloads.

Workload (default): layers3d, 32x16 spectral elements of order 10 times Nz = 256 Fourier planes
(n_x n_y Nz = 13,189,120 real values per field; 6,646,080 complex coefficients), two stacked
dielectric layers plus a drop (eps ratio 20, rho ratio 10, mu ratio 10), V = 2 / 0, dt = 5e-5.
One "step" = one full time step (V, E, psi, phi, P, u), all of it in the CUDA library through the
C-ABI.  Metric: DOF-steps/s, DOF = real values of one scalar field.  The mixed path is the value;
the same line carries the FP64 path's rate and the mixed path's per-field error against it.

Prints one JSON line (rank 0).  --impl reference times the FP64 CPU oracle instead.
"""
from __future__ import annotations

import os

# the oracle legs run on one host core: BLAS and OpenMP pools are fixed before numpy loads
for _v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS", "BLIS_NUM_THREADS"):
    os.environ[_v] = "1"
ORACLE_THREADS = 1


import argparse
import hashlib
import json
import math
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "DOF-steps/s at stated err vs FP64 oracle; time-to-equilibrium warm vs cold"
UNIT = "DOF-steps/s"
L2_FLUSH_BYTES = 256 << 20


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as fh:
            d = json.load(fh)
        return d, "measured"
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "sm_max_mhz": 2070.0}, "fallback"


# ---- workloads that bench.py can time ------------------------------------------------------------
WORKLOADS = {
    "droplet3d": "droplet3d: 16x8 elements order 8 x Nz=64 planes, sphere r=0.25 on the electrode, "
                 "eps/rho/mu ratios 10/2/5, V=2, dt=5e-5",
    "electrode_array3d": "electrode_array3d: 20x6 elements order 12 x Nz=120 planes, ten electrode stripes "
                         "at +-150 V (the paper's normalisation), hemispherical drop, permittivity ratio 32, "
                         "equilibrium system, pseudo-time step 2e-6",
    "patches2d": "patches2d: 16x4 elements order 8, four electrodes at -+0.5 on the wall, half-disc drop, "
                 "eps/rho/mu ratios 5/2/2, dt=1e-4",
    "ensemble2d": "ensemble2d: 256 independent 2D runs (seed 20230515), meshes 4x2..24x12 elements, orders 4..10, "
                  "V~U(0,3), eps ratio logU(2,20), drop radius U(0.15,0.35) on the wall, eta 0.02, dt 1e-4",
    "layers3d": "layers3d: 32x16 elements order 10 x Nz=256 planes, two stacked layers (fluid 1 below y=0.3) plus "
                "a drop r=0.15 at (1,0.65,0.5), eta=0.005, eps/rho/mu ratios 20/10/10, V=2, dt=5e-5",
}


def make_workload(name):
    import workloads
    return getattr(workloads, name)()


# ---- CPU oracle sample (cpu_baseline and --impl reference) -----------------------------------
def oracle_sample(nsteps: int, warmup: int, name: str = "droplet3d"):
    """Steady-state BDF2 steps of the FP64 oracle on the workload's element mesh and physics
    (3D: with Nz = 8 planes; the oracle's sparse LU factorisations per mode make the full plane
    counts take minutes per step).  Returns (DOF-steps/s, seconds, description)."""
    import numpy as np
    from oracle.runner import solver_of
    wl = make_workload(name)
    if isinstance(wl, list):        # an ensemble: its first run stands for the sample
        wl = wl[0]
        name = name + " (first run)"
    if wl.mesh.nz > 1:
        wl.mesh.nz = 8
    sub = ""
    if len(wl.mesh.xb) - 1 > 16:    # bounded sample: at most 16 x 8 elements of the same domain
        import numpy as np
        ex, ey = 16, max(1, (len(wl.mesh.yb) - 1) * 16 // (len(wl.mesh.xb) - 1))
        wl.mesh.xb = np.linspace(wl.mesh.xb[0], wl.mesh.xb[-1], ex + 1)
        wl.mesh.yb = np.linspace(wl.mesh.yb[0], wl.mesh.yb[-1], ey + 1)
        sub = f", {ex}x{ey} of its elements"
    sol = solver_of(wl, init=False)
    Zg, Yg, Xg = np.meshgrid(sol.zc, sol.mesh.Y, sol.mesh.X, indexing="ij")
    sol.set_initial(wl.phi0(Xg, Yg, Zg).reshape(sol.nz, sol.mesh.n2), max_iter=3)
    for _ in range(max(2, warmup)):       # BDF1 + first BDF2 step build the LU factors
        sol.step()
    t0 = time.perf_counter()
    for _ in range(nsteps):
        sol.step()
    dt = time.perf_counter() - t0
    dof = sol.mesh.n2 * sol.nz
    desc = (f"oracle (scipy SuperLU, numpy FFT), {name} element mesh{sub}"
            + (" with Nz=8 planes" if sol.nz > 1 else "") +
            f" ({dof} DOF), {nsteps} steady BDF2 step(s) after {max(2, warmup)} warm-up steps; "
            f"initial-potential iterations capped at 3 (set-up is not timed)")
    return dof * nsteps / dt, dt, desc


def reference_arm(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    steps = max(1, args.steps)
    val, secs, desc = oracle_sample(steps, args.warmup, args.workload)
    line = {"impl": "reference", "metric": METRIC, "value": val, "unit": UNIT, "n_gpus": args.gpus,
            "steps": steps, "warmup": args.warmup, "ms_per_step": secs * 1e3 / steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": f"{args.workload} (oracle sample" +
                                                        (": Nz=8)" if args.workload != "patches2d" else ")")},
            "cpu_baseline": {"value": val, "unit": UNIT, "cores": ORACLE_THREADS, "host_cpus": os.cpu_count(),
                             "kind": "oracle", "sample": desc},
            "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


# ---- clocks ------------------------------------------------------------------------------------
class ClockSampler:
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.f = tempfile.NamedTemporaryFile(mode="w+", suffix=".csv", delete=False)
        try:
            self.p = subprocess.Popen(["nvidia-smi", f"--id={gpu_index}", f"--query-gpu={self.Q}",
                                       "--format=csv,noheader,nounits", "-lms", "100"],
                                      stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.p = None

    def stop(self):
        if self.p is None:
            return None
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except Exception:
            self.p.kill()
        self.f.flush()
        self.f.seek(0)
        rows = [r.split(",") for r in self.f.read().strip().splitlines() if r.strip()]
        os.unlink(self.f.name)
        sm = [float(r[1]) for r in rows if len(r) >= 9 and r[1].strip().replace(".", "").isdigit()]
        if not sm:
            return None
        mx = max(float(r[2]) for r in rows if len(r) >= 9)
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if len(r) >= 9 and "Active" in r[5 + i]
                          and "Not" not in r[5 + i]})
        sm.sort()
        return {"sm_mhz": sm[len(sm) // 2], "sm_max_mhz": mx, "reasons": reasons, "samples": len(sm)}


# ---- algorithmic work per kernel class ----------------------------------------------------------
def transform_kernel(code, fused_y):
    """Kernel(s) of the chosen transform variant (PF_GEMM_* code)."""
    name = {0: "k_gemm_tc", 1: "k_fdm_plane", 6: "k_fdm_cluster<4>", 7: "k_fdm_cluster<2>",
            8: "k_gemm_tc + k_gemm_cp", 9: "k_oz_split + k_gemm_oz"}.get(code, "k_gemm_cp" if code in (3, 4, 5) else "k_gemm")
    return name + (" + k_fdm_y" if fused_y and code not in (0, 1, 6, 7, 8, 9) else "")


# DRAM traffic per launch of a transform kernel, from one ncu capture of an unchanged kernel
# (profiles/): (workload, precision, variant code, fused y) -> bytes
TRANSFORM_DRAM_BYTES_PER_LAUNCH = {("droplet3d", "mixed", 3, 0): 2.24e6, ("layers3d", "mixed", 0, 0): 5.49e7}


def transform_bytes_per_launch(nx, ny, nz, prec):
    """Algorithmic bytes of one transform GEMM launch of a scalar solve: read the planes and the
    eigenbasis, write the planes."""
    w = 8 if prec == 0 else 4
    return w * (2 * nx * ny * nz + max(nx, ny) ** 2)


def fdm_flops_per_step(nx, ny, nz, d3, equilibrium=False, patches=False):
    """Fast-diagonalisation flops of one step: 4 n2 (n_x + n_y) per real plane and solve
    (two GEMM passes each way); solves: V, psi, phi, P and d velocity components (the
    equilibrium system: V, psi, phi), and with electrode patches a second V solve."""
    n2 = nx * ny
    solves = (3 if equilibrium else 4 + (3 if d3 else 2)) + (1 if patches else 0)
    return 4.0 * n2 * (nx + ny) * nz * solves


def warmstart_arm(args):
    """Learned warm start of the equilibrium system (Sec. 2.4, FP64 pseudo-time march): steps and
    wall time to the criterion, warm vs cold, and the error of both against a judge (the cold start
    run to a tolerance ten times tighter).  Opt-in; minutes of GPU time."""
    import numpy as np
    import torch
    import workloads
    from paper_2305_09020_gb300 import native, warmstart
    stream = torch.cuda.Stream()
    tol, cap, every = args.ws_tol, args.ws_cap, 500
    # 8x4 elements of order 6: on the 16x8 order-8 mesh the march at dt 1e-3 left 137 of 164 cold
    # runs above 1e-3 after 10000 steps and 33 of 200 diverged, so no equal-accuracy comparison
    ex, ey, order = 8, 4, 6
    train = warmstart.equilibrium_runs(workloads.warmstart2d(args.ws_train, 1, ex, ey, order))
    test = warmstart.equilibrium_runs(workloads.warmstart2d(args.ws_test, 10001, ex, ey, order))
    t0 = time.perf_counter()
    f_tr, y_tr, st_tr = warmstart.generate(train, tol, cap, every, precision=native.PF_FP64, stream=stream.cuda_stream)
    t_gen = time.perf_counter() - t0
    no = warmstart.make_operator(f_tr, train[0].mesh, seed=0, stream=stream.cuda_stream)
    t0 = time.perf_counter()
    losses = no.train(f_tr, y_tr, batch=64, epochs=args.ws_epochs, lr=1e-3, seed=0)
    t_train = time.perf_counter() - t0
    res = warmstart.evaluate(no, test, tol, cap, every, precision=native.PF_FP64, stream=stream.cuda_stream,
                             judge_tol=tol / 10, judge_steps=4 * cap)
    no.close()
    ec, ew = np.array(res["cold"]["err"]), np.array(res["warm"]["err"])
    same = ew <= 3.0 * ec + 1e-4
    sc, sw = np.array(res["cold"]["steps"]), np.array(res["warm"]["steps"])
    for k in ("cold", "warm"):
        res[k].pop("steps")
        res[k].pop("err")
    line = {"metric": "time-to-equilibrium warm vs cold", "unit": "s", "higher_is_better": False,
            "value": res["warm"]["run_s"], "cold_value": res["cold"]["run_s"],
            "criterion": f"max|phi^(n+1) - phi^n| / dt < {tol:g} (equilibrium system, pseudo-time), exit on the "
                         f"device per run, cap {cap} steps; judge: the cold start to {tol / 10:g}",
            "config": {"workload": f"warm-start ensemble: {ex}x{ey} elements order {order}, V~U(0,3), eps ratio logU(2,20), "
                                   "drop radius U(0.15,0.35) on the wall, eta 0.02; equilibrium system, dt 1e-3, "
                                   "mobility 3e-3, FP64",
                       "train_runs": len(train), "test_runs": len(test), "seeds": "train 1, test 10001",
                       "network": "3-128-384-8192 tanh MLP, 128x64 grid, bilinear to GLL nodes, BF16 weights; "
                                  "prediction shifted on the device to each run's phase mass"},
            "cold": res["cold"], "warm": res["warm"], "judge": res["judge"],
            "warm_runs_at_the_judges_equilibrium": float(same.mean()),
            "steps_median_where_both_agree": {"cold": float(np.median(sc[same])) if same.any() else None,
                                              "warm": float(np.median(sw[same])) if same.any() else None},
            "final_phi_rel_diff": res["final_phi_rel_diff_warm_vs_cold"],
            "train": {"generation_s": t_gen, "training_s": t_train, "epochs": args.ws_epochs,
                      "loss_first": float(losses[0]), "loss_last": float(losses[-1]),
                      "train_runs_reaching_tol": int((st_tr > 0).sum())}}
    print(json.dumps(line))
    return 0


# timed oracle steps of the CPU baseline per workload (about 10-30 s of host work)
ORACLE_STEPS = {"layers3d": 10, "droplet3d": 10, "electrode_array3d": 5, "patches2d": 10}


def fp64_leg(args, wl, dof, prec, gemm_choice, fused_y, fft_tile, stream, flush, barrier):
    """The FP64 path on the same workload: its rate (graph replays, L2 flushed between steps), and
    the per-field relative L2 difference of the mixed path (the timed variant pinned) after
    args.err_steps steps from the same initial state.  The FP64 path is itself held to 1e-11 of
    the FP64 oracle by the parity tests."""
    import numpy as np
    import torch
    from paper_2305_09020_gb300 import native
    ALL_FIELDS = (native.PF_FIELD_V | native.PF_FIELD_E | native.PF_FIELD_PHI | native.PF_FIELD_PSI |
                  native.PF_FIELD_P | native.PF_FIELD_U)
    h64 = native.from_workload(wl, precision=native.PF_FP64, stream=stream.cuda_stream)
    hm = native.from_workload(wl, precision=prec, stream=stream.cuda_stream)
    hm.set_variant(gemm_choice, fuse_y=bool(fused_y), tile=fft_tile)
    n = max(1, args.err_steps)
    h64.step(n)
    hm.step(n)
    f64, fm = h64.get(ALL_FIELDS), hm.get(ALL_FIELDS)
    hm.close()
    err = {}
    for k in f64:
        nrm = float(np.linalg.norm(f64[k]))
        if nrm > 0:
            err[k] = float(np.linalg.norm(fm[k] - f64[k]) / nrm)
    k64 = 3
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(k64)]
    barrier()
    for k in range(k64):
        with torch.cuda.stream(stream):
            flush.fill_(k & 255)
        ev[k][0].record(stream)
        h64.step(1)
        ev[k][1].record(stream)
    barrier()
    ms64 = sum(a.elapsed_time(b) for a, b in ev) / k64
    h64.close()
    return {"value": dof / (ms64 * 1e-3), "unit": UNIT, "ms_per_step": ms64, "steps": k64,
            "variant": "k_oz_split + k_gemm_oz (FP64 default: exact digit products on the tensor cores)",
            "err_steps": n,
            "mixed_rel_l2_vs_fp64": err,
            "note": "relative L2 per field of the mixed path against the FP64 GPU path after err_steps steps "
                    "from the same initial state; the FP64 path matches the FP64 oracle to 1e-11 (tests)"}


def ensemble_arm(args):
    """The batched ensemble of 256 uneven 2D runs: DOF-steps/s of whole-ensemble steps (one CUDA
    graph per step, groups on concurrent streams), then a bounded run to equilibrium with the
    per-run exit on the device (max|u| < tol, checked after every step)."""
    import numpy as np
    import torch
    import workloads
    from paper_2305_09020_gb300 import native
    dev = torch.device("cuda", 0)
    stream = torch.cuda.Stream(device=dev)
    runs = workloads.ensemble2d()
    prec = {"mixed": native.PF_MIXED, "mixed_simt": native.PF_MIXED_SIMT, "fp64": native.PF_FP64}[args.precision]
    dofs = [(w.mesh.ex * w.mesh.order) * (w.mesh.ey * w.mesh.order + 1) for w in runs]
    b = native.Batch(runs, precision=prec, stream=stream.cuda_stream)
    ngroups = b.groups()[0]
    b.step(args.warmup)
    tune = b.autotune(steps=2)
    b.step(2)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    torch.cuda.synchronize(dev)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    clk = ClockSampler(0)
    for k in range(args.steps):
        with torch.cuda.stream(stream):
            flush.fill_(k & 255)
        ev[k][0].record(stream)
        b.step(1)
        ev[k][1].record(stream)
    torch.cuda.synchronize(dev)
    clocks = clk.stop()
    ms = sum(a.elapsed_time(c) for a, c in ev)
    value = sum(dofs) * args.steps / (ms * 1e-3)
    # bounded run to equilibrium: how many runs exit below tol within the cap, and the wall time
    tol, cap = args.ens_tol, args.ens_cap
    t0 = time.perf_counter()
    steps = b.run_to_equilibrium(tol=tol, max_steps=b_steps_taken(args) + cap, check_every=200)
    t_eq = time.perf_counter() - t0
    b.close()
    done = steps[steps > 0]
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64" if prec == native.PF_FP64 else "f32", "data": "synthetic",
            "config": {"workload": WORKLOADS["ensemble2d"], "runs": len(runs), "groups": ngroups,
                       "dof_per_step": int(sum(dofs)), "precision": args.precision,
                       "l2": "flushed between timed steps (256 MiB write)",
                       "group_transform_ms": [round(float(x), 4) for x in tune]},
            "clocks": clocks,
            "run_to_equilibrium": {"tol": tol, "cap_steps": cap, "runs_below_tol": int(done.size),
                                   "diverged": int((steps == -2).sum()), "wall_s": t_eq,
                                   "exit_step_median": float(np.median(done)) if done.size else None,
                                   "criterion": "max|u| < tol per run, checked on the device after every step; "
                                                "a run that exits is frozen"}}
    print(json.dumps(line))
    return 0


def b_steps_taken(args):
    """Steps the ensemble has taken before its run to equilibrium: warm-up, autotuning
    (6 variants x (2 + 1), rounded to even), 2 steady, the timed steps."""
    return args.warmup + 18 + 2 + args.steps


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--precision", default="mixed", choices=["mixed", "mixed_simt", "fp64"])
    ap.add_argument("--workload", default="layers3d", choices=sorted(WORKLOADS),
                    help="layers3d (the default bench line), droplet3d, or the electrode workloads")
    ap.add_argument("--skip-extras", action="store_true", help="only the timed region (for profilers)")
    ap.add_argument("--no-cpu-baseline", action="store_true", help="skip the timed oracle sample")
    ap.add_argument("--no-fp64", action="store_true", help="skip the FP64 rate and the error against it")
    ap.add_argument("--err-steps", type=int, default=20, help="steps of the mixed-vs-FP64 error comparison")
    ap.add_argument("--ens-tol", type=float, default=1e-6, help="ensemble2d: equilibrium tolerance on max|u|")
    ap.add_argument("--ens-cap", type=int, default=2000, help="ensemble2d: steps of the bounded run to equilibrium")
    ap.add_argument("--nz", type=int, default=0,
                    help="override the workload's Fourier plane count (small profiler captures only)")
    ap.add_argument("--variant", type=int, default=None,
                    help="pin the transform variant (a PF_GEMM_* code) instead of autotuning")
    ap.add_argument("--fused-y", type=int, default=0, help="with --variant: run the y pair fused (1) or not (0)")
    ap.add_argument("--fft-tile", type=int, default=0, help="with --variant: pencils per z-transform block (0: heuristic)")
    ap.add_argument("--warmstart", action="store_true", help="learned warm start study instead (minutes)")
    ap.add_argument("--ws-train", type=int, default=1000)
    ap.add_argument("--ws-test", type=int, default=200)
    ap.add_argument("--ws-tol", type=float, default=1e-3)
    ap.add_argument("--ws-cap", type=int, default=20000)
    ap.add_argument("--ws-epochs", type=int, default=300)
    args = ap.parse_args()
    if args.impl == "reference":
        return reference_arm(args)
    if args.warmstart:
        return warmstart_arm(args)
    if args.warmup < 3:
        raise SystemExit("at least 3 warm-up steps")
    if args.workload == "ensemble2d":
        return ensemble_arm(args)

    import numpy as np
    import torch
    import torch.distributed as dist
    import workloads
    from paper_2305_09020_gb300 import native, replicas

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    dev = torch.device("cuda", local)
    stream = torch.cuda.Stream(device=dev)
    prec = {"mixed": native.PF_MIXED, "mixed_simt": native.PF_MIXED_SIMT, "fp64": native.PF_FP64}[args.precision]
    wl = make_workload(args.workload)
    if args.nz > 0:
        wl.mesh.nz = args.nz
    m = wl.mesh
    nx, ny, nz = m.ex * m.order, m.ey * m.order + 1, m.nz
    dof = nx * ny * nz
    h = native.from_workload(wl, precision=prec, stream=stream.cuda_stream)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)

    def barrier():
        torch.cuda.synchronize(dev)
        if world > 1:
            dist.barrier()

    h.step(args.warmup)
    if args.variant is None:
        tuned, _ = h.autotune(steps=5)   # fastest transform variant, y pair, z-transform tile (advances the run)
        gemm_choice, fft_tile, fused_y = tuned % 1000, (tuned // 1000) % 100, tuned // 100000
    else:
        h.set_variant(args.variant, fuse_y=bool(args.fused_y), tile=args.fft_tile)
        gemm_choice, fft_tile, fused_y = args.variant, args.fft_tile, args.fused_y
    h.step(2)
    barrier()
    launches0 = h.profile_read()
    clk = ClockSampler(local)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    barrier()
    torch.cuda.cudart().cudaProfilerStart()    # profilers started with --profile-from-start off see only this
    for k in range(args.steps):
        with torch.cuda.stream(stream):
            flush.fill_(k & 255)               # L2 flush between timed steps (not timed)
        ev[k][0].record(stream)
        h.step(1)
        ev[k][1].record(stream)
    barrier()
    torch.cuda.cudart().cudaProfilerStop()
    clocks = clk.stop()
    ms = sum(a.elapsed_time(b) for a, b in ev)
    launches1 = h.profile_read()
    gpu_launches = sum(launches1[k][1] - launches0[k][1] for k in launches1)
    ms = replicas.max_over_ranks(ms, dev)                       # the slowest replica's time
    units = replicas.gather_counts(dof * args.steps, dev)      # DOF-steps of every replica
    value = replicas.job_rate(units, ms * 1e-3)

    extras = {}
    if not args.skip_extras:
        # per-class device time of the same step, CUDA events on the library's stream
        h.profile(True)
        for k in range(args.steps):
            with torch.cuda.stream(stream):
                flush.fill_(k & 255)
            h.step(1)
        cls = h.profile_read()
        h.profile(False)
        tot = sum(v[0] for v in cls.values())
        top = max(cls, key=lambda k: cls[k][0])
        pk, src = peaks()
        props = torch.cuda.get_device_properties(dev)
        mp = native.measure_peaks()          # this GPU, now: TF32 tensor, FP32 FFMA, FP64 DFMA
        extras["measured_peaks"] = {**{k: round(v, 1) for k, v in mp.items()}, "sms": props.multi_processor_count,
                                    "how": "pf_measure_peaks: tcgen05.mma kind::tf32 128x256x8 loop, one CTA per "
                                           "SM; 8 independent FFMA / DFMA chains per thread; best of 5 launches"}
        per_launch_ms = cls[top][0] / max(1, cls[top][1] - launches1[top][1])
        roof = None
        if top == "gemm":
            flops = fdm_flops_per_step(nx, ny, nz, nz > 1, bool(getattr(wl.scheme, "equilibrium", False)),
                                       wl.vbc.bottom_kind == workloads.BC_PATCHES) * args.steps
            nlaunch = cls["gemm"][1] - launches1["gemm"][1]
            achieved = flops / nlaunch / (per_launch_ms * 1e-3) / 1e12
            if prec == native.PF_MIXED and gemm_choice == 0:
                # 3xTF32: three TF32 MMAs per FP32 product, so the FP32 GEMM's peak is a third of TF32's
                peak = mp["tf32_tflops"] / 3.0
                roof = {"bound": "tensor", "kernel": "k_gemm_tc (3xTF32 tcgen05 fast-diagonalisation transforms)",
                        "peak_source": f"measured TF32 tensor peak {mp['tf32_tflops']:.0f} TFLOP/s / 3 (three TF32 "
                                       "MMAs per FP32 product); achieved counts the FP32 GEMM flops 2MNK"}
            elif prec == native.PF_MIXED and gemm_choice == 8:
                # psi and phi (2 solves) on the FP32 FMA pipe, the others on the tensor cores: the peak
                # of the mix is the flop-weighted harmonic mean of the two peaks
                eq = bool(getattr(wl.scheme, "equilibrium", False))
                n_all = (3 if eq else 4 + (3 if nz > 1 else 2))
                f_simt = 2.0 / n_all
                peak = 1.0 / (f_simt / mp["fp32_tflops"] + (1.0 - f_simt) / (mp["tf32_tflops"] / 3.0))
                roof = {"bound": "tensor", "kernel": "k_gemm_tc + k_gemm_cp (hybrid: psi, phi on FP32 FMA; "
                                                     "V, P, u on 3xTF32 tcgen05)",
                        "peak_source": f"flop-weighted harmonic mean of the measured FP32 FFMA peak "
                                       f"({mp['fp32_tflops']:.1f}) for {2}/{n_all} of the solves and the "
                                       f"measured TF32 peak / 3 ({mp['tf32_tflops'] / 3.0:.0f}) for the rest"}
            elif prec != native.PF_FP64:
                peak = mp["fp32_tflops"]
                roof = {"bound": "alu", "kernel": transform_kernel(gemm_choice, fused_y) + " (FP32 SIMT transforms)",
                        "peak_source": "measured FP32 FFMA peak of this GPU"}
            else:
                peak = mp["fp64_tflops"]
                kind = " (FP64 by digit products)" if gemm_choice == native.PF_GEMM_DIGITS else " (FP64 SIMT transforms)"
                roof = {"bound": "alu", "kernel": transform_kernel(gemm_choice, fused_y) + kind,
                        "peak_source": "measured FP64 DFMA peak of this GPU"}
            traffic = TRANSFORM_DRAM_BYTES_PER_LAUNCH.get((args.workload, args.precision, gemm_choice, fused_y))
            roof.update({"achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
                         "launches_per_step": nlaunch / args.steps, "ms_per_launch": per_launch_ms,
                         "traffic": traffic,
                         "traffic_note": None if traffic is None else
                         "DRAM bytes per transform launch (ncu dram__bytes_read.sum + dram__bytes_write.sum, "
                         "mean over one solve's launches on this workload, profiles/; layers3d captured with "
                         "128 planes and scaled to 256 by the rows processed); algorithmic "
                         f"{transform_bytes_per_launch(nx, ny, nz, prec):.3e} B per launch"})
        else:
            roof = {"bound": "hbm", "kernel": top, "achieved": None, "peak": pk["hbm_gbs"], "unit": "GB/s",
                    "frac": None, "traffic": None, "peak_source": src}
        extras["roofline"] = roof
        extras["kernel_share"] = {k: round(v[0] / tot, 4) for k, v in cls.items() if v[0] > 0}

        # end to end through the C-ABI with host buffers: set phi, u from pinned host memory,
        # step, read V, phi, P, u back into pinned host memory
        # The state fields phi, u go host -> device and back through one pinned buffer (the next
        # step's input is the last step's output, no host-side copy); V, P come back into another.
        n_e2e = min(args.steps, 20)
        hio = torch.empty(4 * dof, dtype=torch.float64, pin_memory=True).numpy()
        hvp = torch.empty(2 * dof, dtype=torch.float64, pin_memory=True).numpy()
        mask_io = native.PF_FIELD_PHI | native.PF_FIELD_U
        mask_vp = native.PF_FIELD_V | native.PF_FIELD_P
        h.get_into(mask_io, hio)
        barrier()
        t0 = time.perf_counter()
        for _ in range(n_e2e):
            h.set(mask_io, hio)
            h.step(1)
            h.get_into(mask_vp, hvp)
            h.get_into(mask_io, hio)
        barrier()
        te = time.perf_counter() - t0
        extras["e2e"] = {"value": dof * n_e2e * world / te, "unit": UNIT,
                         "h2d_bytes_per_step": int(hio.nbytes), "d2h_bytes_per_step": int(hio.nbytes + hvp.nbytes),
                         "steps": n_e2e, "what": "pf_set_fields(phi,u) + pf_step(1) + pf_get_fields(V,P) + "
                                                 "pf_get_fields(phi,u), pinned host buffers, no host-side copies"}
        if prec != native.PF_FP64 and not args.no_fp64:
            extras["fp64"] = fp64_leg(args, wl, dof, prec, gemm_choice, fused_y, fft_tile, stream, flush, barrier)
            extras["fp64"]["mixed_speedup"] = (dof * args.steps / (ms * 1e-3)) / extras["fp64"]["value"]
        if rank == 0 and world == 1 and not args.no_cpu_baseline:
            val, secs, desc = oracle_sample(ORACLE_STEPS.get(args.workload, 10), 2, args.workload)
            extras["cpu_baseline"] = {"value": val, "unit": UNIT, "cores": ORACLE_THREADS, "host_cpus": os.cpu_count(),
                                      "kind": "oracle", "sample": desc}
    h.close()

    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64" if prec == native.PF_FP64 else "f32",
            "data": "synthetic",
            "config": {"workload": WORKLOADS[args.workload] + (f" (Nz overridden to {nz})" if args.nz > 0 else ""),
                       "dof_per_field": dof, "fourier_coeffs_per_field": nx * ny * (nz // 2 + 1),
                       "precision": args.precision, "l2": "flushed between timed steps (256 MiB write)",
                       "fdm_gemm": {0: "tcgen05 3xTF32 (psi, phi: 2-slice TMEM groups, V, P, u: 8-slice groups; correction "
                                       "products in a per-tile region)", 1: "whole solve per plane in shared memory (SIMT)",
                                    2: "SIMT 32x64 tiles", 3: "SIMT 64x64 tiles, cp.async pipeline",
                                    4: "SIMT 32x32 tiles, cp.async pipeline", 5: "SIMT 32x64 tiles, cp.async pipeline",
                                    6: "whole solve per plane on a 4-block cluster (SIMT, distributed shared memory)",
                                    7: "whole solve per plane on a 2-block cluster (SIMT, distributed shared memory)",
                                    8: "hybrid: psi, phi solves SIMT 64x64 cp.async, V, P, u tcgen05 3xTF32 with "
                                       "4-slice accumulation groups",
                                    9: "exact products of 8-bit digits on the tensor cores"}.get(gemm_choice, f"SIMT {gemm_choice}x{gemm_choice} tiles")
                                   + (", y pair fused" if fused_y and gemm_choice not in (0, 1, 6, 7) else "")
                                   + (" (autotuned)" if args.variant is None else " (pinned)"),
                       "fft_pencils_per_block": fft_tile,
                       "parallelism": f"replicas x{world}"},
            "gpu_launches": gpu_launches, "clocks": clocks}
    line.update(extras)
    if rank == 0:
        print(json.dumps(line))
    if world > 1:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())

#!/usr/bin/env python3
"""Benchmark: DOF x timesteps / s of the tau-preconditioned GMRES time stepper.

Workload (default): d = 2, n = 511 x 511 on [-10,10]^2, rho = 2, dt = 0.005, u0 = sech(x)sech(y)e^{i(x+y)},
alpha in {1.2, 1.5, 1.9} (three independent instances), tol 1e-10.  One bench step advances all three
instances by one time step (a GMRES solve each, all three through one rfnse_batch_run call) in the mixed
form (FP32 transforms inside FGMRES, FP64 Arnoldi/Givens, the refinement residual accurate to about
1e-14); the plain FP64 form is timed the same way and reported
beside it, with the difference between the two trajectories.  DOF = complex grid unknowns.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                  [--workload 2d|3d|1d|batched|adjoint|comparators|omega] [--instances K]
  python bench.py --alu-probe | --arnoldi-probe

The metric names two halves, and the default line carries both: the 2-D workload above (the line's
own value) and, under "config_3d", the 3-D workload (n = 255^3 on [-8,8]^3, alpha = 1.7, rho = 1,
dt = 0.01, u0 = exp(-|x|^2/2)e^{ix_1}, tol 1e-8), each with the FP64 form beside the mixed one, the
per-step error of both forms against the CPU oracle's trajectory from the same u^0 ("err_vs_oracle"),
an end-to-end figure with host buffers ("e2e") and the oracle's own throughput on the host cores, all
cores and (2-D) one core ("cpu_baseline").  The roofline objects are the three largest kernel classes
of each workload's step, every class timed launch by launch (CUDA events) in a further serial run
with host-driven loops.  --instances K runs K 511^2 instances instead of three (the throughput
saturates from about 6 on); --no-3d leaves the 3-D half out; --arnoldi-probe times the Arnoldi kernel
alone per column j; --alu-probe measures the FP64 and FP32 FMA rates.

Other workloads: 3d (255^3, mixed), 1d (n = 1023), batched (64 independent 2-D instances with grids
drawn from {127, 255, 511}^2: one step = one graph launch advancing all of them), adjoint (255^2,
20 steps, FP64: one step = a taped forward run plus its reverse pass, dL/du0 and dL/drho),
comparators (255^2: the same run with the sine-transform preconditioner, Strang's circulant and none),
omega (Fig. 1: tau-GMRES iterations versus the TBAN parameter w for five alpha, 1-D n = 2047).

Multi-GPU (torchrun): every rank advances its own copy of the three instances (independent problems,
no collective on the data path; weak scaling); value = all ranks' DOF x steps / max rank time.
--impl reference times the CPU oracle (test infrastructure) on the host cores, rank 0 only.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
from concurrent.futures import ThreadPoolExecutor
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

import workloads as W  # noqa: E402

METRIC = "DOF*timesteps/s"
UNIT = "DOF*timesteps/s"
FP64_ALU_PEAK_FLOPS = 152 * 2 * 2 * 2.07e9   # 152 SMs x 2 FP64 FMA/clk x 2 flop x 2.07 GHz
FP32_ALU_PEAK_FLOPS = 152 * 128 * 2 * 2.07e9  # 152 SMs x 128 FP32 FMA/clk x 2 flop x 2.07 GHz
NOMINAL_HBM_GBS = 7900.0                      # GB300 HBM3e nominal bandwidth (context beside the measured copy)
CSRC = os.path.join(ROOT, "paper_2410_03643_gb300", "csrc")


def measured_hbm_gbs():
    """The machine's measured copy bandwidth (MEASURED_PEAKS.json), else the recipe's fallback."""
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return float(json.load(fh)["hbm_gbs"]), "measured"
    except (OSError, ValueError, KeyError):
        return 6800.0, "fallback"


# Kernel classes timed launch by launch for the roofline objects: rfnse_profile kind (OR of the pass
# flags, +256 for FP32 passes, +1024 for the double-float residual passes, 2048 for the Arnoldi kernel),
# the roofline that bounds the class, its description, and the sources its kernels are compiled from.
_PASS_SRC = ("passes.cuh", "fft_fixed.cuh", "fft_line.cuh", "cplx.cuh")
_DF_SRC = ("toep_df.cu", "dfloat.cuh", "fft_fixed.cuh", "cplx.cuh", "passes.cuh")
KERNEL_CLASSES = {
    "arnoldi": (2048, "alu", "k_mgs_step (cooperative MGS + Givens + convergence test, one launch per Arnoldi "
                             "step)", ("control.cu", "coop.cuh")),
    "fp32_fused_x": (256 | 2 | 8 | 16, "hbm", "line pass <float, F_DST|F_DSCALE|F_TOEP_X> (inverse DST x + "
                                              "(wI+D) sub-solve + Toeplitz x)", _PASS_SRC),
    "fp32_dst": (256 | 2, "hbm", "line pass <float, F_DST> (DST x with the Arnoldi scaling folded in; DST y in 3-D)",
                 _PASS_SRC),
    "fp32_dst_lam": (256 | 2 | 4, "hbm", "line pass <float, F_DST|F_LAM> (DST, divide by (w + i Lambda), DST; last "
                                         "axis)", _PASS_SRC),
    "fp32_toep_acc": (256 | 32, "hbm", "line pass <float, F_TOEP_ACC> (Toeplitz y / z, accumulated)", _PASS_SRC),
    "fp32_all_1d": (256 | 2 | 4 | 8 | 16, "hbm", "line pass <float, all flags> (1-D preconditioner + product)",
                    _PASS_SRC),
    "df_toep_x": (1024 | 16, "hbm", "k_toeplitz_df<F_TOEP_X> (residual Toeplitz x, double-float FFTs)", _DF_SRC),
    "df_toep_acc": (1024 | 32, "hbm", "k_toeplitz_df<F_TOEP_ACC> (residual Toeplitz y / z, double-float FFTs)",
                    _DF_SRC),
}
# The 3-D workload (2^20 points and more) runs these classes as tensor-core digit passes, some of them two
# launches: its descriptions and sources.
_DIG_SRC = ("digit.cu", "digit.cuh", "tc05.cuh")
_DIG32_SRC = ("digit32.cu", "digit.cuh", "tc05.cuh")
CLASSES_3D = {
    "fp32_fused_x": ("k_digit32<F_DST|F_DSCALE>, k_digit32<F_TOEP_X> (inverse S x + (wI+D) sub-solve; Toeplitz x)",
                     _DIG32_SRC),
    "fp32_dst": ("line pass <float, F_INSCALE|F_DST> (S x with the Arnoldi scaling folded in), k_digit32<F_DST> (S y)",
                 _DIG32_SRC + _PASS_SRC),
    "fp32_dst_lam": ("k_digit32<F_DST|F_LAM>, k_digit32<F_DST> (S, divide by (w + i Lambda); S; last axis)",
                     _DIG32_SRC),
    "fp32_toep_acc": ("k_digit32<F_TOEP_ACC> (Toeplitz y / z, accumulated)", _DIG32_SRC),
    "df_toep_x": ("k_digit<F_TOEP_X> (residual Toeplitz x, FP64 digits)", _DIG_SRC),
    "df_toep_acc": ("k_digit<F_TOEP_ACC> (residual Toeplitz y / z, FP64 digits)", _DIG_SRC),
}
PROFILED = {
    "2d": ("arnoldi", "fp32_fused_x", "fp32_dst", "fp32_dst_lam", "fp32_toep_acc", "df_toep_x", "df_toep_acc"),
    "3d": ("arnoldi", "fp32_fused_x", "fp32_dst", "fp32_dst_lam", "fp32_toep_acc", "df_toep_x", "df_toep_acc"),
    "1d": ("arnoldi", "fp32_all_1d", "df_toep_x"),
}

# dram__bytes_read.sum + dram__bytes_write.sum per launch of a class on a workload: the mean over the
# launches of the class captured by ncu in `bench.py --kernel-case 2d|3d` (one mixed solve of the
# workload's grid, the same kernels and vector sizes), with the digest of the class's sources when the
# capture was taken: once a source has changed the figure no longer describes the kernel and the line
# reports traffic null.
TRAFFIC = {
    ("2d", "arnoldi"): (10512064, "2f0ff00eb74a"),
    ("2d", "fp32_fused_x"): (5277952, "bc9364c29794"),
    ("2d", "fp32_dst"): (4206848, "bc9364c29794"),
    ("2d", "fp32_dst_lam"): (4212480, "bc9364c29794"),
    ("2d", "fp32_toep_acc"): (8398976, "bc9364c29794"),
    ("2d", "df_toep_x"): (6342912, "dcc06e68e64c"),
    ("2d", "df_toep_acc"): (8433408, "dcc06e68e64c"),
    ("3d", "arnoldi"): (1280290602, "2f0ff00eb74a"),
    ("3d", "fp32_fused_x"): (654136405, "00ca8716fabd"),
    ("3d", "fp32_dst"): (340353095, "cf52189611c3"),
    ("3d", "fp32_dst_lam"): (568429354, "00ca8716fabd"),
    ("3d", "fp32_toep_acc"): (550043477, "00ca8716fabd"),
    ("3d", "df_toep_x"): (765136512, "839b01b96df8"),
    ("3d", "df_toep_acc"): (749329152, "839b01b96df8"),
}


def source_digest(files) -> str:
    import hashlib
    h = hashlib.sha256()
    for f in files:
        with open(os.path.join(CSRC, f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:12]


def traffic_for(workload_name: str, cls: str):
    """(bytes per launch or None, note)."""
    rec = TRAFFIC.get((workload_name, cls))
    if rec is None:
        return None, "no ncu capture of this class on this workload"
    value, digest = rec
    srcs = CLASSES_3D[cls][1] if workload_name == "3d" and cls in CLASSES_3D else KERNEL_CLASSES[cls][3]
    if digest != source_digest(srcs):
        return None, "stale: the kernel's sources changed since the ncu capture"
    return value, "ncu dram__bytes_read.sum + dram__bytes_write.sum per launch"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="2d", choices=["2d", "3d", "1d", "batched", "adjoint", "comparators", "omega"])
    ap.add_argument("--no-fp64", action="store_true", help="skip the plain FP64 comparison run")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU-oracle baseline")
    ap.add_argument("--serial", action="store_true", help="advance the instances one after another on one stream")
    ap.add_argument("--host-loop", action="store_true",
                    help="drive the GMRES loops from the host (no CUDA graphs; same kernels, for kernel profilers)")
    ap.add_argument("--alu-probe", action="store_true",
                    help="only measure the FP64 and FP32 FMA rates of the GPU and print them")
    ap.add_argument("--arnoldi-probe", action="store_true",
                    help="only time the cooperative Arnoldi kernel (MGS + Givens) per column j on the 2-D and "
                         "3-D grid sizes and print the times")
    ap.add_argument("--no-autotune", action="store_true", help="keep the default launch geometry of the line passes")
    ap.add_argument("--arnoldi-grid", type=int, default=0,
                    help="force the Arnoldi kernel's launch after tuning (rfnse_set_arnoldi_grid: > 0 blocks of "
                         "the grid-wide kernel, -8 / -16 one cluster of that many CTAs; 0 = as tuned)")
    ap.add_argument("--no-lockstep", action="store_true",
                    help="batches run one CUDA graph branch per instance instead of the lock-step launches")
    ap.add_argument("--lockstep", action="store_true",
                    help="batches run in lock-step even below the default instance count (mixed form)")
    ap.add_argument("--no-3d", action="store_true",
                    help="default 2d workload: leave out the 3-D 255^3 half of the metric (config_3d)")
    ap.add_argument("--kernel-case", default=None, choices=["2d", "3d"],
                    help="only run a small case for kernel profilers: one mixed solve of the workload's grid "
                         "with host-driven loops, restart 2 and at most 4 Arnoldi steps (a 255^3 case holds "
                         "about 4 GB on the device), then exit")
    ap.add_argument("--cpu-sample", default=None, help=argparse.SUPPRESS)
    ap.add_argument("--cpu-steps", type=int, default=2, help=argparse.SUPPRESS)
    ap.add_argument("--cpu-state", default=None, help=argparse.SUPPRESS)
    ap.add_argument("--instances", type=int, default=3,
                    help="2d workload: number of 511^2 instances advanced together (alphas cycle through "
                         "1.2, 1.5, 1.9); the default 3 is the headline configuration")
    return ap.parse_args()


def workload(name, instances=3):
    """[(problem, u0)] and a description."""
    if name == "2d":
        alphas = [W.CONFIG_2D_ALPHAS[i % len(W.CONFIG_2D_ALPHAS)] for i in range(instances)]
        inst = [W.config_2d(a)[:2] for a in alphas]
        tag = "" if instances == 3 else f"_x{instances}"
        desc = {"workload": "2d_n511x511_alpha{1.2,1.5,1.9}_rho2_dt0.005_tol1e-10" + tag, "d": 2, "n": [511, 511],
                "box": [-10, 10], "alphas": alphas, "instances": instances}
    elif name == "3d":
        p, u0, _ = W.config_3d()
        inst = [(p, u0)]
        desc = {"workload": "3d_n255^3_alpha1.7_rho1_dt0.01_tol1e-8", "d": 3, "n": [255, 255, 255],
                "box": [-8, 8], "alphas": [1.7], "instances": 1}
    elif name == "batched":
        inst, _ = W.config_batched()
        desc = {"workload": "batched_64x2d_n{127,255,511}^2_seed2410_dt0.005_tol1e-10", "d": 2,
                "instances": len(inst), "dof_per_step": int(sum(p.size for p, _ in inst)),
                "sampling": "n_x, n_y iid from {127,255,511}; alpha~U[1.1,1.95]; rho~U[0.5,3]; k~U[-3,3]"}
    else:
        p, u0, _ = W.config_1d()
        inst = [(p, u0)]
        desc = {"workload": "1d_n1023_alpha1.5_rho2_dt0.01_tol1e-10", "d": 1, "n": [1023], "box": [-20, 20],
                "alphas": [1.5], "instances": 1}
    return inst, desc


# --- clocks -------------------------------------------------------------------------------------
class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 50 ms while active."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []
        self.t_on = self.t_off = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
            time.sleep(0.3)
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append((time.time(), line.strip()))

    def mark_on(self):
        self.t_on = time.time()

    def mark_off(self):
        self.t_off = time.time()

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        time.sleep(0.1)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = [l for t, l in self.lines if self.t_on is not None and self.t_on - 0.05 <= t <= self.t_off + 0.05]
        sm, smmax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            f = [x.strip() for x in r.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smmax.append(float(f[2]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smmax) if smmax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# --- distributed helpers ------------------------------------------------------------------------
def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def reduce_max(value: float, world: int, device=None) -> float:
    if world <= 1:
        return value
    import torch
    import torch.distributed as dist
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def weak_value(world: int, units_per_rank: float, steps: int, ms_max: float) -> float:
    """Whole-job throughput under weak scaling: every rank processes the same units per step, the job
    takes the slowest rank's time."""
    return world * units_per_rank * steps / (ms_max * 1e-3)


def barrier(world: int):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


# --- the CPU oracle as the baseline / reference arm ---------------------------------------------
def oracle_sample(inst, nsteps: int):
    """The first `nsteps` + 1 steps of the first instance with the CPU oracle, timing the `nsteps`
    regular steps (n >= 1).  Returns (DOF x steps / s, seconds, steps, [u^1 .. u^{nsteps+1}])."""
    from oracle.scheme import SchemeOracle
    p, u0 = inst[0]
    o = SchemeOracle(p)
    u1, _, _ = o.first_step(u0)
    traj = [u1]
    up, uc = u0, u1
    t0 = time.perf_counter()
    for _ in range(nsteps):
        un, _, _ = o.step(up, uc)
        traj.append(un)
        up, uc = uc, un
    dt = time.perf_counter() - t0
    return p.size * nsteps / dt, dt, nsteps, traj


def host_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


def cpu_model() -> str:
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.startswith("Model name:"):
                return line.split(":", 1)[1].strip()
    except (OSError, subprocess.SubprocessError):
        pass
    import platform
    return platform.processor() or platform.machine()


def cpu_sample_child(args):
    """Child of oracle_single_thread: time args.cpu_steps regular oracle steps from the state in
    args.cpu_state (BLAS limited to one thread by the parent's environment) and print one JSON line."""
    from oracle.scheme import SchemeOracle
    inst, _ = workload(args.cpu_sample, 1)
    p = inst[0][0]
    z = np.load(args.cpu_state)
    up, uc = z["u_prev"], z["u_cur"]
    o = SchemeOracle(p)
    t0 = time.perf_counter()
    for _ in range(args.cpu_steps):
        un, _, _ = o.step(up, uc)
        up, uc = uc, un
    dt = time.perf_counter() - t0
    print(json.dumps({"value": p.size * args.cpu_steps / dt, "seconds": dt, "steps": args.cpu_steps}), flush=True)


def oracle_single_thread(name: str, u_prev, u_cur, steps: int):
    """The oracle on one host core: a child process with every BLAS / OpenMP pool set to one thread,
    timing `steps` regular steps from (u_prev, u_cur).  Returns its JSON record or None."""
    import tempfile
    env = dict(os.environ)
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS", "BLIS_NUM_THREADS",
              "VECLIB_MAXIMUM_THREADS", "NUMEXPR_NUM_THREADS"):
        env[k] = "1"
    with tempfile.TemporaryDirectory() as tmp:
        path = os.path.join(tmp, "state.npz")
        np.savez(path, u_prev=u_prev, u_cur=u_cur)
        try:
            r = subprocess.run([sys.executable, os.path.abspath(__file__), "--cpu-sample", name, "--cpu-steps",
                                str(steps), "--cpu-state", path], env=env, capture_output=True, text=True,
                               timeout=900)
        except subprocess.SubprocessError:
            return None
    for line in reversed(r.stdout.splitlines()):
        if line.startswith("{"):
            return json.loads(line)
    return None


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return
    inst, desc = workload(args.workload, args.instances)
    from oracle.scheme import SchemeOracle
    # one bench step = one time step of one instance (instances visited in turn), CPU oracle
    states = []
    for p, u0 in inst:
        o = SchemeOracle(p)
        u1, _, _ = o.first_step(u0)
        states.append([o, u0, u1])
    k = 0

    def one():
        nonlocal k
        st = states[k % len(states)]
        o, up, uc = st
        un, _, _ = o.step(up, uc)
        st[1], st[2] = uc, un
        k += 1
        return o.p.size

    for _ in range(args.warmup):
        one()
    dof = 0
    t0 = time.perf_counter()
    for _ in range(args.steps):
        dof += one()
    dt = time.perf_counter() - t0
    value = dof / dt
    cores = host_cores()
    out = {"metric": METRIC, "value": value, "unit": UNIT, "impl": "reference", "n_gpus": args.gpus,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / max(args.steps, 1),
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
           "data": "synthetic (closed-form initial data of the paper's shape)",
           "config": dict(desc, sample="one time step of one alpha instance per bench step"),
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "cpu": cpu_model(),
                            "sample": f"{args.steps} time steps, instances in turn, numpy/BLAS on {cores} host cores"},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


# --- our CUDA path --------------------------------------------------------------------------------
class Env:
    """What every measurement of the CUDA path shares: torch, the binding, the device and stream, the
    rank layout and the L2-flush buffer."""

    def __init__(self, torch, rfnse, dev, main, rank, world, local):
        self.torch, self.rfnse, self.dev, self.main = torch, rfnse, dev, main
        self.rank, self.world, self.local = rank, world, local
        self.flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)


def roofline_entry(name: str, cls: str, prof, ms_serial: float, nprof: int):
    """The roofline object of one kernel class from its launch-by-launch profile (launches, ms,
    algorithmic flops, algorithmic bytes)."""
    n, pms, fl, by = prof
    kind, bound, desc, _ = KERNEL_CLASSES[cls]
    if name == "3d" and cls in CLASSES_3D:
        desc = CLASSES_3D[cls][0]
    hbm, how = measured_hbm_gbs()
    traffic, tnote = traffic_for(name, cls)
    gbs = by / (pms * 1e-3) / 1e9
    e = {"class": cls, "kernel": desc, "launches": n, "avg_launch_us": 1e3 * pms / n, "total_ms": pms,
         "share_of_step_time": pms / ms_serial if ms_serial > 0 else None,
         "measured": f"CUDA events around every launch of the class (on its stream), serial run of {nprof} "
                     "further bench steps with host-driven loops (the kernels of the graphs)",
         "algorithmic_flops_per_launch": fl / n, "algorithmic_bytes_per_launch": by / n,
         "traffic": (traffic / 1.0) if traffic is not None else None, "traffic_note": tnote}
    if bound == "alu":
        achieved = fl / (pms * 1e-3) / 1e12
        e.update({"bound": "alu", "achieved": achieved, "peak": FP64_ALU_PEAK_FLOPS / 1e12, "unit": "TFLOP/s",
                  "frac": achieved * 1e12 / FP64_ALU_PEAK_FLOPS, "achieved_GBs": gbs, "frac_of_hbm": gbs / hbm,
                  "traffic_GBs": traffic * n / (pms * 1e-3) / 1e9 if traffic is not None else None,
                  "peak_note": "FP64 FMA issue rate: 152 SM x 2 FMA/clk x 2 flop x 2.07 GHz = 1.26 TFLOP/s "
                               "(bench.py --alu-probe measures it); the algorithmic FP64 flops per launch "
                               "(8 (j + 1) + 4 per point) need more time at that rate than its bytes at the "
                               f"copy bandwidth ({how}, beside it)"})
    else:
        e.update({"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                  "frac_of_nominal_hbm": gbs / NOMINAL_HBM_GBS,
                  "traffic_GBs": traffic * n / (pms * 1e-3) / 1e9 if traffic is not None else None,
                  "achieved_TFLOPs": fl / (pms * 1e-3) / 1e12,
                  "peak_note": f"copy bandwidth, {how} (MEASURED_PEAKS.json); algorithmic bytes = every "
                               "operand read once and every result written once"})
        if cls.startswith("df_"):
            e["fp64_equivalent_frac_of_fp64_alu_peak"] = fl / (pms * 1e-3) / FP64_ALU_PEAK_FLOPS
        else:
            e["frac_of_fp32_alu_peak"] = fl / (pms * 1e-3) / FP32_ALU_PEAK_FLOPS
    return e


def rel_errors(got, want):
    return [float(np.linalg.norm((g - w).ravel()) / np.linalg.norm(w.ravel())) for g, w in zip(got, want)]


def measure(args, env: Env, name: str, instances: int, steps: int, warmup: int, oracle_steps: int,
            single_thread_steps: int, e2e_steps: int):
    """One workload through the CUDA path: the mixed form timed (the value), its largest kernel classes
    launch by launch (roofline objects), the FP64 form timed the same way, the per-step error of both
    forms against the CPU oracle, the end-to-end figure through the C ABI with host buffers, and the
    oracle's own throughput on the host cores.  Returns the JSON record."""
    torch, rfnse, dev, main, world, rank = env.torch, env.rfnse, env.dev, env.main, env.world, env.rank
    inst, desc = workload(name, instances)
    concurrent = not args.serial and len(inst) > 1
    pool = ThreadPoolExecutor(max_workers=len(inst)) if concurrent else None
    # several instances advance together through the batch API (one graph launch per step for all);
    # host-driven loops (--host-loop, for kernel profilers) keep one host thread per instance
    use_batch = concurrent and not args.host_loop

    tuning = {}

    def make(precision, device_loop=None, batch=None):
        """The instances in one precision; their line passes autotuned (each grid is timed once per
        process, later contexts reuse the choice) unless --no-autotune."""
        if device_loop is None:
            device_loop = 0 if args.host_loop else 1
        if use_batch if batch is None else batch:
            b = rfnse.Batch([p for p, _ in inst], precision=precision, stream=main, device_loop=device_loop)
            if args.no_lockstep and b.lockstep:
                b.set_lockstep(False)
            if args.lockstep and not b.lockstep and precision == 1:
                b.set_lockstep(True)
            if not args.no_autotune:
                nc, ch = b.autotune(reps=5)
                tuning.setdefault(precision, {"configs": nc, "changed": ch,
                                              "arnoldi_grid": int(b.lib.rfnse_arnoldi_grid(b.ctx[0]))})
            if args.arnoldi_grid:
                for cx in b.ctx:
                    b._check(b.lib.rfnse_set_arnoldi_grid(cx, args.arnoldi_grid), cx)
            for i, (p, u0) in enumerate(inst):
                b.set_state(i, torch.from_numpy(u0.ravel().copy()).to(dev))
            torch.cuda.synchronize()
            return b
        solvers = []
        for p, u0 in inst:
            st = torch.cuda.Stream(device=dev) if concurrent else main
            s = rfnse.Solver(p, precision=precision, stream=st, device_loop=device_loop)
            if not args.no_autotune:
                nc, ch, sp = s.autotune(reps=5)
                tuning.setdefault(precision, {"configs": nc, "changed": ch, "est_speedup": sp,
                                              "arnoldi_grid": int(s.lib.rfnse_arnoldi_grid(s.h))})
            if args.arnoldi_grid:
                s._check(s.lib.rfnse_set_arnoldi_grid(s.h, args.arnoldi_grid))
            s.set_state(torch.from_numpy(u0.ravel().copy()).to(dev))
            solvers.append(s)
        torch.cuda.synchronize()
        return solvers

    def advance(solvers, start_ev=None, serial=False):
        """One bench step: every instance advances one time step (instances in parallel streams)."""
        if isinstance(solvers, rfnse.Batch):
            return [int(v) for v in solvers.run(1)[0][0]]
        if serial or not concurrent:
            return [int(s.run(1)[0][0]) for s in solvers]
        if start_ev is not None:
            for s in solvers:
                s.stream.wait_event(start_ev)
        its = [int(f.result()[0][0]) for f in [pool.submit(s.run, 1) for s in solvers]]
        for s in solvers:
            ev = torch.cuda.Event()
            ev.record(s.stream)
            main.wait_event(ev)
        return its

    def states_of(group):
        if isinstance(group, rfnse.Batch):
            return [group.get_state(i)[1] for i in range(group.count)]
        return [s.get_state()[1] for s in group]

    def close_all(group):
        if isinstance(group, rfnse.Batch):
            group.close()
        else:
            for s in group:
                s.close()

    dof_per_step = sum(p.size for p, _ in inst)

    def timed(solvers, nsteps, nwarm, profile_kind=0, clocks=None, serial=False):
        for _ in range(nwarm):
            advance(solvers, serial=serial)
        torch.cuda.synchronize()
        if profile_kind:
            for s in solvers:
                s.profile(profile_kind)
        launches0 = rfnse.launch_count()
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(nsteps)]
        iters = []
        barrier(world)
        torch.cuda.synchronize()
        if clocks:
            clocks.mark_on()
        for k in range(nsteps):
            env.flush.fill_(float(k))                   # evict L2 between timed steps
            evs[k][0].record(main)
            iters += advance(solvers, evs[k][0], serial=serial)
            evs[k][1].record(main)
        torch.cuda.synchronize()
        if clocks:
            clocks.mark_off()
        barrier(world)
        launches = rfnse.launch_count() - launches0
        ms = sum(a.elapsed_time(b) for a, b in evs)
        prof = None
        if profile_kind:
            tot = [0, 0.0, 0.0, 0.0]
            for s in solvers:
                n, pms, fl, by = s.profile_read()
                tot[0] += n; tot[1] += pms; tot[2] += fl; tot[3] += by
                s.profile(0)
            prof = tot
        return ms, launches, iters, prof

    # headline: mixed form
    mixed = make(1)
    lockstep_note = ("lock-step: every launch of a step covers all instances (work-list line passes, one "
                     "cooperative Gram-Schmidt launch)" if isinstance(mixed, rfnse.Batch) and mixed.lockstep
                     else None)
    clocks = ClockSampler(env.local) if rank == 0 else None
    if clocks:
        clocks.start()
    ms, launches, iters_m, _ = timed(mixed, steps, warmup, clocks=clocks)
    clk = clocks.stop() if clocks else None
    mixed_states = states_of(mixed)   # after warmup + steps, for the FP64 comparison
    close_all(mixed)
    ms_max = reduce_max(ms, world, dev)
    out = {"metric": METRIC, "value": weak_value(world, dof_per_step, steps, ms_max), "unit": UNIT,
           "n_gpus": world, "steps": steps, "warmup": warmup, "ms_per_step": ms_max / steps,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64 (mixed)",
           "data": "synthetic (closed-form initial data of the paper's shape)",
           "config": dict(desc, precision="mixed: FP32 transforms in FGMRES, FP64 Arnoldi/Givens/residual",
                          l2="256 MiB buffer written between timed steps",
                          parallelism=(f"{world} GPU(s), instances replicated per GPU; "
                                       + ("all instances advanced by one batch call per step "
                                          "(rfnse_batch_run: one CUDA graph launch)" if use_batch else
                                          "one CUDA stream and host thread per instance" if concurrent
                                          else "instances in turn on one stream")),
                          control=("host-driven GMRES loops" if args.host_loop
                                   else "device-decided GMRES loops, one CUDA graph per solve"),
                          lockstep=lockstep_note),
           "gpu_launches": launches,
           "iters_per_solve_mean": float(np.mean(iters_m)) if iters_m else None}
    if clk:
        out["clocks"] = clk
    out["autotune"] = ({"mixed": tuning.get(1), "what": "rfnse_autotune: lines per block, FFT threads per line "
                        "and kernel variant of every line-pass configuration, and the Arnoldi kernel's launch "
                        "(arnoldi_grid: > 0 blocks of the grid-wide kernel, < 0 one cluster of that many CTAs), "
                        "chosen by timing (set-up, not timed)"}
                       if not args.no_autotune else None)

    # the largest kernel classes, each timed launch by launch in a further serial run of the same steps
    # with host-driven loops (CUDA events cannot be placed around single kernels inside a running graph;
    # the kernels are the same); in the concurrent region the instances share the SMs, which stretches
    # each launch, so the serial run gives the kernels' own durations
    nprof = max(1, min(steps, 20))
    entries = []
    for cls in PROFILED.get(name, ()):
        prof_solvers = make(1, device_loop=0, batch=False)
        ms_r, _, _, prof = timed(prof_solvers, nprof, min(warmup, 3), profile_kind=KERNEL_CLASSES[cls][0],
                                 serial=True)
        close_all(prof_solvers)
        if prof and prof[0] > 0:
            entries.append(roofline_entry(name, cls, prof, ms_r, nprof))
    entries.sort(key=lambda e: -e["total_ms"])
    for key, e in zip(("roofline", "roofline_second", "roofline_third"), entries):
        out[key] = e
    if entries:
        out["kernel_classes"] = {e["class"]: {"share_of_step_time": e["share_of_step_time"],
                                              "avg_launch_us": e["avg_launch_us"], "frac": e["frac"],
                                              "bound": e["bound"]} for e in entries}

    # plain FP64 form, same protocol, and the distance between the two trajectories
    if not args.no_fp64:
        fp64 = make(0)
        ms64, _, iters64, _ = timed(fp64, steps, warmup)
        ms64 = reduce_max(ms64, world, dev)
        errs = [float(torch.linalg.vector_norm(ua - ub) / torch.linalg.vector_norm(ub))
                for ua, ub in zip(mixed_states, states_of(fp64))]
        out["fp64"] = {"value": weak_value(world, dof_per_step, steps, ms64), "ms_per_step": ms64 / steps,
                       "iters_per_solve_mean": float(np.mean(iters64)) if iters64 else None}
        out["mixed_vs_fp64_rel_l2_after_run"] = max(errs)
        out["mixed_speedup_vs_fp64"] = ms64 / ms_max
        close_all(fp64)
    del mixed_states

    # end to end through the C ABI with host buffers: H2D of the step's inputs, D2H of its result
    if not args.no_e2e and e2e_steps > 0:
        e2e_solvers = make(1, batch=False)
        for s in e2e_solvers:
            s.run(2)  # reach a regular step
        hosts = []
        for s in e2e_solvers:
            up, uc, step = s.get_state()
            pin_up = torch.empty(s.N, dtype=torch.complex128, pin_memory=True)
            pin_uc = torch.empty(s.N, dtype=torch.complex128, pin_memory=True)
            pin_out = torch.empty(s.N, dtype=torch.complex128, pin_memory=True)
            pin_up.copy_(up.cpu())
            pin_uc.copy_(uc.cpu())
            hosts.append([pin_up, pin_uc, pin_out, step])
        torch.cuda.synchronize()
        barrier(world)
        t0 = time.perf_counter()

        def e2e_one(s, h):
            s.set_state_host(h[1].numpy(), h[0].numpy(), h[3])     # H2D of u^{n-1}, u^n
            s.run_host(1, h[2].numpy())                            # step + D2H of u^{n+1}
            h[0], h[1], h[2] = h[1], h[2], h[0]
            h[3] += 1

        for _ in range(e2e_steps):
            if concurrent:
                for f in [pool.submit(e2e_one, s, h) for s, h in zip(e2e_solvers, hosts)]:
                    f.result()
            else:
                for s, h in zip(e2e_solvers, hosts):
                    e2e_one(s, h)
        torch.cuda.synchronize()
        e2e_s = reduce_max(time.perf_counter() - t0, world, dev)
        nb = sum(s.N for s in e2e_solvers) * 16
        out["e2e"] = {"value": weak_value(world, dof_per_step, e2e_steps, 1e3 * e2e_s), "unit": UNIT,
                      "h2d_bytes_per_step": 2 * nb, "d2h_bytes_per_step": nb, "steps": e2e_steps}
        close_all(e2e_solvers)
        del hosts

    # the CPU oracle on the host cores (bounded sample) and the per-step error of both GPU forms against
    # the oracle's trajectory of the first instance (rank 0 at N = 1 only)
    if not args.no_cpu and rank == 0 and world == 1 and oracle_steps > 0:
        v, secs, n, otraj = oracle_sample(inst, oracle_steps)
        p0, u00 = inst[0]
        cores = host_cores()
        out["cpu_baseline"] = {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle", "cpu": cpu_model(),
                               "sample": f"{n} regular time steps of the alpha={p0.alpha} instance ({secs:.1f} s) "
                                         f"after its first step, numpy/BLAS dense-transform oracle on {cores} "
                                         "host cores"}
        if single_thread_steps > 0 and len(otraj) >= 2:
            st1 = oracle_single_thread(name, otraj[-2], otraj[-1], single_thread_steps)
            if st1:
                out["cpu_baseline"]["single_thread"] = {
                    "value": st1["value"], "unit": UNIT, "cores": 1,
                    "sample": f"{st1['steps']} regular time steps of the same instance ({st1['seconds']:.1f} s), "
                              "BLAS and OpenMP pools set to one thread"}
        nk = len(otraj)
        errs = {}
        for precision, label in ((1, "mixed"), (0, "fp64")):
            s = rfnse.Solver(p0, precision=precision, stream=main)
            s.set_state(torch.from_numpy(u00.ravel().copy()).to(dev))
            gt = torch.empty(nk * p0.size, dtype=torch.complex128, device=dev)
            s.run(nk, gt)
            g = gt.cpu().numpy().reshape((nk,) + p0.shape)
            s.close()
            del gt
            e = rel_errors(g, otraj)
            errs[label] = {"steps": nk, "max": max(e), "last": e[-1],
                           "per_step": [float(f"{x:.3g}") for x in e]}
            del g
        out["err_vs_oracle"] = dict(errs, what=f"relative L2 error of u^1..u^{nk} of the alpha={p0.alpha} instance "
                                               "against the FP64 CPU oracle's trajectory from the same u^0",
                                    tol=p0.tol)
    return out


def run_ours(args):
    import torch
    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    from paper_2410_03643_gb300 import build, rfnse
    build.build_library()
    env = Env(torch, rfnse, dev, torch.cuda.current_stream(), rank, world, local)
    headline = args.workload == "2d" and args.instances == 3
    out = measure(args, env, args.workload, args.instances, args.steps, args.warmup,
                  oracle_steps=30 if args.workload in ("2d", "1d") else 1,
                  single_thread_steps=2 if args.workload in ("2d", "1d") else 0,
                  e2e_steps=max(1, min(args.steps, 30 if args.workload != "3d" else 10)))
    # the metric names both halves: the default line also carries the 3-D 255^3 workload, measured the
    # same way (its oracle sample is the first step and one regular step)
    if headline and not args.no_3d:
        sub = measure(args, env, "3d", 1, args.steps, args.warmup, oracle_steps=1, single_thread_steps=0,
                      e2e_steps=max(1, min(args.steps, 10)))
        for k in ("metric", "n_gpus", "higher_is_better", "scaling", "vs_baseline", "data"):
            sub.pop(k, None)
        out["config_3d"] = sub
    if rank == 0:
        print(json.dumps(out), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def run_batched(args):
    """The 64-instance batch: one bench step = one time step of every instance (one graph launch)."""
    import torch
    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    from paper_2410_03643_gb300 import build, rfnse
    build.build_library()
    inst, desc = workload("batched")
    main = torch.cuda.current_stream()
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    dof = sum(p.size for p, _ in inst)

    def timed(precision, clocks=None):
        b = rfnse.Batch([p for p, _ in inst], precision=precision, stream=main)
        if args.no_lockstep and b.lockstep:
            b.set_lockstep(False)
        if not args.no_autotune:
            b.autotune(reps=5)                      # every distinct grid timed once (set-up, not timed)
        for i, (p, u0) in enumerate(inst):
            b.set_state(i, torch.from_numpy(u0.ravel().copy()).to(dev))
        b.run(max(args.warmup, 3))                  # the first steps run instance by instance
        torch.cuda.synchronize()
        l0 = rfnse.launch_count()
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
        its = []
        barrier(world)
        if clocks:
            clocks.mark_on()
        for k in range(args.steps):
            flush.fill_(float(k))
            evs[k][0].record(main)
            it, _ = b.run(1)
            evs[k][1].record(main)
            its.append(it)
        torch.cuda.synchronize()
        if clocks:
            clocks.mark_off()
        ms = sum(a.elapsed_time(e) for a, e in evs)
        launches = rfnse.launch_count() - l0
        states = [b.get_state(i)[1] for i in range(b.count)]
        modes.append(b.lockstep)
        b.close()
        return ms, launches, np.array(its), states

    modes = []

    clocks = ClockSampler(local) if rank == 0 else None
    if clocks:
        clocks.start()
    ms, launches, its, st_mixed = timed(1, clocks)
    clk = clocks.stop() if clocks else None
    ms = reduce_max(ms, world, dev)
    out = {"metric": METRIC, "value": weak_value(world, dof, args.steps, ms), "unit": UNIT, "n_gpus": world,
           "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": ms / args.steps,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64 (mixed)",
           "data": "synthetic (closed-form initial data of the paper's shape, seeded parameters)",
           "config": dict(desc, precision="mixed", l2="256 MiB buffer written between timed steps",
                          parallelism=f"{world} GPU(s); one CUDA graph launch per batch step",
                          lockstep=bool(modes and modes[0])),
           "gpu_launches": launches, "iters_per_solve_mean": float(its.mean())}
    if clk:
        out["clocks"] = clk
    if not args.no_fp64:
        ms64, _, its64, st64 = timed(0)
        ms64 = reduce_max(ms64, world, dev)
        errs = [float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b)) for a, b in zip(st_mixed, st64)]
        out["fp64"] = {"value": world * dof * args.steps / (ms64 * 1e-3), "ms_per_step": ms64 / args.steps,
                       "iters_per_solve_mean": float(its64.mean())}
        out["mixed_vs_fp64_rel_l2_after_run"] = max(errs)
        out["mixed_speedup_vs_fp64"] = ms64 / ms
    if rank == 0:
        print(json.dumps(out), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def run_adjoint(args):
    """The gradient workload (255^2, 20 steps, FP64): one bench step = a taped forward run plus its
    reverse pass (dL/du0 and dL/drho of L = sum |u^N - u_target|^2), checkpoints every 5 steps."""
    import torch
    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    from paper_2410_03643_gb300 import build, rfnse
    build.build_library()
    p, u0, nsteps, u0t, rho_t = W.config_adjoint()
    main = torch.cuda.current_stream()
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    st = rfnse.Solver(p.replace(rho=rho_t), precision=0, stream=main)
    target, _ = st.tape_forward(torch.from_numpy(u0t.ravel().copy()).to(dev), nsteps, 5)
    st.close()
    s = rfnse.Solver(p, precision=0, stream=main)
    x0 = torch.from_numpy(u0.ravel().copy()).to(dev)

    def one():
        uN, _ = s.tape_forward(x0, nsteps, 5)
        return s.tape_backward(2.0 * (uN - target))

    for _ in range(max(args.warmup, 3)):
        one()
    torch.cuda.synchronize()
    l0 = rfnse.launch_count()
    fw, bw = [], []
    clocks = ClockSampler(local) if rank == 0 else None
    if clocks:
        clocks.start()
        clocks.mark_on()
    barrier(world)
    for k in range(args.steps):
        flush.fill_(float(k))
        e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        e0.record(main)
        uN, _ = s.tape_forward(x0, nsteps, 5)
        e1.record(main)
        g0, grho, its = s.tape_backward(2.0 * (uN - target))
        e2.record(main)
        torch.cuda.synchronize()
        fw.append(e0.elapsed_time(e1))
        bw.append(e1.elapsed_time(e2))
    if clocks:
        clocks.mark_off()
    clk = clocks.stop() if clocks else None
    launches = rfnse.launch_count() - l0
    ms = reduce_max(sum(fw) + sum(bw), world, dev)
    out = {"metric": METRIC, "value": weak_value(world, p.size * nsteps, args.steps, ms), "unit": UNIT,
           "n_gpus": world, "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": ms / args.steps,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
           "data": "synthetic (closed-form initial data; target from a seeded perturbation of u0 and rho)",
           "config": {"workload": "adjoint_2d_n255_alpha1.5_rho2_dt0.005_20steps_fp64", "d": 2, "n": [255, 255],
                      "what": "one step = taped forward run + reverse pass (dL/du0, dL/drho), checkpoint every 5",
                      "l2": "256 MiB buffer written between timed steps", "parallelism": f"{world} GPU(s)"},
           "gpu_launches": launches, "forward_ms": sum(fw) / args.steps, "backward_ms": sum(bw) / args.steps,
           "backward_over_forward": sum(bw) / max(sum(fw), 1e-9), "adjoint_arnoldi_steps": its,
           "grad_rho": grho}
    if clk:
        out["clocks"] = clk
    if rank == 0:
        print(json.dumps(out), flush=True)
    s.close()
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def run_comparators(args):
    """tau-GMRES against the comparators of Sec. 5 (C-GMRES with Strang's circulant, plain GMRES) on
    the same time-stepping run: 2-D 255^2, alpha = 1.5, rho = 2, dt = 0.005, tol 1e-10, mixed form."""
    import torch
    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    from paper_2410_03643_gb300 import build, rfnse
    build.build_library()
    p, u0, _ = W.config_2d(1.5, n=255)
    main = torch.cuda.current_stream()
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    res = {}
    for pc, name in ((0, "tau-GMRES"), (1, "C-GMRES"), (2, "GMRES")):
        q = p.replace(precond=pc, restart=256 if pc == 2 else p.restart)
        s = rfnse.Solver(q, precision=1, stream=main)
        s.set_state(torch.from_numpy(u0.ravel().copy()).to(dev))
        s.run(max(args.warmup, 3))
        steps = args.steps if pc != 2 else max(1, min(args.steps, 3))
        torch.cuda.synchronize()
        ms, its = 0.0, []
        for k in range(steps):
            flush.fill_(float(k))
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(main)
            it, _ = s.run(1)
            b.record(main)
            torch.cuda.synchronize()
            ms += a.elapsed_time(b)
            its.append(int(it[0]))
        res[name] = {"value": q.size * steps / (ms * 1e-3), "ms_per_step": ms / steps,
                     "iters_per_solve_mean": float(np.mean(its)), "steps": steps}
        s.close()
    out = {"metric": METRIC, "value": res["tau-GMRES"]["value"], "unit": UNIT, "n_gpus": 1,
           "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": res["tau-GMRES"]["ms_per_step"],
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64 (mixed)",
           "data": "synthetic (closed-form initial data of the paper's shape)",
           "config": {"workload": "comparators_2d_n255_alpha1.5_rho2_dt0.005_tol1e-10", "d": 2, "n": [255, 255],
                      "what": "the same run with the sine-transform preconditioner, Strang's circulant "
                              "(Bluestein DFTs) and none (restart 256)",
                      "l2": "256 MiB buffer written between timed steps"},
           "comparators": res}
    if rank == 0:
        print(json.dumps(out), flush=True)


def run_omega(args):
    """Fig. 1: tau-GMRES iterations at the 2nd time level versus the TBAN parameter w in (0, 4] for
    alpha = 1.1:0.2:1.9 (1-D, [-20,20], rho = 2, sech(x)e^{2ix}, n = 2047, dt = 0.05, tol 1e-8, no
    restart); the line's value is the solve throughput over the whole sweep."""
    import torch
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    from paper_2410_03643_gb300 import build, rfnse
    build.build_library()
    main = torch.cuda.current_stream()
    omegas = [round(0.1 * k, 1) for k in range(1, 41)]
    curves, best, total_ms, nsolve = {}, {}, 0.0, 0
    n = 2047
    for alpha in (1.1, 1.3, 1.5, 1.7, 1.9):
        its = []
        for w in omegas:
            p = W.Problem(d=1, n=(n,), lo=(-20.0,), hi=(20.0,), alpha=alpha, rho=2.0, dt=0.05, tol=1e-8, omega=w,
                          restart=256)
            s = rfnse.Solver(p, precision=0, stream=main)
            u0 = torch.from_numpy(W.u0_sech_1d(p, 2.0)).to(dev)
            s.set_state(u0)
            s.run(1)
            _, u1, _ = s.get_state()
            D = (p.rho * p.dt) * torch.abs(u1) ** 2
            b = -s.apply_A(u0, D) + 2j * u0
            s.solve(D, b)                                    # warm: graph capture
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(main)
            _, it, _ = s.solve(D, b)
            e1.record(main)
            torch.cuda.synchronize()
            total_ms += e0.elapsed_time(e1)
            nsolve += 1
            its.append(it)
            s.close()
        curves[str(alpha)] = its
        best[str(alpha)] = omegas[int(np.argmin(its))]
    out = {"metric": METRIC, "value": n * nsolve / (total_ms * 1e-3), "unit": UNIT, "n_gpus": 1, "steps": nsolve,
           "warmup": 1, "ms_per_step": total_ms / nsolve, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "f64", "data": "synthetic (the 1-D test of Sec. 5.1)",
           "config": {"workload": "omega_sweep_1d_n2047_rho2_dt0.05_tol1e-8", "what": "one step = one solve at "
                      "the 2nd time level; w = 0.1:0.1:4.0 for each alpha"},
           "omega": omegas, "iterations": curves, "best_omega": best}
    print(json.dumps(out), flush=True)


def kernel_case(args):
    """A small run of the workload's kernels for ncu captures: the first time step's predictor solve of
    the workload's grid in the mixed form (host-driven loops, restart 2, at most 4 Arnoldi steps), so
    that every pass class, the Arnoldi kernel and the double-float residual passes launch a few times
    on vectors of the full size."""
    import torch
    from paper_2410_03643_gb300 import build, rfnse
    build.build_library()
    inst, _ = workload(args.kernel_case, 1)
    p, u0 = inst[0]
    p = p.replace(restart=2, max_it=4)
    s = rfnse.Solver(p, precision=1, device_loop=0)
    if not args.no_autotune:
        s.autotune(reps=5)                 # the geometry the bench's solvers launch with
    s.set_state(torch.from_numpy(u0.ravel().copy()).to("cuda"))
    its, _ = s.run(1, allow_noconv=True)
    torch.cuda.synchronize()
    print(json.dumps({"kernel_case": args.kernel_case, "n": list(p.n[:p.d]), "arnoldi_steps": int(its[0]),
                      "launches": rfnse.launch_count()}), flush=True)
    s.close()


def arnoldi_probe():
    """Duration of the cooperative Arnoldi kernel per column j (CUDA events, 20 launches each)."""
    import torch
    from paper_2410_03643_gb300 import build, rfnse
    build.build_library()
    props = torch.cuda.get_device_properties(0)
    out = {"device": props.name, "what": "k_mgs_step: MGS against j+1 basis vectors, Givens, test"}
    for name, n in (("2d_511^2", 511 * 511), ("3d_255^3", 255 ** 3)):
        rows = {}
        for j in (0, 1, 2, 3, 4, 7):
            us, blocks = rfnse.probe_arnoldi(n, j)
            rows[str(j)] = round(us, 2)
        out[name] = {"n": n, "blocks": blocks, "us_per_step_by_j": rows}
    print(json.dumps(out), flush=True)


def alu_probe():
    import torch
    from paper_2410_03643_gb300 import build, rfnse
    build.build_library()
    props = torch.cuda.get_device_properties(0)
    out = {"device": props.name, "sms": props.multi_processor_count,
           "fp64_tflops": rfnse.probe_fma(True) / 1e12, "fp32_tflops": rfnse.probe_fma(False) / 1e12}
    out["fp32_over_fp64"] = out["fp32_tflops"] / out["fp64_tflops"]
    print(json.dumps(out), flush=True)


def main():
    args = parse()
    if args.cpu_sample:
        cpu_sample_child(args)
        return
    if args.kernel_case:
        kernel_case(args)
        return
    if args.alu_probe:
        alu_probe()
        return
    if args.arnoldi_probe:
        arnoldi_probe()
        return
    if args.impl == "reference":
        run_reference(args)
    elif args.workload == "batched":
        run_batched(args)
    elif args.workload == "adjoint":
        run_adjoint(args)
    elif args.workload == "comparators":
        run_comparators(args)
    elif args.workload == "omega":
        run_omega(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()

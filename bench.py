"""Benchmark: PCG_C ground states per second on one GB300 (and N replicas).

A step is one complete ground-state solve of the 2D fast-rotation workload
(256x256 on [-16,16]^2, V = r^2/2, eta = 1000, omega = 0.9, Gaussian-plus-
vortex initial guess, mixed precision: complex64 phase then complex128
refinement, stop at ||H phi - lambda phi||_inf < 1e-8), through the C ABI with
phi already in device memory.  Alongside it the line reports:

  roofline      H phi on a batch of 512 fields of 256x256 complex64 (gpe_apply_H_batch,
                one thread-block cluster per field; 268 MB in + 268 MB out > L2),
                achieved = algorithmic bytes (16 B/point + V once) / CUDA-event
                time, vs the measured HBM peak;
  e2e           the same solve with phi in pinned HOST memory (H2D/D2H copies
                inside the call and inside the timed region);
  accuracy      the mixed solve's energy against this library's FP64 solve of the
                same workload (relative error) and both residuals;
  cpu_baseline  the FP64 CPU oracle on bounded samples of the same workload, on one
                host thread and on every host core (independent solves in parallel),
                scaled by the oracle's own iteration count for a full solve; the
                oracle also re-evaluates E and ||r||_inf at the GPU's result;
  secondary     the 128^3 3D workload (eta = 5000, omega = 0.8), ground states/s;
  batch         the 96-instance parameter sweep in one graph launch per rank (the
                instances split by index over the ranks), ground states/s, beside
                the same instances solved one at a time in FP64;
  grad          the differentiation workload: 16 instances at 256^2 solved in one
                batched launch, then per instance the Hellmann-Feynman derivatives
                and the density-loss gradient through the tangent adjoint solve;
  libfft_baseline  the same workload solved in FP64 by plain PyTorch with
                torch.fft (cuFFT), beside this library's FP64 single-instance solve.

--impl reference runs the CPU oracle as the reference arm.
"""
from __future__ import annotations

import os

# The CPU oracle legs count host threads exactly: numpy's BLAS runs one thread per
# process (set before numpy loads; spawned oracle processes inherit it).
for _v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
    os.environ.setdefault(_v, "1")

import argparse
import json
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

WORKLOAD = "fast256_2d"
METRIC = "ground states/sec to residual 1e-8 (256², 128³); H·φ GB/s vs HBM peak"
UNIT = "ground_states/s"
HPHI_BATCH = 512  # fields of 256x256 complex64 in the H phi roofline batch (268 MB in, 268 MB out)
# ncu summary of the roofline kernel; its line "dram_bytes_per_launch_512_fields: <int>" holds
# dram__bytes_read.sum + dram__bytes_write.sum of one launch over HPHI_BATCH fields, taken from a
# capture of the current kernel (the line is removed when the kernel changes).
HPHI_PROFILE = os.path.join(ROOT, "profiles", "h_batch_flow_256x256_batch_c64.md")
ORACLE_ITERATIONS = os.path.join(ROOT, "tests", "golden", "oracle_iterations.json")


def hphi_traffic():
    try:
        with open(HPHI_PROFILE) as fh:
            for line in fh:
                if line.startswith("dram_bytes_per_launch_512_fields:"):
                    return int(line.split(":", 1)[1].split()[0])
    except OSError:
        pass
    return None


def oracle_iterations(workload):
    """The FP64 oracle's own iteration count for a full solve of `workload`
    (tests/golden/make_oracle_iterations.py)."""
    with open(ORACLE_ITERATIONS) as fh:
        return int(json.load(fh)[workload]["iters"])


def cpu_model():
    try:
        with open("/proc/cpuinfo") as fh:
            for line in fh:
                k = line.split(":", 1)
                if len(k) == 2 and k[0].strip() in ("model name", "Model name"):
                    return k[1].strip()
    except OSError:
        pass
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.startswith("Model name"):
                return line.split(":", 1)[1].strip()
    except Exception:
        pass
    return "unknown"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-secondary", action="store_true")
    ap.add_argument("--no-batch", action="store_true", help="skip the 96-instance batched sweep")
    ap.add_argument("--no-batch-fp64", action="store_true",
                    help="skip the sweep's instances solved one at a time in FP64")
    ap.add_argument("--no-grad", action="store_true", help="skip the 16-instance differentiation workload")
    ap.add_argument("--no-paper", action="store_true", help="skip the 512^2 solves of the paper's Tables 2 and 3")
    ap.add_argument("--no-fp64", action="store_true",
                    help="skip the FP64 legs (accuracy against the FP64 solve, the FP64 roof, the pipe rates)")
    ap.add_argument("--no-fftpass", action="store_true", help="skip H phi on the 256x256x512 field (pass bandwidth)")
    ap.add_argument("--no-libfft", action="store_true",
                    help="skip the library-FFT baseline (torch.fft / cuFFT complex128 PCG_C) and the FP64 solve")
    ap.add_argument("--no-autotune", action="store_true", help="keep the default pass-kernel plans")
    ap.add_argument("--plan", default="", help="E,width for every mode and axis instead of tuning (profiling runs)")
    ap.add_argument("--no-graph", action="store_true",
                    help="launch the same pass kernels from a host loop instead of one graph with a device-side "
                         "loop (for ncu launch lists: ncu cannot profile kernel nodes of graphs with conditional "
                         "nodes)")
    return ap.parse_args()


def dist_env():
    from paper_1611_02045_gb300.replicas import dist_env as _env
    return _env()


def cpu_cores():
    try:
        return len(os.sched_getaffinity(0))
    except Exception:
        return os.cpu_count() or 1


def oracle_sample(seconds=12.0, max_iters=400):
    """Time FP64 oracle PCG_C iterations on the workload (bounded sample):
    (seconds per iteration, iterations timed)."""
    from oracle import gpe_oracle as O
    from paper_1611_02045_gb300 import inputs as I
    w = I.workload(WORKLOAD)
    prob = O.Problem(w["n"], w["L"], w["eta"], w["omega"], w["V"])
    # one iteration first (imports, caches), then grow until the time budget
    t0 = time.perf_counter()
    O.pcg_solve(prob, w["phi0"], O.SolveOptions(max_iter=1))
    t1 = time.perf_counter()
    per = max(t1 - t0, 1e-3) / 2.0
    k = int(max(5, min(max_iters, seconds / per)))
    t0 = time.perf_counter()
    _, rep = O.pcg_solve(prob, w["phi0"], O.SolveOptions(max_iter=k))
    dt = time.perf_counter() - t0
    return dt / max(rep["iters"], 1), rep["iters"]


def _oracle_worker(args):
    seconds, max_iters = args
    return oracle_sample(seconds=seconds, max_iters=max_iters)


def oracle_all_cores(seconds, max_iters, procs):
    """The same bounded sample in `procs` independent processes at once (spawned,
    one per host core): a full solve on each core in parallel is the oracle's
    whole-host throughput.  Returns (mean seconds per iteration per process,
    iterations per process, wall seconds)."""
    import concurrent.futures as cf
    import multiprocessing as mp
    t0 = time.perf_counter()
    with cf.ProcessPoolExecutor(max_workers=procs, mp_context=mp.get_context("spawn")) as ex:
        res = list(ex.map(_oracle_worker, [(seconds, max_iters)] * procs))
    wall = time.perf_counter() - t0
    return statistics.mean(r[0] for r in res), min(r[1] for r in res), wall


def oracle_naive_64():
    """The naive-DFT oracle (explicit O(M^2) sums per line) solving the 64x64
    workload c64_2d to ||r||_inf < 1e-8, and the FFT-backend oracle on the same
    solve: (naive seconds, fft seconds, iterations)."""
    from oracle import gpe_oracle as O
    from paper_1611_02045_gb300 import inputs as I
    w = I.workload("c64_2d")
    out = []
    for backend in ("naive", "fft"):
        prob = O.Problem(w["n"], w["L"], w["eta"], w["omega"], w["V"], backend=backend)
        t0 = time.perf_counter()
        _, rep = O.pcg_solve(prob, w["phi0"], O.SolveOptions())
        out.append((time.perf_counter() - t0, rep["iters"]))
    return out[0][0], out[1][0], out[0][1]


class Clocks:
    """nvidia-smi sampling during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        try:
            self.p = subprocess.Popen(["nvidia-smi", "-i", str(index), f"--query-gpu={self.Q}",
                                       "--format=csv,noheader,nounits", "-lms", "200"],
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
        rows = []
        with open(self.f.name) as fh:
            for line in fh:
                parts = [x.strip() for x in line.split(",")]
                if len(parts) >= 9:
                    rows.append(parts)
        os.unlink(self.f.name)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        reasons = set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            for nm, v in zip(names, r[5:9]):
                if v.strip().lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(rows)}


def run_reference(args, rank, world):
    """Reference arm: the FP64 CPU oracle (numpy) on every host core, bounded
    samples.  Each step times oracle iterations of the workload in one process
    per core (~8 s); a ground state takes the oracle's own full-solve iteration
    count, so the host delivers cores / (seconds per iteration x iterations)
    ground states per second.  ms_per_step is the wall time of a step's sample."""
    if rank != 0:
        return
    iters_per_solve = oracle_iterations(WORKLOAD)
    cores = cpu_cores()
    oracle_all_cores(1.0, 5, cores)  # warm-up: process start, imports
    for _ in range(max(args.warmup - 1, 0)):
        oracle_sample(seconds=0.5, max_iters=5)
    t_iters, walls, ks = [], [], []
    for _ in range(args.steps):
        t_it, k, wall = oracle_all_cores(8.0, 400, cores)
        t_iters.append(t_it)
        walls.append(wall)
        ks.append(k)
    t_it = statistics.mean(t_iters)
    val = cores / (t_it * iters_per_solve)
    ms = 1000.0 * statistics.mean(walls)
    line = {"impl": "reference", "metric": METRIC, "value": val, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "grid": "256x256", "eta": 1000.0, "omega": 0.9,
                       "tol_res_inf": 1e-8, "l2": "n/a (CPU)"},
            "cpu_baseline": {"value": val, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "cpu_model": cpu_model(),
                             "sample": f"each step: {cores} processes (one per host core) each time >= {min(ks)} "
                                       f"FP64 numpy PCG_C iterations of {WORKLOAD} (~8 s); "
                                       f"{t_it * 1e3:.2f} ms per iteration per process; a ground state = the "
                                       f"oracle's own {iters_per_solve} iterations to ||r||_inf < 1e-8 "
                                       f"(tests/golden/oracle_iterations.json)",
                             "ms_per_iteration": t_it * 1e3, "oracle_iters_per_solve": iters_per_solve,
                             "projected_s_per_solve_per_core": t_it * iters_per_solve},
            "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def main():
    args = parse()
    rank, world, local = dist_env()
    if args.impl == "reference":
        run_reference(args, rank, world)
        return

    import torch
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        torch.cuda.set_device(0)
    dev = torch.device("cuda", torch.cuda.current_device())

    from paper_1611_02045_gb300 import build as B
    if rank == 0:
        B.build()
    if world > 1:
        torch.distributed.barrier()
    from paper_1611_02045_gb300 import gpe, inputs as I

    stream = torch.cuda.current_stream()
    w = I.workload(WORKLOAD)
    n, L = w["n"], w["L"]
    N = int(np.prod(n))
    ctx = gpe.Context(n, L, w["eta"], w["omega"], w["V"], prec=gpe.GPE_MIXED)
    # set-up, outside every timed region: the tuner picks the pass-kernel plans
    tune = None
    if args.plan:
        E_, w_ = (int(v) for v in args.plan.split(","))
        for m_ in (0, 1, 2):
            for ax_ in range(len(n)):
                ctx.set_plan(m_, ax_, E_, w_)
        tune = {"plans": f"fixed E={E_}, width={w_}", "seconds": 0.0}
    elif not args.no_autotune:
        t0 = time.perf_counter()
        tune = ctx.autotune(iters=20)
        tune["seconds"] = time.perf_counter() - t0
    phi0_d = torch.from_numpy(w["phi0"].copy()).to(dev)
    phi_d = torch.empty_like(phi0_d)
    l2_flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)  # 256 MB > L2

    opts = gpe.solve_opts_default()  # the library's default loop for this grid
    if args.no_graph:
        opts.use_graph = 0

    def solve_dev():
        phi_d.copy_(phi0_d)
        return ctx.pcg_solve(phi_d, opts, check=True)

    for _ in range(max(args.warmup, 3)):
        rep = solve_dev()
    iters_total, iters_lo = rep["iters"], rep["iters_lo"]

    # ---------------- timed region: K solves, L2 flushed before each ----------------
    def barrier():
        if world > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()

    clocks = Clocks(torch.cuda.current_device())
    barrier()
    step_ms, reps = [], []
    for _ in range(args.steps):
        l2_flush.zero_()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        reps.append(solve_dev())
        ev1.record(stream)
        ev1.synchronize()
        step_ms.append(ev0.elapsed_time(ev1))
    barrier()
    clk = clocks.stop()
    from paper_1611_02045_gb300.replicas import job_throughput, max_over_ranks
    ms = max_over_ranks(statistics.mean(step_ms), dev)
    value = job_throughput(ms, world)
    launches = 0
    for r in reps:
        it, lo, fp = r["iters"], r["iters_lo"], r["iters_fp64"]
        # four precision conversions (c128->c64, c64->c128, c64->ds, ds->c128) and one
        # normalisation kernel per phase; 7 pass kernels per loop-body execution
        # (a phase of k iterations executes its body k + 1 times)
        fp64_phase = (1 + 7 * (fp + 1)) if fp else 0
        if r["loop_kind"] == 3:  # one cluster kernel runs the complex64 phase
            launches += 4 + 2 + 1 + 7 * (it - lo - fp + 1) + fp64_phase
        elif r["loop_kind"] == 2:  # one persistent kernel per phase
            launches += 4 + 2 + 2 + (2 if fp else 0)
        else:
            launches += 4 + (1 + 7 * (lo + 1)) + (1 + 7 * (it - lo - fp + 1)) + fp64_phase

    # ---------------- e2e: phi in pinned host memory ----------------
    phi_h0 = torch.from_numpy(w["phi0"].copy()).pin_memory()
    phi_h = torch.empty_like(phi_h0).pin_memory()
    e2e_ms = []
    for _ in range(args.steps):
        phi_h.copy_(phi_h0)
        l2_flush.zero_()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ctx.pcg_solve(phi_h.data_ptr(), opts, check=True)
        torch.cuda.synchronize()
        e2e_ms.append(1000.0 * (time.perf_counter() - t0))
    e2e_val = job_throughput(max_over_ranks(statistics.mean(e2e_ms), dev), world)

    # ---------------- roofline: H phi on a batch of fields larger than L2 ----------------
    # HPHI_BATCH fields of the workload's grid (gpe_apply_H_batch: the dataflow of row and
    # column units on every SM), complex64: algorithmic bytes = read phi + write H phi
    # per point (16 B) + V once (4 B per grid point, shared by the batch).
    NB = HPHI_BATCH
    g = torch.Generator(device=dev).manual_seed(1)
    hphi = torch.randn(NB * N, dtype=torch.complex64, device=dev, generator=g)
    hout = torch.empty_like(hphi)
    for _ in range(3):
        ctx.apply_H_batch(NB, hphi, hphi, hout)
    torch.cuda.synchronize()
    hms = []
    for _ in range(20):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        ctx.apply_H_batch(NB, hphi, hphi, hout)
        b.record(stream)
        b.synchronize()
        hms.append(a.elapsed_time(b))
    h_ms = statistics.median(hms)
    hbytes = 16 * NB * N + 4 * N
    achieved = hbytes / (h_ms * 1e-3) / 1e9
    peaks = {}
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            peaks = json.load(fh)
    except Exception:
        pass
    peak = float(peaks.get("hbm_gbs", 6800.0))
    del hphi, hout

    # ---------------- arithmetic-pipe rates and the FP64 roof ----------------
    # FP64 mode is bound by the FP64 pipe, not by HBM: H phi in FP64 on a 256^3 complex128
    # field (268 MB in, 268 MB out), flops by the nominal 5 M log2 M model per line transform
    # (3 axes x forward + inverse) plus 20 flops per point for the multipliers and the real-space
    # term, against the measured FP64 fma rate.
    alu, fp64_roof = None, None
    if not args.no_fp64:
        alu = {k: gpe.alu_peak(k) for k in ("fp64_fma", "fp32_fma", "fp32x2_fma")}
    if rank == 0 and not args.no_fp64:
        n3, L3 = (256, 256, 256), (8.0, 8.0, 8.0)
        N3 = int(np.prod(n3))
        with gpe.Context(n3, L3, 5000.0, 0.8, I.harmonic(n3, L3, [1.0, 1.0, 2.0]), prec=gpe.GPE_FP64) as c3:
            g3 = torch.Generator(device=dev).manual_seed(3)
            x3 = torch.randn(N3, dtype=torch.complex128, device=dev, generator=g3)
            y3 = torch.empty_like(x3)
            for _ in range(2):
                c3.apply_H(x3, x3, y3)
            t3 = []
            for _ in range(5):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                c3.apply_H(x3, x3, y3)
                b.record(stream)
                b.synchronize()
                t3.append(a.elapsed_time(b))
            del x3, y3
        ms3 = statistics.median(t3)
        flops3 = (3 * 2 * 5 * 8 + 20) * N3
        ach = flops3 / (ms3 * 1e-3) / 1e9
        fp64_roof = {"kernel": "gpe_apply_H, GPE_FP64, 256^3 complex128 (x, y, z pass kernels)", "bound": "fp64_alu",
                     "achieved": ach, "peak": alu["fp64_fma"], "unit": "GFLOP/s", "frac": ach / alu["fp64_fma"],
                     "ms_per_call": ms3, "hbm_gbs_algorithmic": 40.0 * N3 / (ms3 * 1e-3) / 1e9,
                     "flop_model": "5 M log2 M per line transform x 6 transforms + 20 per point",
                     "peak_source": "gpe_alu_peak(fp64 fma), measured in this run"}

    # ---------------- H phi on one 256x256x512 complex64 field (beyond L2) ----------------
    # By default the x and y parts run as one dataflow launch over the z planes (phi and V in, t
    # out: 20 bytes per point, the planes' y parts staying in L2), then the z pass (f and t in, H phi
    # out: 24).  With a plan set for an axis the three passes run: x (20), y and z (24 each), TMA-fed
    # persistent kernels whose DRAM figures are in profiles/fft_passes_256x256x512_c64.md.  The
    # operator itself needs 20 bytes per point (read phi and V, write H phi).
    fftpass = None
    if rank == 0 and not args.no_fftpass:
        nf3, Lf3 = (256, 256, 512), (8.0, 8.0, 8.0)
        Nf3 = int(np.prod(nf3))
        with gpe.Context(nf3, Lf3, 100.0, 0.5, np.zeros(I.shape_of(nf3)), prec=gpe.GPE_MIXED) as cf3:
            gf = torch.Generator(device=dev).manual_seed(5)
            xf = torch.randn(Nf3, dtype=torch.complex64, device=dev, generator=gf)
            yf = torch.empty_like(xf)

            def time_f3(bytes_per_point, kernels):
                for _ in range(3):
                    cf3.apply_H(xf, xf, yf)
                tf = []
                for _ in range(10):
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    a.record(stream)
                    cf3.apply_H(xf, xf, yf)
                    b.record(stream)
                    b.synchronize()
                    tf.append(a.elapsed_time(b))
                msf = statistics.median(tf)
                gbs = bytes_per_point * Nf3 / (msf * 1e-3) / 1e9
                return {"ms_per_call": msf, "operator_gbs": 20.0 * Nf3 / (msf * 1e-3) / 1e9,
                        "bytes_per_point": bytes_per_point, "passes_gbs": gbs, "passes_frac": gbs / peak,
                        "kernels": kernels}

            fftpass = {"field": "256x256x512 complex64 (268 MB)",
                       **time_f3(20 + 24, "h_batch_flow<256,256> on 512 planes, pass_s_tma<512,8,HMID>")}
            cf3.set_plan(0, 0, *cf3.get_plan(0, 0))  # the caller's own plan, though the same: the passes run
            fftpass["three_passes"] = time_f3(20 + 24 + 24, "pass_hx_bulk<256,8>, pass_s_tma<256,8,HMID>, "
                                                            "pass_s_tma<512,8,HMID>")
            fftpass["per_pass"] = "profiles/fft_passes_256x256x512_c64.md"
            del xf, yf

    # ---------------- secondary: the 128^3 workload ----------------
    secondary = None
    if not args.no_secondary:
        w3 = I.workload("rot128_3d")
        ctx3 = gpe.Context(w3["n"], w3["L"], w3["eta"], w3["omega"], w3["V"], prec=gpe.GPE_MIXED)
        plans3 = None if args.no_autotune else ctx3.autotune(iters=10)["plans"]
        p30 = torch.from_numpy(w3["phi0"].copy()).to(dev)
        p3 = torch.empty_like(p30)
        p3.copy_(p30)
        r3 = ctx3.pcg_solve(p3, check=True)  # warm-up (graph build)
        s3 = []
        for _ in range(2):
            p3.copy_(p30)
            l2_flush.zero_()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            r3 = ctx3.pcg_solve(p3, check=True)
            b.record(stream)
            b.synchronize()
            s3.append(a.elapsed_time(b))
        secondary = {"workload": "rot128_3d", "value": 1000.0 / statistics.mean(s3), "unit": UNIT,
                     "ms_per_step": statistics.mean(s3), "iters": r3["iters"], "iters_lo": r3["iters_lo"],
                     "E": r3["E"], "res_inf": r3["res_inf"], "plans": plans3}
        ctx3.close()

    # ---------------- secondary: the 96-instance batched parameter sweep ----------------
    # The instances are independent: rank r takes those with index = r (mod world), in one
    # graph launch; no data-path collective, the reports are combined on the host.
    batch = None
    if not args.no_batch:
        from paper_1611_02045_gb300.replicas import instance_share, sum_over_ranks
        insts_all = I.sweep_instances(96)
        mine = instance_share(len(insts_all), rank, world)
        insts = [insts_all[i] for i in mine]
        arrays = [I.sweep_arrays(x) for x in insts]
        specs = [dict(n=x["n"], L=x["L"], eta=x["eta"], omega=x["omega"], V=V, prec=gpe.GPE_MIXED)
                 for x, (V, _) in zip(insts, arrays)]
        bphi0 = [torch.from_numpy(p.copy()).to(dev) for _, p in arrays]
        bphi = [torch.empty_like(p) for p in bphi0]
        with gpe.Batch(specs) as B:
            if not args.no_autotune:
                B.autotune(iters=10)
            bts = []
            for k in range(4):  # the first launch builds the graph; three timed launches
                for p, q in zip(bphi, bphi0):
                    p.copy_(q)
                l2_flush.zero_()
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                bs, breps = B.solve(bphi)
                b.record(stream)
                b.synchronize()
                if k:
                    bts.append(a.elapsed_time(b))
        bms = max_over_ranks(statistics.median(bts), dev)
        counts = [sum(r["status"] == gpe.GPE_OK for r in breps), sum(r["iters"] for r in breps),
                  sum(r["iters_fp64"] > 0 for r in breps), len(breps)]
        fp64_ms = None
        if not args.no_batch_fp64:
            # the same instances solved one at a time in FP64 (gpe_pcg_solve, tuned plans)
            fp64_ms, fp64_ok = 0.0, 0
            for x, (V, _), p0 in zip(insts, arrays, bphi0):
                with gpe.Context(x["n"], x["L"], x["eta"], x["omega"], V, prec=gpe.GPE_FP64) as c1:
                    if not args.no_autotune:
                        c1.autotune(iters=10)
                    p1 = p0.clone()
                    c1.pcg_solve(p1.clone())  # builds the graph
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    a.record(stream)
                    r1 = c1.pcg_solve(p1)
                    b.record(stream)
                    b.synchronize()
                    fp64_ms += a.elapsed_time(b)
                    fp64_ok += r1["status"] == gpe.GPE_OK
            fp64_ms = max_over_ranks(fp64_ms, dev)
            counts.append(fp64_ok)
        counts = [int(v) for v in sum_over_ranks(counts, dev)]
        batch = {"workload": "sweep96_2d (32 each of 128^2, 256^2, 512^2 on [-16,16]^2; omega U[0,0.95], "
                             "eta {100,250,500,1000}, kappa {0,0.05})",
                 "value": 96 * 1000.0 / bms, "unit": UNIT, "ms_per_step": bms,
                 "launch": f"one CUDA graph per rank (gpe_batch_solve); instances split by index over "
                           f"{world} rank(s); median of 3 timed launches",
                 "converged": counts[0], "iters_total": counts[1], "fp64_completions": counts[2],
                 "instances": counts[3]}
        if fp64_ms is not None:
            batch["fp64_single_instances"] = {
                "value": 96 * 1000.0 / fp64_ms, "unit": UNIT, "ms_total": fp64_ms, "converged": counts[4],
                "how": "every instance solved alone in FP64 (gpe_pcg_solve, graph loop, tuned plans), "
                       "CUDA events per solve, summed"}
            batch["speedup_vs_fp64_singles"] = fp64_ms / bms
        del bphi, bphi0

    # ---------------- the differentiation workload: 16 instances at 256^2 ----------------
    grad = None
    if not args.no_grad and rank == 0:
        gws = [I.workload("grad256_2d", i) for i in range(16)]
        gspecs = [dict(n=x["n"], L=x["L"], eta=x["eta"], omega=x["omega"], V=x["V"], prec=gpe.GPE_MIXED)
                  for x in gws]
        gphi0 = [torch.from_numpy(x["phi0"].copy()).to(dev) for x in gws]
        gphi = [torch.empty_like(p) for p in gphi0]
        gN = int(np.prod(gws[0]["n"]))
        wt = I.weight(gws[0]["n"], gws[0]["L"])
        rho_t = torch.from_numpy(np.abs(I.normalise(I.anisotropic_gaussian(gws[0]["n"], gws[0]["L"], [0.05, 0.04]),
                                                    gws[0]["n"], gws[0]["L"])) ** 2).to(dev)
        gV = torch.empty(gphi0[0].shape, dtype=torch.float64, device=dev)
        gL = torch.empty_like(gV)
        g_rho = torch.empty_like(gV)
        Vd = [torch.from_numpy(x["V"]).to(dev) for x in gws]
        with gpe.Batch(gspecs) as GB, gpe.Context(gws[0]["n"], gws[0]["L"], gws[0]["eta"], gws[0]["omega"],
                                                 gws[0]["V"], prec=gpe.GPE_FP64) as gc:
            if not args.no_autotune:
                GB.autotune(iters=10)
            gts, adj_iters = [], 0
            for k in range(3):  # the first pass builds the graphs
                for p, q in zip(gphi, gphi0):
                    p.copy_(q)
                l2_flush.zero_()
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                gs, greps = GB.solve(gphi)
                adj_iters = 0
                for x, p, v in zip(gws, gphi, Vd):
                    gc.set_problem(v, x["eta"], x["omega"])
                    gc.energy_grad(p, None, gV)
                    torch.mul(torch.abs(p) ** 2 - rho_t, 2.0 * wt, out=g_rho)
                    adj_iters += gc.density_adjoint(p, g_rho, gL, tol=1e-10, max_iter=3000)["iters"]
                torch.cuda.synchronize()
                if k:
                    gts.append(1000.0 * (time.perf_counter() - t0))
        gms = statistics.median(gts)
        grad = {"workload": "grad256_2d x 16 (256^2, eta 500, omega 0.7, V = r^2/2 + 0.1 S_i)",
                "value": 16 * 1000.0 / gms, "unit": "ground states + gradients / s", "ms_per_step": gms,
                "steps": "batched mixed solve (one graph launch) + per instance gpe_energy_grad (dE/dV, dE/deta, "
                         "dE/domega) and gpe_density_adjoint (tangent solve to 1e-10) in FP64",
                "converged": int(sum(r["status"] == gpe.GPE_OK for r in greps)),
                "adjoint_iters_total": adj_iters, "timing": "host clock around synchronised work, median of 2"}
        del gphi, gphi0, Vd

    # ---------------- context: the paper's 512^2 examples (Tables 2 and 3 of Section 6) ----------------
    # V = r^2/2, eta = 500 on [-16,16]^2 (h = 1/16): the lowest-energy states at omega = 0.9 from
    # phi_d (fixed grid) and at omega = 0.95 by multigrid 64 -> 512 from Thomas-Fermi, mixed
    # precision to ||r||_inf < 1e-8, timed with CUDA events; the paper's Matlab times (laptop,
    # FP64, energy criterion 1e-14) beside them as context only.
    paper = None
    if not args.no_paper and rank == 0:
        from paper_1611_02045_gb300.multigrid import multigrid_solve
        n5, L5 = (512, 512), (16.0, 16.0)
        V5 = I.harmonic(n5, L5)
        popts = gpe.solve_opts_default()
        popts.max_iter = 60000
        with gpe.Context(n5, L5, 500.0, 0.9, V5, prec=gpe.GPE_MIXED) as c5:
            p50 = torch.from_numpy(I.phi_d(n5, L5, 0.9)).to(dev)
            p5 = p50.clone()
            c5.pcg_solve(p5, popts)  # warm-up (graph build)
            p5.copy_(p50)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            r5 = c5.pcg_solve(p5, popts, check=True)
            b.record(stream)
            b.synchronize()
        ms5 = a.elapsed_time(b)
        multigrid_solve([64, 128, 256, 512], L5, 500.0, 0.95, lambda nn, LL: I.harmonic(nn, LL), opts=popts)  # warm-up
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        _, mreps = multigrid_solve([64, 128, 256, 512], L5, 500.0, 0.95, lambda nn, LL: I.harmonic(nn, LL),
                                   opts=popts)
        b.record(stream)
        b.synchronize()
        msm = a.elapsed_time(b)
        paper = {"setting": "512^2 on [-16,16]^2, V = r^2/2, eta = 500 (Section 6, Example eg:diff_initial_fix_grid)",
                 "fixed_grid_omega_0.9_phi_d": {"E": r5["E"], "paper_E": 4.7777, "ms": ms5, "iters": r5["iters"],
                                                "res_inf": r5["res_inf"], "paper_cpu_s": 1051.1},
                 "multigrid_omega_0.95_thomas_fermi": {"E": mreps[-1]["E"], "paper_E": 3.7414, "ms": msm,
                                                       "iters": [r["iters"] for r in mreps],
                                                       "res_inf": mreps[-1]["res_inf"], "paper_cpu_s": 621.9},
                 "note": "paper: Matlab R2015a on a laptop, FP64, stop at |E_{n+1}-E_n| < 1e-14; here mixed "
                         "precision to ||r||_inf < 1e-8 -- context, not a comparison of equal work"}

    # ---------------- accuracy: the same workload solved by this library in FP64 ----------------
    def timed(fn):
        l2_flush.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        out = fn()
        b.record(stream)
        b.synchronize()
        return out, a.elapsed_time(b)

    accuracy, fp64_solve = None, None
    if rank == 0 and not args.no_fp64:
        ctx64 = gpe.Context(n, L, w["eta"], w["omega"], w["V"], prec=gpe.GPE_FP64)
        if not args.no_autotune:
            ctx64.autotune(iters=10)
        p64_0 = torch.from_numpy(w["phi0"].copy()).to(dev)
        p64 = torch.empty_like(p64_0)

        def solve64():
            p64.copy_(p64_0)
            return ctx64.pcg_solve(p64, check=True)

        solve64()  # warm-up (graph build)
        r64, ms64 = timed(solve64)
        ctx64.close()
        fp64_solve = {"value": 1000.0 / ms64, "unit": UNIT, "ms_per_step": ms64, "iters": r64["iters"],
                      "ms_per_iter": ms64 / max(r64["iters"], 1), "E": r64["E"], "res_inf": r64["res_inf"]}
        last = reps[-1]
        accuracy = {"E_mixed": last["E"], "E_fp64": r64["E"],
                    "err_vs_fp64": abs(last["E"] - r64["E"]) / abs(r64["E"]),
                    "res_inf_mixed": last["res_inf"], "res_inf_fp64": r64["res_inf"],
                    "reference": "this library's FP64 solve of the same workload (GPE_FP64, every pass in FP64)"}
        del p64, p64_0

    # ---------------- GPU library baseline: the same FP64 solve with torch.fft (cuFFT) ----------------
    # Reported beside this library's FP64 single-instance solve of the same workload (same algorithm,
    # same stopping rule); neither is the headline, which is the mixed-precision solve above.
    libfft = None
    if not args.no_libfft and rank == 0:
        from baseline.libfft_pcg import LibFFTPCG
        lb = LibFFTPCG(n, L, w["eta"], w["omega"], w["V"], device=dev)
        lb.solve(w["phi0"], max_iter=20)  # warm-up: cuFFT plans, allocator
        lrep, lms = timed(lambda: lb.solve(w["phi0"]))
        libfft = {"kind": "plain PyTorch + torch.fft (cuFFT), complex128 PCG_C (baseline/libfft_pcg.py)",
                  "workload": WORKLOAD, "value": 1000.0 / lms, "unit": UNIT, "ms_per_step": lms,
                  "iters": lrep["iters"], "ms_per_iter": lms / max(lrep["iters"], 1), "status": lrep["status"],
                  "E": lrep["E"], "res_inf": lrep["res_inf"], "gb300_fp64": fp64_solve}
        del lb

    # ---------------- CPU baseline (oracle, bounded samples) ----------------
    cpu = None
    if rank == 0 and not args.no_cpu_baseline:
        from oracle import gpe_oracle as O
        it_or = oracle_iterations(WORKLOAD)
        t_it, k = oracle_sample(seconds=10.0)
        cores = cpu_cores()
        t_all, k_all, _ = oracle_all_cores(10.0, 400, cores)
        cpu = {"value": cores / (t_all * it_or), "unit": UNIT, "cores": cores, "kind": "oracle",
               "cpu_model": cpu_model(),
               "sample": f"{cores} processes (one per host core) each timing >= {k_all} FP64 numpy PCG_C "
                         f"iterations of {WORKLOAD} ({t_all * 1e3:.1f} ms/iteration per process), scaled by the "
                         f"oracle's own {it_or} iterations per solve (tests/golden/oracle_iterations.json)",
               "single_core": {"value": 1.0 / (t_it * it_or), "ms_per_iteration": t_it * 1e3, "iters_timed": k},
               "oracle_iters_per_solve": it_or}
        t_naive, t_fft, it64 = oracle_naive_64()
        cpu["naive_dft_64"] = {"workload": "c64_2d (64x64, complex128, ||r||_inf < 1e-8)", "iters": it64,
                               "s_per_solve_naive_dft": t_naive, "s_per_solve_fft": t_fft, "cores": 1}
        # the oracle re-evaluates the energy and residual at the GPU's mixed-precision answer
        po = O.Problem(n, L, w["eta"], w["omega"], w["V"])
        ph = phi_d.detach().cpu().numpy().astype(np.complex128)
        lam = O.chemical_potential(po, ph)
        E_or = O.energy(po, ph)
        cpu["oracle_check_of_gpu_result"] = {
            "res_inf": float(np.max(np.abs(O.apply_H(po, ph, ph) - lam * ph))), "E": E_or,
            "E_rel_diff_vs_gpu": abs(E_or - reps[-1]["E"]) / abs(E_or), "norm": float(O.norm(po, ph))}

    if rank == 0:
        last = reps[-1]
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": max(args.warmup, 3), "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "c64 + double-single/FP32 refinement + f64 scalars", "data": "synthetic",
            "config": {"workload": WORKLOAD, "grid": "256x256", "domain": "[-16,16]^2", "eta": 1000.0,
                       "omega": 0.9, "V": "r^2/2", "precision": "mixed (c64 phase, c128 refinement)",
                       "tol_res_inf": 1e-8, "iters": last["iters"], "iters_c64": last["iters_lo"],
                       "iters_fp64": last["iters_fp64"],
                       "loop": {3: "cluster (complex64 phase) + graph (refinement)", 2: "persistent kernel",
                                1: "graph", 0: "host loop"}[last["loop_kind"]],
                       "loop_note": last.get("note", ""),
                       "E": last["E"], "res_inf": last["res_inf"],
                       "l2": "flushed (256 MB write) before every step", "parallelism": f"replicas{world}",
                       "plans": tune and tune["plans"], "autotune_s": tune and tune["seconds"]},
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak, "traffic": hphi_traffic(),
                         "traffic_source": os.path.relpath(HPHI_PROFILE, ROOT),
                         "kernel": "h_batch_flow (gpe_apply_H_batch: row and column units of 16 lines from one "
                                   "ticket queue on persistent blocks, TMA-fed stages, TMA reduce-add of the "
                                   "column part)",
                         "grid": f"{NB} x 256x256", "bytes_per_launch": hbytes,
                         "ms_per_launch": h_ms, "peak_source": "MEASURED_PEAKS.json hbm_gbs (measured)"},
            "e2e": {"value": e2e_val, "unit": UNIT, "h2d_bytes_per_step": 16 * N, "d2h_bytes_per_step": 16 * N},
            "gpu_launches": launches,
            "clocks": clk,
            "accuracy": accuracy,
            "alu_peaks_gflops": alu,
            "fft_passes": fftpass,
            "fp64_roofline": fp64_roof,
            "cpu_baseline": cpu,
            "secondary": secondary,
            "batch": batch,
            "grad": grad,
            "paper_examples": paper,
            "libfft_baseline": libfft,
        }
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()

#!/usr/bin/env python
"""Benchmark of the two-step reconstruction on the 1024-pixel, 9.27M-row
SKA-Mid-like workload (FP32 operator, FP64 reductions, 5 major cycles x 100
FISTA iterations per step, split at 10 % of max |uv|).

One step = one complete two-step reconstruction (every row of the hot path:
degrid + residual, grid + adjoint FFT, PSF / filters / K^, step size,
lambda and sigma estimates, FISTA minor cycles, image updates) over the
workload's visibilities, already resident in HBM.

value  = visibilities passed through a degrid + grid pair per second of
         degrid + grid kernel time (FFT excluded, timed separately), summed
         over all ranks / the slowest rank's kernel time.
e2e    = the same visibilities per second of wall time of the public call
         with host buffers: pinned host -> device copy of the visibilities,
         the reconstruction, device -> host copy of both images.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
Multi-GPU (torchrun, one rank per GPU): every rank reconstructs its own
independent observation (its own sky seed); no data-path collective.
"""
from __future__ import annotations

import argparse
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

METRIC = "vis/s grid+degrid, FISTA iters/s, time-to-ε: chosen vs plain form on 1 GB300"
UNIT = "vis/s"
L2_FLUSH_BYTES = 256 << 20
N_MAJOR, FISTA_ITERS = 5, 100


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["mine", "reference"], default="mine")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-sample-rows", type=int, default=1_000_000)
    ap.add_argument("--precision", default="fp32", choices=["fp32", "fp32_kahan", "fp64"])
    ap.add_argument("--no-time-to-eps", action="store_true")
    # smaller schedules for profiler captures only (a bench line needs the defaults)
    ap.add_argument("--n-major", type=int, default=N_MAJOR)
    ap.add_argument("--fista-iters", type=int, default=FISTA_ITERS)
    ap.add_argument("--eps", type=float, default=1e-6)
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--record-traffic", nargs="+", default=None, metavar="NCU_CSV",
                    help="write the DRAM traffic of one FISTA pass, from ncu --page raw --csv "
                         "exports, to profiles/")
    ap.add_argument("--batched-channels", type=int, default=64)
    ap.add_argument("--no-c1", action="store_true",
                    help="skip the 128-pixel oracle reconstruction of the CPU baseline")
    ap.add_argument("--oracle-phases", default=None, help=argparse.SUPPRESS)
    return ap.parse_args()


def dist_env():
    return (int(os.environ.get("RANK", 0)), int(os.environ.get("LOCAL_RANK", 0)),
            int(os.environ.get("WORLD_SIZE", 1)))


def reduce_over_ranks(pg, device, maxes, sums):
    """Max over ranks of `maxes` (times) and sum over ranks of `sums`
    (work units); identity without a process group."""
    if pg is None:
        return list(maxes), list(sums)
    import torch
    t = torch.tensor([float(x) for x in maxes], device=device, dtype=torch.float64)
    v = torch.tensor([float(x) for x in sums], device=device, dtype=torch.float64)
    pg.all_reduce(t, op=pg.ReduceOp.MAX)
    pg.all_reduce(v, op=pg.ReduceOp.SUM)
    return t.tolist(), v.tolist()


# ---------------------------------------------------------------------------
# the oracle on the host cores (cpu_baseline leg and --impl reference)
# ---------------------------------------------------------------------------
def oracle_vis_rate(w, rows: int):
    """Oracle degrid + grid (FFT time measured separately and removed) on the
    first `rows` rows of the workload, single host thread."""
    import numpy as np
    from oracle.gridding import GriddedOperator
    rows = min(rows, w.nvis)
    A = GriddedOperator(w.u[0][:rows], w.v[0][:rows], w.npix, w.pixel_size)
    x = np.zeros((w.npix, w.npix))
    x[w.npix // 2, w.npix // 2] = 1.0
    t0 = time.perf_counter()
    A.forward(x)
    t1 = time.perf_counter()
    A.adjoint(w.vis[0][:rows])
    t2 = time.perf_counter()
    g = np.zeros((A.ngrid, A.ngrid), complex)
    t3 = time.perf_counter()
    np.fft.fft2(g)
    np.fft.ifft2(g)
    t4 = time.perf_counter()
    t = (t2 - t0) - (t4 - t3)
    return rows / t, t, rows


def _oracle_rows_worker(path, lo, hi, npix, pixel_size):
    """(pool worker, one BLAS thread) oracle degrid + grid of rows [lo, hi) of
    the sample file; returns the seconds spent."""
    import numpy as np
    from oracle.gridding import GriddedOperator
    d = np.load(path)
    A = GriddedOperator(d["u"][lo:hi], d["v"][lo:hi], npix, pixel_size)
    x = np.zeros((npix, npix))
    x[npix // 2, npix // 2] = 1.0
    t0 = time.perf_counter()
    A.forward(x)
    A.adjoint(d["vis"][lo:hi])
    return time.perf_counter() - t0


def oracle_phases(spec):
    """Time the oracle's phases on this process's BLAS threads (the parent
    sets them): degrid + grid of `rows` sample rows (FFT time removed), one
    forward + inverse Ng^2 FFT, one FISTA iteration of the 1024-pixel
    problem (M = 8, J = 4), and, if asked, the full 128-pixel two-step and
    single-step reconstruction.  With spec["pool"] > 1 the degrid + grid
    rows are split over that many single-thread worker processes (spawned).
    Prints one JSON object."""
    import numpy as np
    out = {"threads": spec["threads"]}
    d = np.load(spec["data"])
    npix, ps, rows = int(d["npix"]), float(d["pixel_size"]), int(spec["rows"])
    rows = min(rows, d["u"].size)
    if spec.get("pool", 1) > 1:
        import multiprocessing as mp
        k = spec["pool"]
        os.environ["OPENBLAS_NUM_THREADS"] = os.environ["OMP_NUM_THREADS"] = "1"
        os.environ["MKL_NUM_THREADS"] = "1"
        ctx = mp.get_context("spawn")
        bounds = [(rows * i // k, rows * (i + 1) // k) for i in range(k)]
        with ctx.Pool(k) as pool:
            pool.starmap(_oracle_rows_worker, [(spec["data"], 0, 64, npix, ps)] * k)   # warm
            t0 = time.perf_counter()
            pool.starmap(_oracle_rows_worker, [(spec["data"], a, b, npix, ps) for a, b in bounds])
            wall = time.perf_counter() - t0
        out["grid_degrid"] = {"rows": rows, "s": wall, "vis_per_s": rows / wall,
                              "processes": k}
    else:
        t = _oracle_rows_worker(spec["data"], 0, rows, npix, ps)
        out["grid_degrid"] = {"rows": rows, "s": t, "vis_per_s": rows / t, "processes": 1}
    ng = 2 * npix
    g = np.zeros((ng, ng), complex)
    t0 = time.perf_counter()
    np.fft.fft2(g)
    np.fft.ifft2(g)
    out["fft_ng2_pair_ms"] = 1000 * (time.perf_counter() - t0)
    if spec.get("fista"):
        from oracle import solver as osv
        from oracle.wavelets import Dictionary
        rng = np.random.default_rng(0)
        hh = np.exp(-0.5 * (osv.radial_frequency(npix) / (0.1 * npix)) ** 2)
        prob = osv.Problem("low", Dictionary(npix, 8, 4), hh, rng.standard_normal((npix, npix)),
                           0.1)
        t0 = time.perf_counter()
        osv.fista(prob, 1)
        t1 = time.perf_counter()
        osv.fista(prob, 2)
        t2 = time.perf_counter()
        out["fista_iteration_1024px_s"] = (t2 - t1) - (t1 - t0)
    if spec.get("c1"):
        import synth
        from oracle import imaging as oi
        w = synth.small_fp64()
        ro = oi.ReconOptions(n_major=5, fista_iters=200, lambda_rule="max_fixed",
                             lambda_low=1e-3, lambda_full=1e-3, lambda_single=1e-3)
        t0 = time.perf_counter()
        low, full = oi.reconstruct_two_step(w.vis[0], w.u[0], w.v[0], 128, w.pixel_size,
                                            w.ell_px, w.delta_px, ro)
        t1 = time.perf_counter()
        single = oi.reconstruct_single_step(w.vis[0], w.u[0], w.v[0], 128, w.pixel_size, ro)
        t2 = time.perf_counter()
        out["c1_two_step_s"] = t1 - t0
        out["c1_single_step_s"] = t2 - t1
        if spec.get("c1_images"):
            np.savez(spec["c1_images"], low=low.image, full=full.image, single=single.image)
    print(json.dumps(out), flush=True)


def host_cores():
    """(nproc, cores this process may run on)"""
    n = os.cpu_count() or 1
    try:
        aff = len(os.sched_getaffinity(0))
    except Exception:
        aff = n
    return n, aff


def run_oracle_phases(spec, threads):
    """oracle_phases in a fresh interpreter whose BLAS / OpenMP pools have
    `threads` threads (set before numpy loads)."""
    env = dict(os.environ)
    for k in ("OPENBLAS_NUM_THREADS", "OMP_NUM_THREADS", "MKL_NUM_THREADS"):
        env[k] = str(threads)
    spec = dict(spec, threads=threads)
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--oracle-phases",
                        json.dumps(spec)], env=env, capture_output=True, text=True, cwd=ROOT)
    if r.returncode != 0:
        raise RuntimeError(f"oracle timing failed: {r.stderr[-2000:]}")
    return json.loads(r.stdout.strip().splitlines()[-1])


def cpu_baseline_leg(w, rows, tmpdir, c1=True):
    """The oracle timed on this host: single-threaded and on all cores."""
    import numpy as np
    nproc, cores = host_cores()
    path = os.path.join(tmpdir, "oracle_sample.npz")
    n = min(max(rows, 1), w.nvis)
    n_all = min(w.nvis, max(n, 250_000 * cores))
    np.savez(path, u=np.asarray(w.u[0][:n_all]), v=np.asarray(w.v[0][:n_all]),
             vis=np.asarray(w.vis[0][:n_all]), npix=w.npix, pixel_size=w.pixel_size)
    c1_path = os.path.join(tmpdir, "c1_oracle_images.npz")
    one = run_oracle_phases({"data": path, "rows": n, "fista": True, "c1": c1,
                             "c1_images": c1_path if c1 else ""}, 1)
    allc = run_oracle_phases({"data": path, "rows": n_all, "fista": True, "pool": cores},
                             cores)
    value = one["grid_degrid"]["vis_per_s"]
    out = {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
           "sample": (f"oracle degrid+grid of the first {n} rows of this workload (FFT time "
                      f"removed), one thread, {one['grid_degrid']['s']:.1f} s"),
           "nproc": nproc, "cores_available": cores,
           "single_thread": {"grid_degrid_vis_per_s": value,
                             "fft_2048sq_pair_ms": one["fft_ng2_pair_ms"],
                             "fista_iteration_1024px_s": one.get("fista_iteration_1024px_s"),
                             "c1_two_step_s": one.get("c1_two_step_s"),
                             "c1_single_step_s": one.get("c1_single_step_s")},
           "all_cores": {"cores": cores,
                         "grid_degrid_vis_per_s": allc["grid_degrid"]["vis_per_s"],
                         "grid_degrid_rows": allc["grid_degrid"]["rows"],
                         "grid_degrid_processes": allc["grid_degrid"]["processes"],
                         "fista_iteration_1024px_s": allc.get("fista_iteration_1024px_s"),
                         "fista_threads": cores,
                         "fft_2048sq_pair_ms": allc["fft_ng2_pair_ms"],
                         "note": "degrid+grid split over single-thread processes; the FISTA "
                                 "iteration on the BLAS thread pool; numpy's FFT is "
                                 "single-threaded"}}
    return out, (c1_path if c1 and os.path.exists(c1_path) else None)


def run_reference(args):
    rank, _, world = dist_env()
    if rank != 0:
        return
    # one BLAS / OpenMP thread: the oracle as a single-threaded program
    for k in ("OPENBLAS_NUM_THREADS", "OMP_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ[k] = "1"
    import synth
    w = synth.ska_mid_like(device="cpu" if not _cuda_ok() else "cuda")
    for _ in range(max(args.warmup, 0)):
        oracle_vis_rate(w, min(args.cpu_sample_rows // 4, w.nvis))
    rates, secs = [], []
    for _ in range(args.steps):
        r, t, rows = oracle_vis_rate(w, args.cpu_sample_rows)
        rates.append(r)
        secs.append(t)
    value = sum(args.cpu_sample_rows for _ in rates) / sum(secs)
    sample = (f"oracle degrid+grid of the first {args.cpu_sample_rows} rows of the "
              f"{w.name} workload per step, FFT time removed")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
            "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1000 * statistics.mean(secs), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(w, "fp64"),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1,
                             "kind": "oracle", "sample": sample,
                             "nproc": host_cores()[0]},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def _cuda_ok():
    try:
        import torch
        return torch.cuda.is_available()
    except Exception:
        return False


def workload_config(w, precision, n_major=N_MAJOR, fista_iters=FISTA_ITERS):
    return {"workload": w.name, "npix": w.npix, "nvis": int(w.nvis),
            "partition": f"ell = 10% of max|uv| ({w.ell_px:.1f} px), delta = {w.delta_px} px",
            "n_major": n_major, "fista_iters": fista_iters, "precision": precision,
            "lambda": "0.05 ||i~_n||_2 2^n (both steps)", "wavelets": "db1-db8, 4 levels",
            "es_kernel": "W=7, 2x oversampling",
            "l2": "flushed between timed steps (256 MiB write)"}


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------
class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.QUERY}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except Exception:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, mx, reasons = [], [], set()
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
            for n, v in zip(names, f[5:9]):
                if v.lower() in ("active", "1"):
                    reasons.add(n)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx),
                "reasons": sorted(reasons), "samples": len(sm)}


# ---------------------------------------------------------------------------
def record_traffic(paths, precision):
    """DRAM bytes per span of the FISTA kernel families from ncu raw-page CSV
    exports of one FISTA pass, the files (one kernel each, or several) given
    in launch order (synthesis levels J..1, the spectral step's kernels,
    analysis levels 1..J)."""
    import csv
    fams = {}
    launches = []
    for path in paths:
        with open(path) as f:
            rows = [r for r in csv.reader(f)]
        start = next(i for i, r in enumerate(rows) if "Kernel Name" in r)   # after ncu's log lines
        rows = rows[start:]
        h = rows[0]
        units = rows[1]
        idx = {n: i for i, n in enumerate(h)}
        scale = {"byte": 1.0, "Kbyte": 1e3, "Mbyte": 1e6, "Gbyte": 1e9}
        for r in rows[2:]:
            name = r[idx["Kernel Name"]]
            b = 0.0
            for m in ("dram__bytes_read.sum", "dram__bytes_write.sum"):
                b += float(r[idx[m]].replace(",", "")) * scale[units[idx[m]]]
            launches.append((name, b))
    # (one launch per level, in order)
    syn = [b for n, b in launches if "fine_synthesis" in n]
    ana = [b for n, b in launches
           if "analysis_level_kernel" in n or "fine_analysis_kernel" in n]
    if syn:
        fams["synth"], fams["synth_l1"] = sum(syn[:-1]), syn[-1]
    if ana:
        fams["analysis_l1"], fams["analysis"] = ana[0], sum(ana[1:])
    for n, b in launches:
        base = n.split("(")[0].split("<")[0].split("::")[-1].replace("void ", "").strip()
        # (the operator kernels' traffic depends on the call's partition, so
        # only the per-pass families are recorded)
        for fam, kname in (("spec_mul", "spec_mul_kernel"), ("spec_mul", "spec_col_kernel"),
                           ("fft_r2c", "row_r2c_kernel"), ("fft_c2r", "row_c2r_kernel")):
            if base == kname and fam not in fams:
                fams[fam] = b
    rec = {"precision": precision, "workload": "ska-mid-like-1024px-9266880vis",
           "note": "DRAM read + write bytes per span of each kernel family, from ncu; valid "
                   "while the kernel sources hash to source_sha256",
           "families": {f: {"dram_bytes_per_span": b, "source_sha256": kernel_source_digest(f)}
                        for f, b in fams.items()}}
    with open(TRAFFIC_FILE, "w") as f:
        json.dump(rec, f, indent=1)
    print(json.dumps(rec))


def main():
    args = parse()
    if args.oracle_phases:
        oracle_phases(json.loads(args.oracle_phases))
        return
    if args.record_traffic:
        record_traffic(args.record_traffic, args.precision)
        return
    if args.impl == "reference":
        run_reference(args)
        return
    import numpy as np
    import torch
    import synth

    rank, local_rank, world = dist_env()
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    pg = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
        pg = dist
    if rank == 0:
        from paper_2406_18356_gb300 import _build
        _build.build()
    if pg:
        pg.barrier()
    import paper_2406_18356_gb300 as ms
    ms.load_library()

    w = synth.ska_mid_like(seed=rank, device=str(dev))
    plan = ms.Plan(w.u[0], w.v[0], w.npix, w.pixel_size, w.ell_px, w.delta_px,
                   precision=args.precision, device=local_rank)
    opts = ms.ReconOptions(n_major=args.n_major, fista_iters=args.fista_iters)
    vis = torch.from_numpy(w.vis[0]).to(dev).to(plan.complex_dtype)
    low = torch.empty((w.npix, w.npix), dtype=plan.real_dtype, device=dev)
    img = torch.empty_like(low)
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device=dev)

    for _ in range(max(args.warmup, 3)):
        plan.reconstruct_two_step(vis, opts, low_out=low, out=img)
    torch.cuda.synchronize()

    # ---- timed region (captured-graph minor cycles) ----
    clocks = ClockSampler(local_rank) if rank == 0 else None
    if clocks:
        clocks.start()
        time.sleep(0.3)
    if pg:
        pg.barrier()
    torch.cuda.synchronize()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.nvtx.range_push("timed")   # lets a profiler capture just this region
    ev0.record()
    tot = dict(vis=0, grid_ms=0.0, fft_ms=0.0, minor_ms=0.0, iters=0, elapsed=0.0)
    for _ in range(args.steps):
        flush.fill_(1.0)
        _, _, st = plan.reconstruct_two_step(vis, opts, low_out=low, out=img)
        tot["vis"] += st.gridded_vis
        tot["grid_ms"] += st.grid_ms
        tot["fft_ms"] += st.fft_ms
        tot["minor_ms"] += st.minor_ms
        tot["iters"] += st.total_iterations
        tot["elapsed"] += st.elapsed_ms
    ev1.record()
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_pop()
    if pg:
        pg.barrier()
    clk = clocks.stop() if clocks else None
    wall_ms = ev0.elapsed_time(ev1)
    grid_s = tot["grid_ms"] / 1000.0
    vis_total = tot["vis"]
    (wall_ms, grid_s), (vis_total,) = reduce_over_ranks(pg, dev, [wall_ms, grid_s],
                                                        [vis_total])
    value = vis_total / grid_s
    ms_per_step = wall_ms / args.steps
    fista_rate = tot["iters"] / (tot["minor_ms"] / 1000.0)
    # a pass: four levels each way and the spectral step's three kernels; a
    # major cycle: its residual image (7) and the minor cycle's set-up and
    # update (7); a step: the last residual image and its set-up (2344 of the
    # launch list's at one major cycle of 100 iterations)
    kernels_per_pass = 2 * 4 + 3
    passes_per_cycle = math.ceil((args.fista_iters + 1) / 8) * 8
    launches_per_step = 2 * (args.n_major * (passes_per_cycle * kernels_per_pass + 7 + 7) + 7 + 7)
    gpu_launches = launches_per_step * args.steps

    # ---- per-kernel durations: the same steps with every kernel family
    #      bracketed by CUDA events on the plan's stream ----
    roofline = None
    prof = None
    if rank == 0:
        plan.kernel_profile(reset=True)
        plan.set_profiling(True)
        for _ in range(args.steps):
            flush.fill_(1.0)
            plan.reconstruct_two_step(vis, opts, low_out=low, out=img)
        prof = plan.kernel_profile(reset=True)
        plan.set_profiling(False)
        roofline = roofline_of(prof, w, plan, args)

    # ---- end to end through the public call with host buffers ----
    e2e = None
    if not args.no_e2e:
        hvis = torch.from_numpy(w.vis[0]).to(plan.complex_dtype).pin_memory()
        hlow = torch.empty((w.npix, w.npix), dtype=plan.real_dtype).pin_memory()
        himg = torch.empty_like(hlow).pin_memory()
        dvis = torch.empty_like(vis)
        plan.reconstruct_two_step(vis, opts, low_out=low, out=img)
        torch.cuda.synchronize()
        if pg:
            pg.barrier()
        t0 = time.perf_counter()
        e2e_vis = 0
        for _ in range(args.steps):
            flush.fill_(1.0)
            dvis.copy_(hvis, non_blocking=True)
            _, _, st = plan.reconstruct_two_step(dvis, opts, low_out=low, out=img)
            hlow.copy_(low, non_blocking=True)
            himg.copy_(img, non_blocking=True)
            torch.cuda.synchronize()
            e2e_vis += st.gridded_vis
        e2e_s = time.perf_counter() - t0
        (e2e_s,), (e2e_vis,) = reduce_over_ranks(pg, dev, [e2e_s], [e2e_vis])
        e2e = {"value": e2e_vis / e2e_s, "unit": UNIT,
               "h2d_bytes_per_step": int(hvis.numel() * hvis.element_size()),
               "d2h_bytes_per_step": int(2 * hlow.numel() * hlow.element_size()),
               "ms_per_step": 1000 * e2e_s / args.steps}

    # the interleaved two-image pipeline (Sect. 6's sketch) on the same data
    # and schedule: n_major cycles per node, both nodes' minor cycles batched
    interleaved = None
    if rank == 0:
        plan.reconstruct_interleaved(vis, opts)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        _, _, _, ist = plan.reconstruct_interleaved(vis, opts)
        e1.record()
        torch.cuda.synchronize()
        interleaved = {"ms": e0.elapsed_time(e1), "two_step_ms": ms_per_step,
                       "fista_iterations": int(sum(s_.total_iterations for s_ in ist)),
                       "note": "node L (V_L) and node H (V_H), each n_major cycles of "
                               "fista_iters; the two-step runs n_major per step in sequence"}

    tte = None
    errors = {}
    if rank == 0 and not args.no_time_to_eps:
        tte, low64, img64 = time_to_eps(ms, w, dev, args.eps)
        if args.precision != "fp64":
            # the timed run's images against the plain FP64 form of the same schedule
            rel = lambda a, b: float((a.double().cpu() - b).norm() / b.norm())
            errors["vs_fp64_gpu"] = {"two_step_low": rel(low, low64),
                                     "two_step_full": rel(img, img64),
                                     "workload": w.name}
    plan.close()

    batched = None
    if rank == 0 and not args.no_batched:
        batched = batched_leg(ms, dev, args.batched_channels, args.precision)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        import tempfile
        with tempfile.TemporaryDirectory() as tmp:
            cpu, c1_path = cpu_baseline_leg(w, args.cpu_sample_rows, tmp, c1=not args.no_c1)
            if c1_path:
                errors["c1_vs_oracle"] = c1_error_vs_oracle(ms, dev, c1_path, args.precision)

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
                "steps": args.steps, "warmup": max(args.warmup, 3), "ms_per_step": ms_per_step,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
                "dtype": "f32" if args.precision != "fp64" else "f64", "data": "synthetic",
                "config": workload_config(w, args.precision, args.n_major, args.fista_iters),
                "fista_iters_per_s": fista_rate,
                "step_breakdown_ms": {"grid_degrid": tot["grid_ms"] / args.steps,
                                      "fft_grid": tot["fft_ms"] / args.steps,
                                      "minor_cycles": tot["minor_ms"] / args.steps},
                "gpu_launches": gpu_launches,
                "roofline": roofline, "cpu_baseline": cpu, "e2e": e2e, "clocks": clk,
                "time_to_eps": tte, "batched": batched, "interleaved": interleaved,
                "image_rel_l2_errors": errors or None,
                "kernel_ms_per_step": {k: round(v[1] / args.steps, 4) for k, v in prof.items()}
                if prof else None}
        print(json.dumps(line), flush=True)
    if pg:
        pg.barrier()
        pg.destroy_process_group()


def time_to_eps(ms, w, dev, eps, ref_iters=3000, max_iters=4000):
    """Time to the same objective tolerance, chosen form against plain form,
    on this GPU.  Problems: the first minor cycle of each step of the
    two-step method on this workload: step one's (Eq. LowRes) on i~_L1, and
    step two's (Eq. FullRes) on i~_H1 with i^_L from a plain FP64 step one
    of the benchmark schedule (5 x 100).  Both forms get the same input
    images (computed in FP64).  F* is the lowest objective of a ref_iters
    iteration plain FP64 run of each problem; each form then runs FISTA from
    zero until F(beta_k) <= F* (1 + eps) (the library's objective target;
    the device flag is read every 32 iterations), timed with CUDA events.
    Chosen form: FP32 data with FP64 reductions (the FP32 + Kahan plan).
    Also returns the FP64 two-step images (the plain form of the benchmark
    schedule) for the error of the FP32 images."""
    import numpy as np
    import torch
    plan64 = ms.Plan(w.u[0], w.v[0], w.npix, w.pixel_size, w.ell_px, w.delta_px,
                     precision="fp64", device=dev.index or 0)
    vis64 = torch.from_numpy(w.vis[0]).to(dev).to(plan64.complex_dtype)
    low64, img64, _ = plan64.reconstruct_two_step(vis64, ms.ReconOptions(n_major=N_MAJOR,
                                                                         fista_iters=FISTA_ITERS))
    res = {"low": plan64.grid("L", vis64), "full": plan64.grid("H", vis64)}
    lam = {k: plan64.lam(r, 0.05, 1) for k, r in res.items()}
    s2 = plan64.sigma2_hat(res["full"])
    kw = {"low": {}, "full": {"l_low": low64, "sigma2": s2, "eta2": 1e-3 * s2}}
    fstar = {}
    for k in ("low", "full"):
        _, st = plan64.minor_cycle(k, res[k], lam[k], ref_iters, **kw[k])
        fstar[k] = float(np.min(st.trace))
    out = {"eps": eps, "reference_iterations": ref_iters, "max_iters": max_iters,
           "workload": f"{w.name}: first minor cycle of step one and of step two",
           "target": "F(beta_k) <= F* (1 + eps), F* from the long plain FP64 run",
           "f_star": fstar,
           "chosen_parts": "FP32 data, Kahan-compensated gridding, FP64 reductions; the "
                           "batched form is measured in the batched leg; the learned warm "
                           "start needs a trained network and is not part of this leg"}
    for form, plan in (("plain", plan64), ("chosen", None)):
        if plan is None:
            plan = ms.Plan(w.u[0], w.v[0], w.npix, w.pixel_size, w.ell_px, w.delta_px,
                           precision="fp32_kahan", device=dev.index or 0)
        cast = lambda t: t.to(plan.real_dtype).contiguous()
        rec = {}
        for k in ("low", "full"):
            kk = {a: (cast(b) if torch.is_tensor(b) else b) for a, b in kw[k].items()}
            plan.set_objective_target(float("-inf"))
            plan.minor_cycle(k, cast(res[k]), lam[k], 16, **kk)   # warm: K^, graph
            plan.set_objective_target(fstar[k] * (1 + eps))
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            _, st = plan.minor_cycle(k, cast(res[k]), lam[k], max_iters, **kk)
            e1.record()
            torch.cuda.synchronize()
            plan.set_objective_target(float("-inf"))
            rec[k] = {"ms": e0.elapsed_time(e1), "iterations": st.iterations,
                      "reached": bool(st.converged), "objective": st.objective}
        rec["ms"] = rec["low"]["ms"] + rec["full"]["ms"]
        out[form] = rec
        if form == "chosen":
            plan.close()
    out["speedup"] = out["plain"]["ms"] / out["chosen"]["ms"]
    plan64.close()
    return out, low64.double().cpu(), img64.double().cpu()


def c1_error_vs_oracle(ms, dev, c1_path, precision):
    """Relative L2 error of this form's 128-pixel two-step and single-step
    images (5 x 200, lambda = 1e-3 max|i~_1|) against the FP64 oracle's."""
    import numpy as np
    import torch
    import synth
    ref = np.load(c1_path)
    w = synth.small_fp64()
    plan = ms.Plan(w.u[0], w.v[0], 128, w.pixel_size, w.ell_px, w.delta_px,
                   precision=precision, device=dev.index or 0)
    opts = ms.ReconOptions(n_major=5, fista_iters=200, lambda_rule="max_fixed",
                           lambda_low=1e-3, lambda_full=1e-3, lambda_single=1e-3)
    tv = torch.from_numpy(w.vis[0]).to(dev).to(plan.complex_dtype)
    low, img, _ = plan.reconstruct_two_step(tv, opts)
    single, _ = plan.reconstruct_single_step(tv, opts)
    plan.close()
    rel = lambda a, b: float(np.linalg.norm(a.double().cpu().numpy() - b) / np.linalg.norm(b))
    return {"workload": w.name, "precision": precision, "two_step_low": rel(low, ref["low"]),
            "two_step_full": rel(img, ref["full"]), "single_step": rel(single, ref["single"])}


def batched_leg(ms, dev, nchan, precision, steps=3):
    """The batched form on nchan channels x 1024^2 (the layout of the main
    workload, uv scaled per channel over 350-1050 MHz, U(0, 0.5) random
    flagging per channel): one degrid + grid pass over both partitions of
    every channel, as one batched call pair against one call pair per
    (channel, partition) job; every channel's step-one minor cycle as one
    batched call against one call per channel; and the whole two-step
    reconstruction of every channel (5 + 5 major cycles of 100 iterations)
    as one batched call against one call per channel.  The gridding layout
    (tile side, rows per work item) is the autotuner's pick on channel 0.
    Visibility values are random (the kernels' time does not depend on
    them)."""
    import torch
    import synth
    t0 = time.perf_counter()
    w = synth.multi_channel(npix=1024, nchan=nchan, seed=11)
    gen_s = time.perf_counter() - t0
    tile, chunk, tune_ms = ms.ms_plan_autotune(w.u[:1], w.v[:1], w.npix, w.pixel_size, w.ell_px,
                                               w.delta_px, flags=w.flags[:1],
                                               precision=precision, device=dev.index or 0)
    plan = ms.Plan(w.u, w.v, w.npix, w.pixel_size, w.ell_px, w.delta_px, flags=w.flags,
                   precision=precision, device=dev.index or 0, tile=tile, chunk=chunk)
    del w.u, w.v
    g = torch.Generator(device=dev).manual_seed(3)
    jobs = [(c, p) for c in range(nchan) for p in ("L", "H")]
    vis = {c: torch.randn(plan.nvis, dtype=plan.complex_dtype, device=dev, generator=g)
           for c in range(nchan)}
    imgs = [torch.randn((w.npix, w.npix), dtype=plan.real_dtype, device=dev, generator=g)
            for _ in jobs]
    vin = [vis[c] for c, _ in jobs]
    vout = [torch.zeros(plan.nvis, dtype=plan.complex_dtype, device=dev) for _ in jobs]
    dirty = [torch.empty((w.npix, w.npix), dtype=plan.real_dtype, device=dev) for _ in jobs]
    rows = sum(plan.partition_counts(c)[p] for c, p in jobs)

    def batched_pass():
        plan.degrid_batch(jobs, imgs, vis_obs=vin, outs=vout)
        plan.grid_batch(jobs, vout, outs=dirty)

    def per_job_pass():
        for (c, p), x, vo, o, d in zip(jobs, imgs, vin, vout, dirty):
            plan.degrid(p, x, vo, out=o, chan=c)
            plan.grid(p, o, out=d, chan=c)

    out = {"workload": f"{nchan} channels x 1024^2, 350-1050 MHz, U(0,0.5) flagging, "
                       f"L and H partitions of every channel ({len(jobs)} jobs)",
           "rows_per_pass": int(rows), "precision": precision,
           "host_uv_generation_s": round(gen_s, 1),
           "autotuned_layout": {"tile": tile, "chunk": chunk, "degrid_grid_ms_chan0": tune_ms}}
    for name, fn in (("batched", batched_pass), ("per_job", per_job_pass)):
        fn()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(steps):
            fn()
        e1.record()
        torch.cuda.synchronize()
        ms_ = e0.elapsed_time(e1) / steps
        out[name] = {"ms_per_pass": ms_, "vis_per_s": rows / (ms_ / 1000.0)}
    # kernel time of the batched degrid + grid launches (FFT, pad, crop excluded)
    plan.kernel_profile(reset=True)
    plan.set_profiling(True)
    batched_pass()
    prof = plan.kernel_profile(reset=True)
    plan.set_profiling(False)
    kms = sum(prof[k][1] for k in ("degrid", "grid", "fold"))
    out["batched"]["kernel_ms_grid_degrid"] = kms
    out["batched"]["kernel_vis_per_s"] = rows / (kms / 1000.0)
    out["speedup_batched_vs_per_job"] = out["per_job"]["ms_per_pass"] / out["batched"]["ms_per_pass"]
    # the batched minor cycle: step one's problem (Eq. LowRes) of every
    # channel, on its L partition's dirty image, FISTA_ITERS iterations each,
    # as one batched call against one minor-cycle call per channel
    fjobs = [{"step": "low", "chan": c, "residual": dirty[2 * c],
              "lam": plan.lam(dirty[2 * c], 0.05, 1)} for c in range(nchan)]
    plan.minor_cycle_batch(fjobs, FISTA_ITERS)   # workspace, graph
    _, bst = plan.minor_cycle_batch(fjobs, FISTA_ITERS)
    per_job_ms = 0.0
    for j in fjobs:
        plan.minor_cycle("low", j["residual"], j["lam"], FISTA_ITERS, chan=j["chan"])
    for j in fjobs:
        _, st = plan.minor_cycle("low", j["residual"], j["lam"], FISTA_ITERS, chan=j["chan"])
        per_job_ms += st.minor_ms
    job_its = nchan * (FISTA_ITERS + 1)
    out["minor_cycle"] = {
        "jobs": nchan, "iterations": FISTA_ITERS,
        "batched_ms": bst[0].minor_ms, "per_job_ms": per_job_ms,
        "batched_job_iterations_per_s": job_its / (bst[0].minor_ms / 1000.0),
        "per_job_iterations_per_s": job_its / (per_job_ms / 1000.0),
        "speedup_batched_vs_per_job": per_job_ms / bst[0].minor_ms}
    # the whole method on every channel (config 4's end-to-end form)
    opts = ms.ReconOptions(n_major=N_MAJOR, fista_iters=FISTA_ITERS)
    vlist = [vis[c] for c in range(nchan)]
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    _, _, rst = plan.reconstruct_two_step_batch(vlist, opts)
    e1.record()
    torch.cuda.synchronize()
    batched_ms = e0.elapsed_time(e1)
    e0.record()
    for c in range(nchan):
        plan.reconstruct_two_step(vlist[c], opts, chan=c)
    e1.record()
    torch.cuda.synchronize()
    per_ch_ms = e0.elapsed_time(e1)
    gridded = sum(st.gridded_vis for st in rst)
    out["two_step"] = {
        "channels": nchan, "schedule": f"{N_MAJOR} + {N_MAJOR} major cycles x {FISTA_ITERS}",
        "batched_ms": batched_ms, "per_channel_ms": per_ch_ms,
        "speedup_batched_vs_per_channel": per_ch_ms / batched_ms,
        "fista_iterations": int(sum(st.total_iterations for st in rst)),
        "gridded_vis": int(gridded), "gridded_vis_per_s": gridded / (batched_ms / 1000.0)}
    plan.close()
    return out


def _peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return d["hbm_gbs"], "measured"
    except Exception:
        return 6800.0, "fallback"


def fused_spectral_step(N, rsz):
    """Whether the library runs the spectral step fused with shared-memory
    column transforms (N a power of two whose blocks fit in shared memory)."""
    return N & (N - 1) == 0 and 16 <= N <= (8192 if rsz == 4 else 4096)


def family_bytes(fam, N, M, J, rsz, plan, ext=None):
    """Algorithmic HBM bytes of one span of a kernel family (what the
    operation must move at least once; per minor-cycle pass for the FISTA
    families, per call for the operator families).  rsz = bytes of a real,
    ext: only the (2 ext + 1)^2 grid cells around the origin are in use (None
    or N: all (2N)^2).

      analysis_l1  read the gradient image, read B_k and B_k-1 and write B_k+1
                   over the level-1 detail subbands (3 M (N/2)^2 each), write
                   the level-1 approximations: (1 + 9 M/4 + M/4) N^2 rsz.
      analysis     levels 2..J: read LL_j-1, the prox traffic of the detail
                   subbands, write LL_j (level J: the approximation goes
                   through the prox as well).
      synth_l1     read the level-1 details and approximations of all bases
                   (M N^2 values), write x: (M + 1) N^2 rsz.
      synth        levels J..2: read details + approximation input, write
                   LL_j-1.
      spec_mul     per half-plane element read X_k, X_k-1, B (complex) and
                   K (real), write S (complex): 9 rsz; fused with the column
                   transforms (N a power of two): read the row spectra Z,
                   X_k-1, B and K, write Z and X_k: 11 rsz.
      fft_r2c /    (our row transforms, N a power of two) read N^2 reals, write
      fft_c2r      the N (N/2 + 1) half-plane values, or the reverse.
      degrid       per row: packed cell (4 B) + offsets (2 rsz) + observed and
                   residual value (2 x 2 rsz), plus one read of the complex
                   grid's cells in use.
      grid         per row: packed cell + offsets + value (4 + 4 rsz), plus one
                   write of the complex grid's cells in use.
      fold         (the design's reduction of the gridding tiles) every work
                   item's scratch tile read once, the grid's cells in use
                   written once.
    """
    q = lambda j: (N >> j) ** 2   # subband side^2 at level j
    grid = 2 * rsz * (4 * N * N if ext is None or ext >= N else (2 * ext + 1) ** 2)
    if fam == "analysis_l1":
        return (N * N + 9 * M * q(1) + M * q(1)) * rsz
    if fam == "analysis":
        b = 0
        for j in range(2, J + 1):
            b += M * q(j - 1) + 9 * M * q(j) + (M * q(j) if j < J else 3 * M * q(j))
        return b * rsz
    if fam == "synth_l1":
        return (M * N * N + N * N) * rsz
    if fam == "synth":
        b = 0
        for j in range(2, J + 1):
            b += 3 * M * q(j) + M * q(j) + M * q(j - 1)
        return b * rsz
    if fam == "spec_mul":
        return (11 if fused_spectral_step(N, rsz) else 9) * rsz * N * (N // 2 + 1)
    if fam in ("fft_r2c", "fft_c2r") and fused_spectral_step(N, rsz):
        return N * N * rsz + N * (N // 2 + 1) * 2 * rsz
    if fam == "degrid":
        counts = plan.partition_counts()
        rows = (counts["L"] + counts["H"]) / 2.0
        return rows * (4 + 2 * rsz + 4 * rsz) + grid
    if fam == "grid":
        # per row: packed cell (4 B) + offsets (2 rsz) + value (2 rsz)
        counts = plan.partition_counts()
        rows = (counts["L"] + counts["H"]) / 2.0
        return rows * (4 + 4 * rsz) + grid
    if fam == "fold":
        # the design's reduction: read every work item's scratch tile, write
        # the cells in use once (mean of the two partitions' calls)
        b = 0.0
        for part in ("L", "H"):
            items, cells, cell_bytes = plan.partition_layout(part)
            b += items * cells * cell_bytes + grid
        return b / 2.0
    return None


FAMILY_SOURCE = {"synth": "wavelet_kernels.cu", "synth_l1": "wavelet_kernels.cu",
                 "analysis": "wavelet_kernels.cu", "analysis_l1": "wavelet_kernels.cu",
                 "spec_mul": "spectral_kernels.cu", "fft_r2c": "spectral_kernels.cu",
                 "fft_c2r": "spectral_kernels.cu", "degrid": "grid_kernels.cu",
                 "grid": "grid_kernels.cu", "fold": "grid_kernels.cu"}
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "dram_traffic_1024px_fp32.json")


def kernel_sources(name):
    """A kernel source and the csrc headers that it includes, directly or
    through one another."""
    import re
    csrc = os.path.join(ROOT, "paper_2406_18356_gb300", "csrc")
    found, todo = [], [name]
    while todo:
        f = todo.pop()
        path = os.path.join(csrc, f)
        if f in found or not os.path.exists(path):   # (include/mstep.h has no kernels)
            continue
        found.append(f)
        with open(path) as fh:
            todo += re.findall(r'^\s*#\s*include\s+"([^"]+)"', fh.read(), re.M)
    return [os.path.join(csrc, f) for f in sorted(found)]


def kernel_source_digest(fam):
    """sha256 of the sources that define a family's kernels, headers included:
    a recorded DRAM traffic is valid only for the same kernels."""
    import hashlib
    h = hashlib.sha256()
    for path in kernel_sources(FAMILY_SOURCE[fam]):
        with open(path, "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()


def recorded_traffic(fam, precision):
    """DRAM bytes (read + write) of one span of family `fam` from the
    committed ncu capture, or None when the capture is absent, of another
    precision, or the kernels changed since it was taken."""
    try:
        with open(TRAFFIC_FILE) as f:
            rec = json.load(f)
    except (OSError, ValueError):
        return None
    fr = rec.get("families", {}).get(fam)
    if not fr or rec.get("precision") != precision or fam not in FAMILY_SOURCE:
        return None
    if fr.get("source_sha256") != kernel_source_digest(fam):
        return None
    return fr.get("dram_bytes_per_span")


def roofline_of(prof, w, plan, args):
    """Roofline of the dominant kernel family of the library (largest share of
    kernel time, cuFFT's transforms excluded): algorithmic bytes of one span (family_bytes)
    over the span's average CUDA-event duration, against the measured HBM
    copy bandwidth."""
    hbm, kind = _peaks()
    rsz = 4 if args.precision != "fp64" else 8
    N, M, J = w.npix, 8, 4
    ext = plan.grid_extent() if plan is not None else None
    ours_fft = fused_spectral_step(N, rsz)   # else the FISTA transforms are cuFFT's
    mine = {k: v for k, v in prof.items()
            if (ours_fft or not k.startswith("fft")) and k != "fft_grid" and v[0] > 0}
    fam = max(mine, key=lambda k: mine[k][1])
    launches, total_ms = mine[fam]
    avg_s = total_ms / launches / 1000.0
    bytes_ = family_bytes(fam, N, M, J, rsz, plan, ext)
    others = {}
    for k, (n, t) in mine.items():
        b = family_bytes(k, N, M, J, rsz, plan, ext)
        if b:
            others[k] = round(b / (t / n / 1000.0) / 1e9 / hbm, 4)
    if bytes_ is None:
        return {"bound": "hbm", "kernel": fam, "achieved": None, "peak": hbm, "unit": "GB/s",
                "frac": None, "traffic": None, "peak_kind": kind, "frac_by_family": others}
    achieved = bytes_ / avg_s / 1e9
    traffic = recorded_traffic(fam, args.precision) if w.npix == 1024 else None
    return {"bound": "hbm", "kernel": fam, "achieved": achieved, "peak": hbm, "unit": "GB/s",
            "frac": achieved / hbm, "traffic": traffic,
            "traffic_source": os.path.relpath(TRAFFIC_FILE, ROOT) if traffic else None,
            "peak_kind": f"{kind} (hbm_gbs burst copy)",
            "algorithmic_bytes_per_launch": bytes_, "avg_launch_us": avg_s * 1e6,
            "launches": launches, "frac_by_family": others}


if __name__ == "__main__":
    main()

#!/usr/bin/env python
"""Benchmark of the HDF hot path on one GB300 (or N independent replicas).

A step is one pass of the hot path over the benchmark workload with the points already in
HBM: hdf_build (centre/scale, Chebyshev degree, radial cores, radial-basis Gram, eigen
truncation, radial factors, harmonics + U) followed by K~ V for the workload's V block.

Default workload (name in config.workload): mixture3_matern -- n = 1,000,000 points in R^3
from an 8-component isotropic Gaussian mixture (means U[-2,2]^3, sigma 0.3), Matern-3/2
with l = 1, tol = 1e-8, V with 64 N(0,1) columns, FP32 bulk (FP64 radial basis and cores).
The tolerance is beyond the degree cap (Matern-3/2 coefficients decay like i^-4), so the
factor is built at p = p_max and the achieved error is measured and reported.

Printed: one JSON line (rank 0).  value = points per second of whole steps, summed over
ranks; e2e = the same through the C ABI from pinned host buffers (H2D of x and V, build,
K~ V, D2H of Y; parts_ms: the device times of the copies, the build and the products of
each of its steps).  The roofline object describes the dominant kernel of the step.  The
FP64-bulk form of the same step is timed beside it (detail.fp64).

Other workloads (--workload):
  ball3_gauss     the plain FP64 method: n = 2,000 points uniform in the unit ball (d = 3), Gaussian
                  l = 0.5, tol 1e-6, one N(0,1) vector; step = hdf_build + K~ v with FP64 bulk,
                  the FP32-bulk form beside it; both checked against the dense kernel matrix; L2
                  is flushed before each step.
  cube4_gauss     the differentiation row: n = 500,000 points in [-1,1]^4, Gaussian l = 0.8,
                  tol 1e-6, FP32; step = hdf_build + hdf_matvec_adjoint (gradient of w^T K~ v
                  with respect to the points and l); the dominant kernel is the adjoint kernel.
  batch512_gauss  the batching row: 512 ragged sets (n log-uniform in [1000, 65536]), FP32;
                  step = hdf_build_batched + hdf_batch_matvec with 8 columns per set; value =
                  points of all sets per second.
  fig1_cauchy     the time-vs-n row (Fig. 1): N(0,I) points scaled to max norm 1, Cauchy l = 1,
                  tol 1e-3, FP32; step = one hdf_build at every (d, n), d in {3,4,5,6}, n in
                  {1e4, 1e5, 1e6, 1e7}; value = points of the sweep per second; detail holds
                  the build time of each (d, n) and the slope of log time against log n.
  fig3_rank5      the error-vs-rank row (Fig. 3, HDF only): 5,000 points in d = 5, four kernels
                  (sigma = 1) and ten tolerances, FP64; step = one hdf_build per (kernel, tol);
                  detail holds rank and the achieved |K - K~|_F / |K|_F of each against the
                  dense kernel matrix.
  krr8_clusters   the kernel-ridge-regression row (Sec. 4.2): 13,760 training and 6,880 test
                  points in d = 8 (synthetic stand-in for the paper's dataset), 30 k-means
                  clusters, Gaussian l = 0.5, lambda = 1, HDF blocks at tol 1e-3 (FP32 bulk);
                  step = hdf_kmeans + hdf_krr_build + hdf_krr_solve (rtol 1e-6) +
                  hdf_kernel_matvec for the test predictions; value = training points / s.
  normal5_cauchy  the large-rank row: n = 4,000,000 points in d = 5 (rotated standard normal,
                  standardised), Cauchy l = 2, tol 1e-4, FP32, 16 columns; U would take about
                  1.4 TB, so hdf_build keeps the matrix-free rows (the harmonic tails Z and the
                  first level factor times the radial factor) and K~V runs over them on the
                  tensor cores; step = hdf_build + K~V.
  cross3_gauss    the non-symmetric row: X = 1,000,000 mixture points, Y = 250,000 points of a
                  wider Gaussian cloud, Gaussian l = 1.5, tol 1e-6, FP32; step = hdf_build_cross
                  + K~ V (V: 16 columns over Y) + K~^T W (W: 16 columns over X); value = points
                  of both sets per second.

--impl reference times the CPU oracle (the only other implementation of this method here)
on a bounded sample of the same workload.
"""
import argparse
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

PEAKS_FALLBACK = {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}
# DRAM bytes (read + write) per stored U element, from one ncu capture of each kernel at the
# benchmark size (n = 1,000,000; dram__bytes_read.sum + dram__bytes_write.sum over n * ldU); the
# roofline's traffic is this figure times n * ldU of the timed launch.  Set an entry to None
# when its kernel changes, until it is captured again.
TRAFFIC_PER_U_ELEMENT = {"k_uwriter": 4.171, "k_tc_utv": 4.276, "k_tc_uw": 4.069}
METRICS = {
    "ball3_gauss": "factor-build points/s (build + K~v step) of the plain FP64 method, FP32 bulk beside it, vs the dense kernel matrix",
    "mixture3_matern": "factor-build points/s (build + K~V step) at stated rel. error, FP32 bulk vs FP64",
    "normal5_cauchy": "factor-build points/s (build + 16-column K~V of a matrix-free factor: U not stored), FP32 bulk",
    "cube4_gauss": "adjoint step points/s (build + gradient of w^T K~ v w.r.t. points and l), FP32 bulk",
    "batch512_gauss": "batched factor-build points/s (512 sets, build + 8-column K~V each), FP32 bulk",
    "fig1_cauchy": "factor-build points/s over the time-vs-n sweep (Cauchy l=1, tol 1e-3, d 3-6, n 1e4-1e7), "
                   "FP32 bulk",
    "fig3_rank5": "factor-build points/s over the error-vs-rank sweep (4 kernels x 10 tolerances, n=5000, d=5), "
                  "FP64 bulk",
    "krr8_clusters": "kernel ridge regression training points/s (k-means + HDF diagonal blocks + block-"
                     "preconditioned CG to rtol 1e-6 + test predictions), FP64 solve",
    "cross3_gauss": "cross factor-build points/s (build of K(X,Y) ~= U S V^T + 16-column K~V and K~^T W), "
                    "FP32 bulk",
}
FP32_LANES_PER_SM, NSM, SM_MAX_MHZ = 128, 152, 2070.0
# points of the oracle's bounded sample where its U (n x rank, FP64) grows fast with the rank
ORACLE_CAP = {"normal5_cauchy": 1500}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="mixture3_matern")
    ap.add_argument("--n", type=int, default=None, help="override n (same distribution)")
    ap.add_argument("--p-max", type=int, default=64)
    ap.add_argument("--no-fp64", action="store_true", help="skip the FP64 comparison")
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU oracle baseline")
    ap.add_argument("--no-solve", action="store_true", help="skip the solve measurement of the default workload")
    ap.add_argument("--nsets", type=int, default=None, help="batch512_gauss: number of sets (default 512)")
    ap.add_argument("--cpu-n", type=int, default=12000, help="oracle sample size")
    ap.add_argument("--oracle-once", action="store_true", help=argparse.SUPPRESS)
    return ap.parse_args()


def load_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            pk = json.load(fh)
        return pk, "measured"
    except Exception:
        return dict(PEAKS_FALLBACK), "fallback"


class ClockSampler:
    """nvidia-smi sampling of SM clocks and throttle reasons while the timed region runs."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.idx = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            f = [t.strip() for t in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax.append(float(f[2]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def max_over_ranks(ms, ws, dev):
    """The slowest rank's time (all-reduce MAX over the process group; the value itself for
    one process).  dev: the device the group's backend reduces on (cuda for NCCL, cpu for gloo)."""
    if ws <= 1:
        return float(ms)
    import torch
    t = torch.tensor([float(ms)], device=dev, dtype=torch.float64)
    torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank, ws, steps, ms_total):
    """Units processed by all ranks per second over the slowest rank's time (replicas: every
    rank processes the same units_per_rank each step)."""
    return ws * units_per_rank * steps / (ms_total / 1e3)


def blas_threads():
    """Threads of the BLAS that numpy loaded (threadpoolctl when present, else the OpenBLAS
    query function found in the process's mapped libraries); None if unknown."""
    try:
        from threadpoolctl import threadpool_info
        n = [i.get("num_threads") for i in threadpool_info() if i.get("user_api") == "blas"]
        if n:
            return int(n[0])
    except Exception:
        pass
    import ctypes
    import numpy  # noqa: F401  (loads the BLAS)
    try:
        with open("/proc/self/maps") as fh:
            libs = sorted({ln.split()[-1] for ln in fh if "openblas" in ln.lower() and ".so" in ln})
    except OSError:
        libs = []
    for path in libs:
        try:
            L = ctypes.CDLL(path)
        except OSError:
            continue
        for sym in ("scipy_openblas_get_num_threads64_", "openblas_get_num_threads64_", "openblas_get_num_threads"):
            fn = getattr(L, sym, None)
            if fn is not None:
                fn.restype = ctypes.c_int
                return int(fn())
    return None


SINGLE_THREAD_WORKLOADS = ("ball3_gauss", "mixture3_matern", "normal5_cauchy", "cube4_gauss", "batch512_gauss")
SINGLE_THREAD_ENV = {"OMP_NUM_THREADS": "1", "OPENBLAS_NUM_THREADS": "1", "MKL_NUM_THREADS": "1"}


def oracle_single_thread(args, workload):
    """The same oracle sample timed in a child process whose BLAS runs one thread (the paper's
    setting, Sec. 4: single-threaded).  Returns (seconds, points, blas threads) or None."""
    env = dict(os.environ)
    env.update(SINGLE_THREAD_ENV)
    cmd = [sys.executable, os.path.abspath(__file__), "--oracle-once", "--workload", workload,
           "--cpu-n", str(args.cpu_n), "--p-max", str(args.p_max)]
    try:
        out = subprocess.run(cmd, env=env, capture_output=True, text=True, timeout=600)
        for ln in out.stdout.splitlines()[::-1]:
            if ln.startswith("{"):
                r = json.loads(ln)
                return r["seconds"], r["points"], r["blas_threads"]
    except Exception:
        pass
    return None


def oracle_once(args):
    """Child side of oracle_single_thread: one untimed and one timed oracle step of the sample."""
    import numpy as np
    from paper_2202_03655_gb300 import workloads as W
    w = workload_params(args)
    if args.workload in ("mixture3_matern", "normal5_cauchy"):
        ns = min(args.cpu_n, w["n"], ORACLE_CAP.get(args.workload, w["n"]))
        x = W.points(args.workload, n=ns)
        V = np.random.default_rng(1).standard_normal((ns, w["ncols"]))
        cpu_oracle_step(x, w, V, args.p_max)
        sec = cpu_oracle_step(x, w, V, args.p_max)
    else:
        x, off, ells = oracle_sample(args, w)
        ns = int(off[-1])
        cpu_oracle_work(args, w, x, off, ells)
        sec = cpu_oracle_work(args, w, x, off, ells)
    print(json.dumps({"seconds": sec, "points": ns, "blas_threads": blas_threads()}), flush=True)
    return 0


def cpu_baseline_line(value, sample, args, workload, cores=None):
    """cpu_baseline object: the all-cores figure (value), the BLAS thread count it used, and the
    single-threaded figure of the same sample."""
    bt = blas_threads()
    out = {"value": value, "unit": "points/s", "cores": cores or bt or os.cpu_count(), "kind": "oracle",
           "sample": sample, "host_cpus": os.cpu_count(), "blas_threads": bt}
    one = oracle_single_thread(args, workload) if workload in SINGLE_THREAD_WORKLOADS else None
    if one:
        sec, pts, bt1 = one
        out["single_thread"] = {"value": pts / sec, "unit": "points/s", "cores": 1, "blas_threads": bt1}
    return out


def workload_params(args):
    from paper_2202_03655_gb300 import workloads as W
    w = dict(W.WORKLOADS[args.workload])
    if args.n:
        w["n"] = args.n
    return w


def exact_rows_matvec(x, kname, ell, v, rows):
    """(K v)[rows] for the exact kernel with plain torch FP64 ops (an accuracy check only)."""
    import numpy as np
    import torch
    out = []
    for s in range(0, len(rows), 128):
        r = torch.from_numpy(np.asarray(rows[s:s + 128])).to(x.device)
        z = torch.cdist(x[r], x) / ell
        if kname == "gaussian":
            K = torch.exp(-0.5 * z * z)
        elif kname == "cauchy":
            K = 1.0 / (1.0 + z * z)
        elif kname == "matern32":
            K = (1 + 3 ** 0.5 * z) * torch.exp(-(3 ** 0.5) * z)
        else:
            K = (1 + 5 ** 0.5 * z + 5.0 / 3.0 * z * z) * torch.exp(-(5 ** 0.5) * z)
        out.append((K @ v).cpu().numpy())
        del K, z
    return np.concatenate(out)


def cpu_oracle_step(x, w, V, p_max):
    """One oracle step (build + K~ V) on the host; returns seconds."""
    from oracle import hdf as ohdf
    t = time.perf_counter()
    fo = ohdf.build(x, w["kernel"], w["ell"], w["tol"], p_max=p_max)
    ohdf.matvec(fo, V)
    return time.perf_counter() - t


def oracle_sample(args, w):
    """(x, offsets, lengthscales) of the bounded CPU sample of a workload."""
    import numpy as np
    from paper_2202_03655_gb300 import workloads as W
    if args.workload == "batch512_gauss":
        xb, off, ells = W.batch_sets(W.rng(w["idx"]), nsets=w["nsets"], d=w["d"])
        k = 1
        while k < len(ells) and off[k] < args.cpu_n:
            k += 1
        return xb[:off[k]], off[:k + 1], ells[:k]
    ns = min(args.cpu_n if args.workload != "cube4_gauss" else min(args.cpu_n, 2000), w["n"])
    return W.points(args.workload, n=ns), np.array([0, ns]), np.array([w["ell"]])


def cpu_oracle_work(args, w, x, off, ells):
    """The oracle's form of one step on the sample; returns seconds."""
    import numpy as np
    from oracle import hdf as ohdf
    t = time.perf_counter()
    for s in range(len(ells)):
        xs = x[off[s]:off[s + 1]]
        g = np.random.default_rng(1)
        fo = ohdf.build(xs, w["kernel"], float(ells[s]), w["tol"], p_max=args.p_max)
        if args.workload == "cube4_gauss":
            v, wv = g.standard_normal(len(xs)), g.standard_normal(len(xs))
            ohdf.adjoint_fd(fo, xs, v, wv)
        else:
            ohdf.matvec(fo, g.standard_normal((len(xs), w["ncols"])))
    return time.perf_counter() - t


def cross_oracle_sample(args, w):
    """Bounded CPU sample of the cross workload: the first 4/5 of cpu_n points of X and 1/5 of Y."""
    from paper_2202_03655_gb300 import workloads as W
    mx, ny = max(1, (4 * args.cpu_n) // 5), max(1, args.cpu_n // 5)
    x, y = W.cross_sets(args.workload)
    return x[:mx], y[:ny]


def cross_oracle_work(w, x, y, p_max):
    """The oracle's form of one cross step on the sample; returns seconds."""
    import numpy as np
    from oracle import cross as ocross
    g = np.random.default_rng(1)
    t = time.perf_counter()
    fo = ocross.build_xy(x, y, w["kernel"], w["ell"], w["tol"], p_max=p_max)
    ocross.matvec_xy(fo, g.standard_normal((len(y), w["ncols"])))
    ocross.matvec_xy_t(fo, g.standard_normal((len(x), w["ncols"])))
    return time.perf_counter() - t


def run_reference(args):
    """The CPU oracle as the reference arm: bounded samples of the workload, steps timed."""
    ws, rank, _ = dist()
    if rank != 0:
        return 0
    import numpy as np
    from paper_2202_03655_gb300 import workloads as W
    w = workload_params(args)
    if args.workload == "krr8_clusters":
        from oracle import krr as okrr
        xs, ys, xq, _, init_s = W.krr_data(args.workload, n=min(args.cpu_n, 3000))

        def work():
            t = time.perf_counter()
            lab, _, _ = okrr.kmeans(xs, init_s)
            wo, _, _, _ = okrr.krr_fit(xs, ys, lab, w["kernel"], w["ell"], w["lam"], w["tol"], rtol=1e-6)
            okrr.kernel_matvec(xq, xs, w["kernel"], w["ell"], wo)
            return time.perf_counter() - t

        for _ in range(args.warmup):
            work()
        ts = [work() for _ in range(args.steps)]
        tot = sum(ts)
        val = len(xs) * args.steps / tot
        line = {"impl": "reference", "metric": METRICS[args.workload], "value": val, "unit": "points/s",
                "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
                "ms_per_step": 1e3 * tot / args.steps, "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                "config": {"workload": args.workload, "n_train_sample": len(xs), "d": w["d"], "p_max": args.p_max},
                "cpu_baseline": {"value": val, "unit": "points/s", "cores": blas_threads() or os.cpu_count(), "kind": "oracle",
                                 "sample": f"the regression recipe at {len(xs)} training points, FP64 numpy"},
                "e2e": {"value": val, "unit": "points/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(line), flush=True)
        return 0
    if args.workload in ("fig1_cauchy", "fig3_rank5"):
        from oracle import hdf as ohdf
        if args.workload == "fig1_cauchy":
            ns = min(args.cpu_n, 20000)
            jobs = [(W.maxnorm1_points(args.workload, ns, d), w["kernel"], w["ell"], w["tol"]) for d in (3, 4)]
            what = f"oracle builds of {ns} points in d = 3 and 4, Cauchy l = 1, tol 1e-3"
        else:
            ns = min(args.cpu_n, 2000)
            xs = W.maxnorm1_points(args.workload, w["n"], w["d"])[:ns]
            jobs = [(xs, kn, ell, 1e-3) for kn, ell in w["kernels"]]
            what = f"oracle builds of the first {ns} points, the four kernels at tol 1e-3"

        def work():
            t = time.perf_counter()
            for xj, kn, ell, tol in jobs:
                ohdf.build(xj, kn, ell, tol, p_max=args.p_max)
            return time.perf_counter() - t

        for _ in range(args.warmup):
            work()
        ts = [work() for _ in range(args.steps)]
        tot = sum(ts)
        npts = sum(len(j[0]) for j in jobs)
        val = npts * args.steps / tot
        line = {"impl": "reference", "metric": METRICS[args.workload], "value": val, "unit": "points/s",
                "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
                "ms_per_step": 1e3 * tot / args.steps, "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                "config": {"workload": args.workload, "points_per_step": npts, "p_max": args.p_max},
                "cpu_baseline": {"value": val, "unit": "points/s", "cores": blas_threads() or os.cpu_count(), "kind": "oracle",
                                 "sample": what + ", FP64 numpy"},
                "e2e": {"value": val, "unit": "points/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(line), flush=True)
        return 0
    if args.workload == "cross3_gauss":
        x, y = cross_oracle_sample(args, w)
        for _ in range(args.warmup):
            cross_oracle_work(w, x, y, args.p_max)
        ts = [cross_oracle_work(w, x, y, args.p_max) for _ in range(args.steps)]
        tot = sum(ts)
        ns = len(x) + len(y)
        val = ns * args.steps / tot
        line = {"impl": "reference", "metric": METRICS[args.workload], "value": val, "unit": "points/s",
                "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
                "ms_per_step": 1e3 * tot / args.steps, "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                "config": {"workload": args.workload, "m": w.get("n"), "n": w.get("n_y"), "m_sample": len(x),
                           "n_sample": len(y), "d": w["d"],
                           "kernel": w["kernel"], "lengthscale": w["ell"], "tol": w["tol"], "ncols": w["ncols"],
                           "p_max": args.p_max},
                "cpu_baseline": {"value": val, "unit": "points/s", "cores": blas_threads() or os.cpu_count(), "kind": "oracle",
                                 "sample": f"first {len(x)} points of X and {len(y)} of Y, build_xy + K~V + "
                                           f"K~^T W ({w['ncols']} columns), FP64 numpy"},
                "e2e": {"value": val, "unit": "points/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(line), flush=True)
        return 0
    if args.workload in ("cube4_gauss", "batch512_gauss"):
        x, off, ells = oracle_sample(args, w)
        for _ in range(args.warmup):
            cpu_oracle_work(args, w, x, off, ells)
        ts = [cpu_oracle_work(args, w, x, off, ells) for _ in range(args.steps)]
        tot = sum(ts)
        ns = int(off[-1])
        val = ns * args.steps / tot
        what = ("build + frozen-structure adjoint by central differences (oracle.hdf.adjoint_fd)"
                if args.workload == "cube4_gauss" else f"build + K~V ({w['ncols']} columns) of each set")
        line = {"impl": "reference", "metric": METRICS[args.workload], "value": val, "unit": "points/s",
                "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
                "ms_per_step": 1e3 * tot / args.steps, "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                "config": {"workload": args.workload, "n": w.get("n"), "n_sample": ns, "sets": len(ells), "d": w["d"],
                           "kernel": w["kernel"], "tol": w["tol"], "ncols": w["ncols"], "p_max": args.p_max},
                "cpu_baseline": {"value": val, "unit": "points/s", "cores": blas_threads() or os.cpu_count(), "kind": "oracle",
                                 "sample": f"{ns} points ({len(ells)} set(s)) of the workload, {what}"},
                "e2e": {"value": val, "unit": "points/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(line), flush=True)
        return 0
    ns = min(args.cpu_n, w["n"], ORACLE_CAP.get(args.workload, w["n"]))
    x = W.points(args.workload, n=ns)
    V = np.random.default_rng(1).standard_normal((ns, w["ncols"]))
    for _ in range(args.warmup):
        cpu_oracle_step(x, w, V, args.p_max)
    ts = [cpu_oracle_step(x, w, V, args.p_max) for _ in range(args.steps)]
    tot = sum(ts)
    val = ns * args.steps / tot
    cores = blas_threads() or os.cpu_count()
    line = {"impl": "reference", "metric": METRICS[args.workload], "value": val,
            "unit": "points/s", "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * tot / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": args.workload, "n": w["n"], "n_sample": ns, "d": w["d"], "kernel": w["kernel"],
                       "lengthscale": w["ell"], "tol": w["tol"], "ncols": w["ncols"], "p_max": args.p_max},
            "cpu_baseline": cpu_baseline_line(val, f"first {ns} of the {w['n']} points of the workload, full step "
                                                   f"(build + K~V, {w['ncols']} columns), FP64 numpy",
                                              args, args.workload, cores),
            "e2e": {"value": val, "unit": "points/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def _setup(args):
    import torch
    ws, rank, local = dist()
    if ws > 1:
        import torch.distributed as tdist
        torch.cuda.set_device(local)
        tdist.init_process_group("nccl")
    dev = torch.device("cuda", local if ws > 1 else 0)
    torch.cuda.set_device(dev)
    return ws, rank, dev


def _timed(args, ws, rank, dev, stream, one_step):
    """W warm-up steps, then K steps between CUDA events with clocks sampled; max over ranks."""
    import torch
    from paper_2202_03655_gb300 import hdf
    for _ in range(max(args.warmup, 0)):
        one_step(False)
    torch.cuda.synchronize()
    sampler = ClockSampler(dev.index) if rank == 0 else None
    if ws > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    if sampler:
        sampler.start()
    l0 = hdf.launch_count()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    recs = []
    e0.record(stream)
    for _ in range(args.steps):
        recs.append(one_step(True))
    e1.record(stream)
    torch.cuda.synchronize()
    if ws > 1:
        torch.distributed.barrier()
    launches = hdf.launch_count() - l0
    clocks = sampler.stop() if sampler else None
    ms_total = max_over_ranks(e0.elapsed_time(e1), ws, dev)
    return ms_total, recs, launches, clocks


def _timed_flushed(args, ws, rank, dev, stream, one_step):
    """As _timed, for inputs smaller than L2: before each step L2 is flushed by a 256 MiB write
    outside the step's events, each step is timed by its own event pair, and the total is their
    sum (max over ranks)."""
    import torch
    from paper_2202_03655_gb300 import hdf
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    for _ in range(max(args.warmup, 0)):
        one_step(False)
    torch.cuda.synchronize()
    sampler = ClockSampler(dev.index) if rank == 0 else None
    if ws > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    if sampler:
        sampler.start()
    l0 = hdf.launch_count()
    recs, pairs = [], []
    for _ in range(args.steps):
        flush.fill_(1)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        recs.append(one_step(True))
        e1.record(stream)
        pairs.append((e0, e1))
    torch.cuda.synchronize()
    if ws > 1:
        torch.distributed.barrier()
    launches = hdf.launch_count() - l0
    clocks = sampler.stop() if sampler else None
    ms_total = max_over_ranks(sum(a.elapsed_time(b) for a, b in pairs), ws, dev)
    return ms_total, recs, launches, clocks


def bench_plain(args):
    """The plain FP64 method on the small configuration (ball3_gauss: 2,000 points uniform in the
    unit ball, Gaussian l = 0.5, tol 1e-6): a step is hdf_build + K~ v (one column) with FP64 bulk;
    the FP32-bulk form of the same step is timed beside it, and both results are checked against
    the dense 2,000 x 2,000 kernel matrix."""
    import numpy as np
    import torch
    from paper_2202_03655_gb300 import hdf, workloads as W
    ws, rank, dev = _setup(args)
    w = workload_params(args)
    n, d = w["n"], w["d"]
    x_np = W.points(args.workload, n=n)
    v_np = W.rng(w["idx"] + 100).standard_normal(n)
    x = torch.from_numpy(x_np).to(dev)
    vs = {"fp64": torch.from_numpy(v_np).to(dev), "fp32": torch.from_numpy(v_np).float().to(dev)}
    ys = {k: torch.empty_like(v) for k, v in vs.items()}
    stream = torch.cuda.current_stream(dev)

    def stepper(prec):
        def one(keep):
            f = hdf.build(x, w["kernel"], w["ell"], w["tol"], precision=prec, p_max=args.p_max, stream=stream)
            f.matvec_ptr(vs[prec].data_ptr(), n, 1, ys[prec].data_ptr(), n, stream=stream)
            rec = None
            if keep:
                torch.cuda.current_stream(dev).synchronize()
                rec = (f.info, f.matvec_timings())
            f.free()
            return rec
        return one

    ms_total, recs, launches, clocks = _timed_flushed(args, ws, rank, dev, stream, stepper("fp64"))
    ms32, recs32, _, _ = _timed_flushed(args, ws, rank, dev, stream, stepper("fp32"))
    value = whole_job_rate(n, ws, args.steps, ms_total)
    # accuracy against the dense kernel matrix (outside the timed regions)
    z = torch.cdist(x, x) / w["ell"]
    Kv = torch.exp(-0.5 * z * z) @ vs["fp64"]
    del z
    err = {k: float(torch.linalg.norm(ys[k].double() - Kv) / torch.linalg.norm(Kv)) for k in ys}
    info, info32 = recs[-1][0], recs32[-1][0]
    r, ldu = info.rank, info.ldu
    nF = sum(info.s_k[k] for k in range(info.L + 1))
    mv = np.mean([q[1] for q in recs], axis=0)
    uw_ms = float(np.mean([q[0].t_ms[5] for q in recs]))
    peaks, peak_src = load_peaks()
    hbm = float(peaks.get("hbm_gbs", PEAKS_FALLBACK["hbm_gbs"]))
    kernels = {"k_uwriter": (uw_ms, n * (r * 8 + d * 8 + nF * 8)),
               "k_utv_tile": (float(mv[0]), n * r * 8 + n * 8),
               "k_uw_tile": (float(mv[2]), n * r * 8 + n * 8)}
    dom = max(kernels, key=lambda k: kernels[k][0])
    t_dom, b_dom = kernels[dom]
    roof = {"kernel": dom, "bound": "hbm", "achieved": b_dom / (t_dom / 1e3) / 1e9, "peak": hbm, "unit": "GB/s",
            "peak_source": peak_src + " copy bandwidth (burst)", "traffic": None,
            "algorithmic_bytes": b_dom, "ms_per_launch": t_dom,
            "note": "2,000 points: every launch is latency-bound; the fraction is reported, not a target"}
    roof["frac"] = roof["achieved"] / roof["peak"]
    # end to end from pinned host buffers: H2D of x and v, FP64 build + K~ v, D2H of y
    xh, vh = torch.from_numpy(x_np).pin_memory(), torch.from_numpy(v_np).pin_memory()
    yh = torch.empty_like(vh).pin_memory()
    xd = torch.empty_like(x)
    b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    k2 = max(1, min(args.steps, 5))

    def e2e_step():
        xd.copy_(xh, non_blocking=True)
        vs["fp64"].copy_(vh, non_blocking=True)
        f = hdf.build(xd, w["kernel"], w["ell"], w["tol"], precision="fp64", p_max=args.p_max, stream=stream)
        f.matvec_ptr(vs["fp64"].data_ptr(), n, 1, ys["fp64"].data_ptr(), n, stream=stream)
        yh.copy_(ys["fp64"], non_blocking=True)
        f.free()

    e2e_step()
    torch.cuda.synchronize()
    b0.record(stream)
    for _ in range(k2):
        e2e_step()
    b1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = b0.elapsed_time(b1) / k2
    e2e = {"value": ws * n / (e2e_ms / 1e3), "unit": "points/s", "h2d_bytes_per_step": n * d * 8 + n * 8,
           "d2h_bytes_per_step": n * 8, "ms_per_step": e2e_ms}
    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu:
        V = np.random.default_rng(1).standard_normal((n, 1))
        cpu_oracle_step(x_np, w, V, args.p_max)
        ts = cpu_oracle_step(x_np, w, V, args.p_max)
        cpu = cpu_baseline_line(n / ts, f"all {n} points, one full step (build + K~v), FP64 numpy", args,
                                args.workload)
    if rank == 0:
        line = {"metric": METRICS[args.workload], "value": value, "unit": "points/s", "n_gpus": ws,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_total / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
                "data": "synthetic",
                "config": {"workload": args.workload, "n": n, "d": d, "kernel": w["kernel"], "lengthscale": w["ell"],
                           "tol": w["tol"], "ncols": 1, "p_max": args.p_max, "p": info.p, "rank": r, "ldu": ldu,
                           "parallelism": f"replicas{ws}", "l2": "L2 flushed (256 MiB write) before each step"},
                "e2e": e2e, "roofline": roof, "cpu_baseline": cpu, "clocks": clocks, "gpu_launches": launches,
                "detail": {"rel_err_vs_dense": err["fp64"], "err_bound": info.err_bound,
                           "build_ms": float(np.mean([q[0].t_ms[7] for q in recs])),
                           "build_phase_ms": [float(t) for t in info.t_ms],
                           "kernel_ms": {k: v[0] for k, v in kernels.items()},
                           "fp32": {"ms_per_step": ms32 / args.steps, "points_per_s": whole_job_rate(n, ws, args.steps, ms32),
                                    "rank": info32.rank, "rel_err_vs_dense": err["fp32"],
                                    "build_ms": float(np.mean([q[0].t_ms[7] for q in recs32]))}}}
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def _cpu_baseline(args, w):
    x, off, ells = oracle_sample(args, w)
    ts = cpu_oracle_work(args, w, x, off, ells)
    ns = int(off[-1])
    what = ("build + frozen-structure adjoint by central differences" if args.workload == "cube4_gauss"
            else f"build + K~V ({w['ncols']} columns) of each set")
    return cpu_baseline_line(ns / ts, f"{ns} points ({len(ells)} set(s)) of the workload, {what}, FP64 numpy",
                             args, args.workload)


def bench_adjoint(args):
    """Differentiation row: build + adjoint (gradient of w^T K~ v w.r.t. the points and l)."""
    import numpy as np
    import torch
    from paper_2202_03655_gb300 import hdf, workloads as W
    ws, rank, dev = _setup(args)
    w = workload_params(args)
    n, d = w["n"], w["d"]
    x_np = W.points(args.workload, n=n)
    g = W.rng(w["idx"] + 100)
    v_np = g.standard_normal(n).astype(np.float32)
    w_np = g.standard_normal(n).astype(np.float32)
    x = torch.from_numpy(x_np).to(dev)
    v, wv = torch.from_numpy(v_np).to(dev), torch.from_numpy(w_np).to(dev)
    stream = torch.cuda.current_stream(dev)
    a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def one(keep):
        f = hdf.build(x, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
        a0.record(stream)
        G, dl, val = f.adjoint(x, v, wv, stream=stream)
        a1.record(stream)
        a1.synchronize()
        rec = (f.info, a0.elapsed_time(a1), val) if keep else None
        f.free()
        return rec

    ms_total, recs, launches, clocks = _timed(args, ws, rank, dev, stream, one)
    info = recs[-1][0]
    adj_ms = float(np.mean([r[1] for r in recs]))
    value = whole_job_rate(n, ws, args.steps, ms_total)
    # accuracy outside the timed region: sampled rows of K~ v against the exact kernel
    f = hdf.build(x, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
    y = f.matvec(v)
    # the solve on this factor (A6 Gram U^T U on the tensor cores + host LU of the core, A8
    # Woodbury apply with one refinement step); the second solve reuses the factored core.
    # lambda grows with n as in kernel ridge regression, so that the condition number of
    # lambda I + K~ (largest eigenvalue ~ n times the mean kernel value) stays within what an
    # FP32 factor resolves; the work timed does not depend on lambda
    lam = 1e-4 * n
    s0 = time.perf_counter()
    xs = f.solve(lam, v, refine_steps=1)
    torch.cuda.synchronize()
    solve_first_ms = 1e3 * (time.perf_counter() - s0)
    s0 = time.perf_counter()
    xs = f.solve(lam, v, refine_steps=1)
    torch.cuda.synchronize()
    solve_again_ms = 1e3 * (time.perf_counter() - s0)
    gram_ms = float(f.info.t_ms[6])
    res = lam * xs + f.matvec(xs) - v
    solve_res = float(torch.linalg.norm(res.double()) / torch.linalg.norm(v.double()))
    ldu_s = f.info.ldu
    gram_flops = 3 * 2.0 * n * ldu_s * ldu_s        # three TF32 products per multiply-add
    pk, _ = load_peaks()
    tf32_peak = float(pk.get("bf16_tflops", PEAKS_FALLBACK["bf16_tflops"])) * 1.1 / 2.25
    rows = np.sort(W.rng(7).choice(n, 512, replace=False))
    exact = exact_rows_matvec(x, w["kernel"], w["ell"], v.double(), rows)
    approx = y[torch.from_numpy(rows).to(dev)].double().cpu().numpy()
    rel_err = float(np.linalg.norm(approx - exact) / np.linalg.norm(exact))
    f.free()
    # roofline of the adjoint: per point the contraction (w_i a + v_i b) . dU_i/dx_i over the r
    # columns and d + 1 derivative directions, 2 r (d + 1) FP32 flops, against the FP32 FMA peak
    r = info.rank
    flops = 2.0 * n * r * (d + 1)
    peak_alu = NSM * FP32_LANES_PER_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12
    roof = {"kernel": "k_adjoint (with its U^T v, U^T w)", "bound": "alu",
            "achieved": flops / (adj_ms / 1e3) / 1e12, "peak": peak_alu, "unit": "TFLOP/s",
            "peak_source": "FP32 FMA: 152 SMs x 128 lanes x 2 x 2070 MHz (no measured FP32 peak)",
            "traffic": None, "algorithmic_flops": flops, "ms_per_launch": adj_ms}
    roof["frac"] = roof["achieved"] / roof["peak"]
    # end to end from pinned host buffers: H2D x, v, w; build; adjoint; D2H of the gradient
    xh = torch.from_numpy(x_np).pin_memory()
    vh, wh = torch.from_numpy(v_np).pin_memory(), torch.from_numpy(w_np).pin_memory()
    Gh = torch.empty((n, d), dtype=torch.float32).pin_memory()
    xd, vd, wd = torch.empty_like(x), torch.empty_like(v), torch.empty_like(wv)
    torch.cuda.synchronize()
    b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    k2 = max(1, min(args.steps, 3))

    def e2e_step():
        xd.copy_(xh, non_blocking=True); vd.copy_(vh, non_blocking=True); wd.copy_(wh, non_blocking=True)
        f = hdf.build(xd, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
        G, dl, val = f.adjoint(xd, vd, wd, stream=stream)
        Gh.copy_(G, non_blocking=True)
        f.free()

    e2e_step()              # one untimed step
    torch.cuda.synchronize()
    b0.record(stream)
    for _ in range(k2):
        e2e_step()
    b1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = b0.elapsed_time(b1) / k2
    e2e = {"value": ws * n / (e2e_ms / 1e3), "unit": "points/s", "h2d_bytes_per_step": n * d * 8 + 2 * n * 4,
           "d2h_bytes_per_step": n * d * 4 + 16, "ms_per_step": e2e_ms}
    cpu = _cpu_baseline(args, w) if (rank == 0 and ws == 1 and not args.no_cpu) else None
    if rank == 0:
        line = {"metric": METRICS[args.workload], "value": value, "unit": "points/s", "n_gpus": ws,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_total / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
                "data": "synthetic",
                "config": {"workload": args.workload, "n": n, "d": d, "kernel": w["kernel"], "lengthscale": w["ell"],
                           "tol": w["tol"], "p_max": args.p_max, "p": info.p, "rank": r, "ldu": info.ldu,
                           "parallelism": f"replicas{ws}", "l2": f"inputs larger than L2 (U is {n * info.ldu * 4 / 1e9:.1f} GB)"},
                "e2e": e2e, "roofline": roof, "cpu_baseline": cpu, "clocks": clocks, "gpu_launches": launches,
                "detail": {"adjoint_ms": adj_ms, "build_ms": float(info.t_ms[7]),
                           "solve": {"lambda": lam, "first_ms": solve_first_ms, "again_ms": solve_again_ms,
                                     "gram_ms": gram_ms, "residual": solve_res,
                                     "gram_tensor_tflops": gram_flops / (gram_ms / 1e3) / 1e12 if gram_ms > 0 else None,
                                     "gram_tensor_frac_of_tf32": (gram_flops / (gram_ms / 1e3) / 1e12 / tf32_peak)
                                     if gram_ms > 0 else None,
                                     "tf32_peak_source": "measured bf16 cuBLAS burst x 1.1/2.25 (nominal TF32/BF16)"},
                           "rel_err_sampled_vs_exact": rel_err, "err_bound": info.err_bound,
                           "value_f": recs[-1][2]}}
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def bench_mfree(args):
    """Large-rank row: hdf_build (matrix-free rows, chosen by the build) + K~V with 16 columns."""
    import numpy as np
    import torch
    from paper_2202_03655_gb300 import hdf, workloads as W
    ws, rank, dev = _setup(args)
    w = workload_params(args)
    n, d, c = w["n"], w["d"], w["ncols"]
    x_np = W.points(args.workload, n=n)
    V_np = np.asfortranarray(W.rng(w["idx"] + 100).standard_normal((n, c)).astype(np.float32))
    x = torch.from_numpy(x_np).to(dev)
    Vc = torch.from_numpy(np.ascontiguousarray(V_np.T)).to(dev)
    Yc = torch.empty_like(Vc)
    stream = torch.cuda.current_stream(dev)

    # the matrix-free form is what the build picks at the full size (U would not fit); the flag
    # keeps it at reduced --n too
    mf = hdf.FLAG_MATRIX_FREE

    def one(keep):
        f = hdf.build(x, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream, flags=mf)
        f.matvec_ptr(Vc.data_ptr(), n, c, Yc.data_ptr(), n, stream=stream)
        rec = (f.info, f.matvec_timings()) if keep else None
        f.free()
        return rec

    ms_total, recs, launches, clocks = _timed(args, ws, rank, dev, stream, one)
    info = recs[-1][0]
    mv = np.array([r[1] for r in recs]).mean(axis=0)          # U^T V, reduce, U W (ms)
    value = whole_job_rate(n, ws, args.steps, ms_total)
    # accuracy outside the timed region: sampled rows of K~ V against the exact kernel
    f = hdf.build(x, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream, flags=mf)
    f.matvec_ptr(Vc.data_ptr(), n, c, Yc.data_ptr(), n, stream=stream)
    rows = np.sort(W.rng(7).choice(n, 256, replace=False))
    exact = exact_rows_matvec(x, w["kernel"], w["ell"], Vc.t().double(), rows)
    approx = Yc.t()[torch.from_numpy(rows).to(dev)].double().cpu().numpy()
    rel_err = float(np.linalg.norm(approx - exact) / np.linalg.norm(exact))
    f.free()
    # roofline: the two products are tensor-core GEMMs over the stored Z rows (tcgen05, 3xTF32:
    # three TF32 products per multiply-add for FP32 accuracy); the algorithmic work is that of
    # K~V on the factor, 2 n r c flops per product, i.e. 3 x 2 n r c TF32 flops, against the TF32
    # rate (measured BF16 cuBLAS burst x 1.1 / 2.25, the nominal TF32 / BF16 ratio)
    r = info.rank
    flops = 2.0 * n * r * c
    pk, pk_src = load_peaks()
    tf32_peak = float(pk.get("bf16_tflops", PEAKS_FALLBACK["bf16_tflops"])) * 1.1 / 2.25
    kern = {"k_tc_mf_utv": float(mv[0]), "k_tc_mf_uw": float(mv[2])}
    dom = max(kern, key=kern.get)
    roof = {"kernel": dom, "bound": "tensor", "achieved": 3 * flops / (kern[dom] / 1e3) / 1e12, "peak": tf32_peak,
            "unit": "TFLOP/s", "peak_source": f"{pk_src} bf16 cuBLAS burst x 1.1/2.25 (nominal TF32/BF16 ratio)",
            "traffic": None, "algorithmic_flops": 3 * flops, "useful_fp32_tflops": flops / (kern[dom] / 1e3) / 1e12,
            "ms_per_launch": kern[dom]}
    roof["frac"] = roof["achieved"] / roof["peak"]
    # end to end from pinned host buffers: H2D x and V; build; K~V; D2H of Y
    xh = torch.from_numpy(x_np).pin_memory()
    Vh = torch.from_numpy(np.ascontiguousarray(V_np.T)).pin_memory()
    Yh = torch.empty_like(Vh).pin_memory()
    xd = torch.empty_like(x)
    torch.cuda.synchronize()
    b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    k2 = max(1, min(args.steps, 2))

    def e2e_step():
        xd.copy_(xh, non_blocking=True)
        Vc.copy_(Vh, non_blocking=True)
        f = hdf.build(xd, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream,
                      flags=mf)
        f.matvec_ptr(Vc.data_ptr(), n, c, Yc.data_ptr(), n, stream=stream)
        Yh.copy_(Yc, non_blocking=True)
        f.free()

    e2e_step()
    torch.cuda.synchronize()
    b0.record(stream)
    for _ in range(k2):
        e2e_step()
    b1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = b0.elapsed_time(b1) / k2
    e2e = {"value": ws * n / (e2e_ms / 1e3), "unit": "points/s", "h2d_bytes_per_step": n * d * 8 + n * c * 4,
           "d2h_bytes_per_step": n * c * 4, "ms_per_step": e2e_ms}
    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu:
        ns = min(args.cpu_n, n, ORACLE_CAP[args.workload])
        ts = cpu_oracle_step(x_np[:ns], w, V_np[:ns].astype(np.float64), args.p_max)
        cpu = cpu_baseline_line(ns / ts, f"first {ns} of the {n} points, one full step (build + K~V, {c} columns), "
                                         "FP64 numpy", args, args.workload)
    if rank == 0:
        line = {"metric": METRICS[args.workload], "value": value, "unit": "points/s", "n_gpus": ws,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_total / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
                "data": "synthetic",
                "config": {"workload": args.workload, "n": n, "d": d, "kernel": w["kernel"], "lengthscale": w["ell"],
                           "tol": w["tol"], "ncols": c, "p_max": args.p_max, "p": info.p, "reached": bool(info.reached),
                           "rank": r, "ldu": info.ldu, "matrix_free": bool(info.matrix_free),
                           "U_bytes_if_stored": n * info.ldu * 4, "stored_bytes": n * info.mf_row * 4,
                           "parallelism": f"replicas{ws}", "l2": "inputs larger than L2 (the stored rows are "
                           f"{n * info.mf_row * 4 / 1e9:.0f} GB)"},
                "e2e": e2e, "roofline": roof, "cpu_baseline": cpu, "clocks": clocks, "gpu_launches": launches,
                "detail": {"rel_err_sampled_vs_exact": rel_err, "err_bound": info.err_bound,
                           "cheb_tail": info.cheb_tail, "build_ms": float(info.t_ms[7]),
                           "build_phase_ms": [float(info.t_ms[q]) for q in range(8)],
                           "kv_ms": float(mv.sum()), "kernel_ms": {"k_tc_mf_utv": float(mv[0]),
                                                                    "k_reduce_scale": float(mv[1]),
                                                                    "k_tc_mf_uw": float(mv[2])},
                           "s_k": [int(info.s_k[k]) for k in range(info.L + 1)]}}
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def bench_batch(args):
    """Batching row: hdf_build_batched + hdf_batch_matvec over 512 ragged sets."""
    import numpy as np
    import torch
    from paper_2202_03655_gb300 import hdf, workloads as W
    ws, rank, dev = _setup(args)
    w = workload_params(args)
    c, d = w["ncols"], w["d"]
    xb, off, ells = W.batch_sets(W.rng(w["idx"]), nsets=args.nsets or w["nsets"], d=d)
    N = int(off[-1])
    x = torch.from_numpy(xb).to(dev)
    V_np = W.rng(w["idx"] + 100).standard_normal((c, N)).astype(np.float32)     # column-major N x c
    Vc = torch.from_numpy(V_np).to(dev)
    Yc = torch.empty_like(Vc)
    stream = torch.cuda.current_stream(dev)
    m0, m1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def one(keep):
        b = hdf.build_batched(x, off, w["kernel"], ells, w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
        m0.record(stream)
        b.matvec_ptr(Vc.data_ptr(), N, c, Yc.data_ptr(), N, stream=stream)
        m1.record(stream)
        rec = None
        if keep:
            m1.synchronize()
            infos = [b.info(s) for s in range(b.nsets)]
            rec = (b.timings(), m0.elapsed_time(m1), infos)
        b.free()
        return rec

    ms_total, recs, launches, clocks = _timed(args, ws, rank, dev, stream, one)
    value = whole_job_rate(N, ws, args.steps, ms_total)
    tms, mv_ms, infos = recs[-1]
    ranks = np.array([i.rank for i in infos])
    ldus = np.array([i.ldu for i in infos])
    sizes = np.diff(off)
    u_bytes = int(np.sum(sizes * ranks) * 4)
    # accuracy outside the timed region: 4 sets, 256 sampled rows each, against the exact kernel
    b = hdf.build_batched(x, off, w["kernel"], ells, w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
    b.matvec_ptr(Vc.data_ptr(), N, c, Yc.data_ptr(), N, stream=stream)
    torch.cuda.synchronize()
    errs = []
    for s in np.linspace(0, len(ells) - 1, 4).astype(int):
        a, e = int(off[s]), int(off[s + 1])
        rows = np.sort(W.rng(7 + s).choice(e - a, min(256, e - a), replace=False))
        exact = exact_rows_matvec(x[a:e], w["kernel"], float(ells[s]), Vc[0, a:e].double(), rows)
        approx = Yc[0, a:e][torch.from_numpy(rows).to(dev)].double().cpu().numpy()
        errs.append(float(np.linalg.norm(approx - exact) / np.linalg.norm(exact)))
    b.free()
    # roofline: the persistent build kernel writes every set's U (HBM write bound)
    peaks, peak_src = load_peaks()
    hbm = float(peaks.get("hbm_gbs", PEAKS_FALLBACK["hbm_gbs"]))
    build_kernel_ms = float(tms[5])
    roof = {"kernel": "batched build graph (k_batch_radial + k_batch_urows per size class)", "bound": "hbm",
            "achieved": u_bytes / (build_kernel_ms / 1e3) / 1e9, "peak": hbm, "unit": "GB/s",
            "peak_source": peak_src + " copy bandwidth (burst)", "traffic": None,
            "algorithmic_bytes": u_bytes, "ms_per_launch": build_kernel_ms}
    roof["frac"] = roof["achieved"] / roof["peak"]
    # end to end from pinned host buffers: H2D x and V, batched build + matvec, D2H Y
    xh = torch.from_numpy(xb).pin_memory()
    Vh = torch.from_numpy(V_np).pin_memory()
    Yh = torch.empty_like(Vh).pin_memory()
    xd = torch.empty_like(x)
    torch.cuda.synchronize()
    b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    k2 = max(1, min(args.steps, 3))

    def e2e_step():
        xd.copy_(xh, non_blocking=True); Vc.copy_(Vh, non_blocking=True)
        bb = hdf.build_batched(xd, off, w["kernel"], ells, w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
        bb.matvec_ptr(Vc.data_ptr(), N, c, Yc.data_ptr(), N, stream=stream)
        Yh.copy_(Yc, non_blocking=True)
        bb.free()

    e2e_step()              # one untimed step
    torch.cuda.synchronize()
    b0.record(stream)
    for _ in range(k2):
        e2e_step()
    b1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = b0.elapsed_time(b1) / k2
    e2e = {"value": ws * N / (e2e_ms / 1e3), "unit": "points/s", "h2d_bytes_per_step": N * d * 8 + N * c * 4,
           "d2h_bytes_per_step": N * c * 4, "ms_per_step": e2e_ms}
    cpu = _cpu_baseline(args, w) if (rank == 0 and ws == 1 and not args.no_cpu) else None
    if rank == 0:
        line = {"metric": METRICS[args.workload], "value": value, "unit": "points/s", "n_gpus": ws,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_total / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
                "data": "synthetic",
                "config": {"workload": args.workload, "sets": len(ells), "points": N, "d": d, "kernel": w["kernel"],
                           "tol": w["tol"], "ncols": c, "p_max": args.p_max, "U_bytes": int(np.sum(sizes * ldus) * 4),
                           "parallelism": f"replicas{ws}", "l2": "inputs larger than L2"},
                "e2e": e2e, "roofline": roof, "cpu_baseline": cpu, "clocks": clocks, "gpu_launches": launches,
                "detail": {"build_phase_ms": [float(t) for t in tms], "kv_ms": mv_ms,
                           "kv_gbs": (2 * u_bytes + N * c * 8) / (mv_ms / 1e3) / 1e9,
                           "rel_err_sampled_vs_exact": errs, "rank_total": int(ranks.sum()),
                           "p_range": [int(min(i.p for i in infos)), int(max(i.p for i in infos))]}}
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def bench_cross(args):
    """Non-symmetric row: hdf_build_cross + K~ V + K~^T W."""
    import numpy as np
    import torch
    from paper_2202_03655_gb300 import hdf, workloads as W
    ws, rank, dev = _setup(args)
    w = workload_params(args)
    c, d = w["ncols"], w["d"]
    x_np, y_np = W.cross_sets(args.workload)
    m, n = len(x_np), len(y_np)
    g = W.rng(w["idx"] + 100)
    V_np = g.standard_normal((c, n)).astype(np.float32)        # column-major n x c (over Y)
    W_np = g.standard_normal((c, m)).astype(np.float32)        # column-major m x c (over X)
    x, y = torch.from_numpy(x_np).to(dev), torch.from_numpy(y_np).to(dev)
    Vc, Wc = torch.from_numpy(V_np).to(dev), torch.from_numpy(W_np).to(dev)
    Yc = torch.empty((c, m), dtype=torch.float32, device=dev)
    Zc = torch.empty((c, n), dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)
    lib = hdf.lib()
    t0, t1, t2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))

    def products(f):
        hdf._check(lib.hdf_matvec(f._h, hdf._vp(Vc.data_ptr()), n, c, hdf._vp(Yc.data_ptr()), m,
                                  hdf._vp(stream.cuda_stream)))
        t1.record(stream)
        hdf._check(lib.hdf_matvec_transpose(f._h, hdf._vp(Wc.data_ptr()), m, c, hdf._vp(Zc.data_ptr()), n,
                                            hdf._vp(stream.cuda_stream)))

    def one(keep):
        f = hdf.build_cross(x, y, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max,
                            stream=stream)
        t0.record(stream)
        products(f)
        t2.record(stream)
        rec = None
        if keep:
            t2.synchronize()
            rec = (f.info, t0.elapsed_time(t1), t1.elapsed_time(t2), f.matvec_timings())
        f.free()
        return rec

    ms_total, recs, launches, clocks = _timed(args, ws, rank, dev, stream, one)
    value = whole_job_rate(m + n, ws, args.steps, ms_total)
    info = recs[-1][0]
    kv_ms = float(np.mean([r[1] for r in recs]))
    kvt_ms = float(np.mean([r[2] for r in recs]))
    mv = np.mean([r[3] for r in recs], axis=0)          # K~ V: U_Y^T V, reduce, U_X W
    uw_ms = float(np.mean([r[0].t_ms[5] for r in recs]))
    r, ldu = info.rank, info.ldu
    nF = sum(info.s_k[k] for k in range(info.L + 1))
    # accuracy outside the timed region: sampled rows of K~ V and K~^T W against the exact kernel
    f = hdf.build_cross(x, y, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
    products(f)
    torch.cuda.synchronize()
    f.free()
    rows = torch.from_numpy(np.sort(W.rng(7).choice(m, 256, replace=False))).to(dev)
    cols = torch.from_numpy(np.sort(W.rng(8).choice(n, 256, replace=False))).to(dev)
    ell = w["ell"]
    Kr = torch.exp(-0.5 * (torch.cdist(x[rows], y) / ell) ** 2)
    err_y = float(torch.linalg.norm(Yc[0, rows].double() - Kr @ Vc[0].double()) / torch.linalg.norm(Kr @ Vc[0].double()))
    del Kr
    Kc = torch.exp(-0.5 * (torch.cdist(y[cols], x) / ell) ** 2)
    err_z = float(torch.linalg.norm(Zc[0, cols].double() - Kc @ Wc[0].double()) / torch.linalg.norm(Kc @ Wc[0].double()))
    del Kc
    # roofline of the dominant kernel of the step
    peaks, peak_src = load_peaks()
    hbm = float(peaks.get("hbm_gbs", PEAKS_FALLBACK["hbm_gbs"]))
    kernels = {
        "k_uwriter (X and Y sides, two launches)": (uw_ms, (m + n) * (r * 4 + d * 8 + nF * 4)),
        "k_tc_utv (U_Y^T V)": (float(mv[0]), n * r * 4 + n * c * 4),
        "k_tc_uw (U_X W)": (float(mv[2]), m * r * 4 + m * c * 4),
    }
    dom = max(kernels, key=lambda k: kernels[k][0])
    t_dom, b_dom = kernels[dom]
    roof = {"kernel": dom, "bound": "hbm", "achieved": b_dom / (t_dom / 1e3) / 1e9, "peak": hbm, "unit": "GB/s",
            "peak_source": peak_src + " copy bandwidth (burst)", "traffic": None,
            "algorithmic_bytes": b_dom, "ms_per_launch": t_dom}
    roof["frac"] = roof["achieved"] / roof["peak"]
    # end to end from pinned host buffers: H2D of X, Y, V, W; build; both products; D2H of both
    xh, yh = torch.from_numpy(x_np).pin_memory(), torch.from_numpy(y_np).pin_memory()
    Vh, Wh = torch.from_numpy(V_np).pin_memory(), torch.from_numpy(W_np).pin_memory()
    Yh, Zh = torch.empty_like(Yc, device="cpu").pin_memory(), torch.empty_like(Zc, device="cpu").pin_memory()
    xd, yd = torch.empty_like(x), torch.empty_like(y)
    torch.cuda.synchronize()
    b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    k2 = max(1, min(args.steps, 3))

    def e2e_step():
        xd.copy_(xh, non_blocking=True); yd.copy_(yh, non_blocking=True)
        Vc.copy_(Vh, non_blocking=True); Wc.copy_(Wh, non_blocking=True)
        f = hdf.build_cross(xd, yd, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max,
                            stream=stream)
        products(f)
        Yh.copy_(Yc, non_blocking=True); Zh.copy_(Zc, non_blocking=True)
        f.free()

    e2e_step()              # one untimed step
    torch.cuda.synchronize()
    b0.record(stream)
    for _ in range(k2):
        e2e_step()
    b1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = b0.elapsed_time(b1) / k2
    e2e = {"value": ws * (m + n) / (e2e_ms / 1e3), "unit": "points/s",
           "h2d_bytes_per_step": (m + n) * d * 8 + (m + n) * c * 4, "d2h_bytes_per_step": (m + n) * c * 4,
           "ms_per_step": e2e_ms}
    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu:
        xs, ys = cross_oracle_sample(args, w)
        ts = cross_oracle_work(w, xs, ys, args.p_max)
        cpu = {"value": (len(xs) + len(ys)) / ts, "unit": "points/s", "cores": blas_threads() or os.cpu_count(), "kind": "oracle",
               "sample": f"first {len(xs)} points of X and {len(ys)} of Y, build_xy + K~V + K~^T W "
                         f"({c} columns), FP64 numpy"}
    if rank == 0:
        line = {"metric": METRICS[args.workload], "value": value, "unit": "points/s", "n_gpus": ws,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_total / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
                "data": "synthetic",
                "config": {"workload": args.workload, "m": m, "n": n, "d": d, "kernel": w["kernel"],
                           "lengthscale": w["ell"], "tol": w["tol"], "ncols": c, "p_max": args.p_max, "p": info.p,
                           "rank": r, "ldu": ldu, "U_bytes": (m + n) * ldu * 4, "parallelism": f"replicas{ws}",
                           "l2": "inputs larger than L2"},
                "e2e": e2e, "roofline": roof, "cpu_baseline": cpu, "clocks": clocks, "gpu_launches": launches,
                "detail": {"build_ms": float(np.mean([r_[0].t_ms[7] for r_ in recs])),
                           "build_phase_ms": [float(t) for t in info.t_ms], "kv_ms": kv_ms, "kvt_ms": kvt_ms,
                           "kernel_ms": {k: v[0] for k, v in kernels.items()},
                           "rel_err_sampled_vs_exact": {"K~V": err_y, "K~^T W": err_z},
                           "err_bound": info.err_bound}}
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def bench_fig1(args):
    """Time-vs-n row: hdf_build over the (d, n) grid of Fig. 1."""
    import numpy as np
    import torch
    from paper_2202_03655_gb300 import hdf, workloads as W
    ws, rank, dev = _setup(args)
    w = workload_params(args)
    stream = torch.cuda.current_stream(dev)
    sizes = [int(n) for n in w["sizes"] if not args.n or n <= args.n]
    grid = [(d, n) for d in w["dims"] for n in sizes]
    pts = {(d, n): torch.from_numpy(W.maxnorm1_points(args.workload, n, d)).to(dev) for d, n in grid}
    ev = {k: (torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for k in grid}
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)     # larger than the 129 MB L2

    def one(keep):
        flush.zero_()
        rec = {}
        for k in grid:
            e0, e1 = ev[k]
            e0.record(stream)
            f = hdf.build(pts[k], w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
            e1.record(stream)
            if keep:
                rec[k] = f.info
            f.free()
        if keep:
            torch.cuda.synchronize()
            rec = {k: (v, ev[k][0].elapsed_time(ev[k][1])) for k, v in rec.items()}
        return rec

    ms_total, recs, launches, clocks = _timed(args, ws, rank, dev, stream, one)
    total_pts = sum(n for _, n in grid)
    value = whole_job_rate(total_pts, ws, args.steps, ms_total)
    table = []
    for d in w["dims"]:
        ts = []
        for n in sizes:
            ms = float(np.median([r[(d, n)][1] for r in recs]))
            I = recs[-1][(d, n)][0]
            ts.append(ms)
            table.append({"d": d, "n": n, "build_ms": ms, "points_per_s": n / (ms / 1e3), "p": I.p,
                          "rank": I.rank, "reached": bool(I.reached), "err_bound": I.err_bound})
        big = [i for i, n in enumerate(sizes) if n >= 100_000]
        if len(big) >= 2:
            slope = float(np.polyfit(np.log([sizes[i] for i in big]), np.log([ts[i] for i in big]), 1)[0])
            table.append({"d": d, "loglog_slope_n_ge_1e5": slope})
    # roofline: the U writer of the largest d = 3 build
    dmax = (w["dims"][0], sizes[-1])
    I = recs[-1][dmax][0]
    n = dmax[1]
    nF = sum(I.s_k[k] for k in range(I.L + 1))
    ub = n * (I.rank * 4 + dmax[0] * 8 + nF * 4)
    peaks, peak_src = load_peaks()
    hbm = float(peaks.get("hbm_gbs", PEAKS_FALLBACK["hbm_gbs"]))
    t5 = float(np.mean([r[dmax][0].t_ms[5] for r in recs]))
    roof = {"kernel": f"k_uwriter (d = {dmax[0]}, n = {n})", "bound": "hbm", "achieved": ub / (t5 / 1e3) / 1e9,
            "peak": hbm, "unit": "GB/s", "peak_source": peak_src + " copy bandwidth (burst)", "traffic": None,
            "algorithmic_bytes": ub, "ms_per_launch": t5}
    roof["frac"] = roof["achieved"] / roof["peak"]
    # end to end: H2D of the points of the sweep, every build, D2H of each factor's metadata
    host = {k: v.cpu().pin_memory() for k, v in pts.items()}
    torch.cuda.synchronize()
    b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    b0.record(stream)
    for k in grid:
        pts[k].copy_(host[k], non_blocking=True)
        f = hdf.build(pts[k], w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
        f.free()
    b1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = b0.elapsed_time(b1)
    e2e = {"value": ws * total_pts / (e2e_ms / 1e3), "unit": "points/s",
           "h2d_bytes_per_step": int(sum(n * d * 8 for d, n in grid)), "d2h_bytes_per_step": 0, "ms_per_step": e2e_ms}
    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu:
        from oracle import hdf as ohdf
        xs = W.maxnorm1_points(args.workload, min(args.cpu_n, 20000), 3)
        t = time.perf_counter()
        ohdf.build(xs, w["kernel"], w["ell"], w["tol"], p_max=args.p_max)
        ts_ = time.perf_counter() - t
        cpu = {"value": len(xs) / ts_, "unit": "points/s", "cores": blas_threads() or os.cpu_count(), "kind": "oracle",
               "sample": f"one oracle build of {len(xs)} points, d = 3, FP64 numpy"}
    if rank == 0:
        line = {"metric": METRICS[args.workload], "value": value, "unit": "points/s", "n_gpus": ws,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_total / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
                "config": {"workload": args.workload, "dims": list(w["dims"]), "sizes": sizes, "kernel": w["kernel"],
                           "lengthscale": w["ell"], "tol": w["tol"], "p_max": args.p_max,
                           "parallelism": f"replicas{ws}",
                           "l2": "L2 flushed by a 256 MB write at the start of every step (inside the timed region)"},
                "e2e": e2e, "roofline": roof, "cpu_baseline": cpu, "clocks": clocks, "gpu_launches": launches,
                "detail": {"builds": table}}
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def bench_fig3(args):
    """Error-vs-rank row: hdf_build over (kernel, tol) on 5,000 points in d = 5, errors from the
    dense kernel matrix (outside the timed region)."""
    import numpy as np
    import torch
    from paper_2202_03655_gb300 import hdf, workloads as W
    ws, rank, dev = _setup(args)
    w = workload_params(args)
    n, d = w["n"], w["d"]
    stream = torch.cuda.current_stream(dev)
    x_np = W.maxnorm1_points(args.workload, n, d)
    x = torch.from_numpy(x_np).to(dev)
    cfgs = [(kn, ell, tol) for kn, ell in w["kernels"] for tol in w["tols"]]
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)     # larger than the 129 MB L2

    def build(cfg):
        kn, ell, tol = cfg
        try:
            return hdf.build(x, kn, ell, tol, precision="fp64", p_max=args.p_max, stream=stream)
        except hdf.HdfError as e:            # a size limit at the degree cap: recorded, not fatal
            return str(e)

    def one(keep):
        flush.zero_()
        out = {}
        for cfg in cfgs:
            f = build(cfg)
            if isinstance(f, str):
                out[cfg] = f
                continue
            out[cfg] = f.info if keep else None
            f.free()
        return out if keep else None

    ms_total, recs, launches, clocks = _timed(args, ws, rank, dev, stream, one)
    value = whole_job_rate(n * len(cfgs), ws, args.steps, ms_total)
    # achieved errors against the dense matrix, per (kernel, tol)
    D = torch.cdist(x, x)
    rows = []
    total_ms = {}
    for kn, ell in w["kernels"]:
        z = D / ell
        if kn == "gaussian":
            K = torch.exp(-0.5 * z * z)
        elif kn == "cauchy":
            K = 1.0 / (1.0 + z * z)
        elif kn == "matern32":
            K = (1 + 3 ** 0.5 * z) * torch.exp(-(3 ** 0.5) * z)
        else:
            K = (1 + 5 ** 0.5 * z + 5.0 / 3.0 * z * z) * torch.exp(-(5 ** 0.5) * z)
        kn_norm = torch.linalg.norm(K)
        for tol in w["tols"]:
            f = build((kn, ell, tol))
            if isinstance(f, str):
                rows.append({"kernel": kn, "tol": tol, "status": f})
                continue
            if f.info.rank <= 40000:           # exact: K~ = U S U^T from the exported factor
                U, S = f.export()
                Ut = torch.from_numpy(U).to(dev)
                Kt = (Ut * torch.from_numpy(S).to(dev)) @ Ut.T
                err = float(torch.linalg.norm(K - Kt) / kn_norm)
                how = "exact"
                del Ut, Kt
            else:                               # E |(K - K~) g|^2 = |K - K~|_F^2 over 256 N(0, I) probes
                G = torch.randn((n, 256), dtype=torch.float64, device=dev, generator=torch.Generator(dev).manual_seed(5))
                R = K @ G - f.matvec(G)
                err = float(torch.sqrt((R * R).sum() / 256) / kn_norm)
                how = "256-probe estimate (standard error <= 9%)"
                del G, R
            rows.append({"kernel": kn, "sigma": 1.0, "tol": tol, "p": f.info.p, "reached": bool(f.info.reached),
                         "rank": f.info.rank, "rel_fro_err": err, "err_how": how, "err_bound": f.info.err_bound,
                         "build_ms": f.info.t_ms[7]})
            f.free()
    del D
    # roofline: U writer of the largest factor of the sweep
    big = max((r for r in rows if "rank" in r), key=lambda r: r["rank"])
    f = build((big["kernel"], dict(w["kernels"])[big["kernel"]], big["tol"]))
    I = f.info
    nF = sum(I.s_k[k] for k in range(I.L + 1))
    ub = n * (I.rank * 8 + d * 8 + nF * 8)
    t5 = float(I.t_ms[5])
    f.free()
    peaks, peak_src = load_peaks()
    hbm = float(peaks.get("hbm_gbs", PEAKS_FALLBACK["hbm_gbs"]))
    roof = {"kernel": f"k_uwriter<double> ({big['kernel']}, tol {big['tol']}, rank {big['rank']})", "bound": "hbm",
            "achieved": ub / (t5 / 1e3) / 1e9, "peak": hbm, "unit": "GB/s",
            "peak_source": peak_src + " copy bandwidth (burst)", "traffic": None, "algorithmic_bytes": ub,
            "ms_per_launch": t5, "note": "U is 5,000 rows: L2-resident, small launch"}
    roof["frac"] = roof["achieved"] / roof["peak"]
    xh = torch.from_numpy(x_np).pin_memory()
    torch.cuda.synchronize()
    b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    b0.record(stream)
    x.copy_(xh, non_blocking=True)
    for cfg in cfgs:
        f = build(cfg)
        if not isinstance(f, str):
            f.free()
    b1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = b0.elapsed_time(b1)
    e2e = {"value": ws * n * len(cfgs) / (e2e_ms / 1e3), "unit": "points/s", "h2d_bytes_per_step": n * d * 8,
           "d2h_bytes_per_step": 0, "ms_per_step": e2e_ms}
    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu:
        from oracle import hdf as ohdf
        ns = min(args.cpu_n, 2000)
        t = time.perf_counter()
        ohdf.build(x_np[:ns], "cauchy", 1.0, 1e-3, p_max=args.p_max)
        ts_ = time.perf_counter() - t
        cpu = {"value": ns / ts_, "unit": "points/s", "cores": blas_threads() or os.cpu_count(), "kind": "oracle",
               "sample": f"one oracle build of the first {ns} points, Cauchy, tol 1e-3, FP64 numpy"}
    if rank == 0:
        line = {"metric": METRICS[args.workload], "value": value, "unit": "points/s", "n_gpus": ws,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_total / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                "config": {"workload": args.workload, "n": n, "d": d, "kernels": [k for k, _ in w["kernels"]],
                           "tols": list(w["tols"]), "p_max": args.p_max, "parallelism": f"replicas{ws}",
                           "l2": "L2 flushed by a 256 MB write at the start of every step (inside the timed region)"},
                "e2e": e2e, "roofline": roof, "cpu_baseline": cpu, "clocks": clocks, "gpu_launches": launches,
                "detail": {"sweep": rows}}
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def bench_krr(args):
    """Kernel-ridge-regression row: k-means, block operator, PCG, predictions."""
    import numpy as np
    import torch
    from paper_2202_03655_gb300 import hdf, workloads as W
    ws, rank, dev = _setup(args)
    w = workload_params(args)
    xtr_np, ytr_np, xte_np, yte_np, init = W.krr_data(args.workload)
    ntr, nte, d = len(xtr_np), len(xte_np), w["d"]
    xtr, ytr, xte = (torch.from_numpy(a).to(dev) for a in (xtr_np, ytr_np, xte_np))
    stream = torch.cuda.current_stream(dev)
    rtol, max_iter = 1e-6, 5000
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)     # larger than the 129 MB L2

    def fit_predict(xa, ya, xq):
        labels, _, km_it = hdf.kmeans(xa, init, stream=stream)
        K = hdf.KRR(xa, labels, w["kernel"], w["ell"], w["lam"], w["tol"], precision="fp32", p_max=args.p_max,
                    stream=stream)
        wv, it, res = K.solve(ya, rtol=rtol, max_iter=max_iter, stream=stream)
        pred = hdf.kernel_matvec(xq, xa, w["kernel"], w["ell"], wv, stream=stream)
        return K, km_it, it, res, pred

    def one(keep):
        flush.zero_()
        K, km_it, it, res, pred = fit_predict(xtr, ytr, xte)
        rec = (K.info(), km_it, it, res, pred) if keep else None
        K.free()
        return rec

    ms_total, recs, launches, clocks = _timed(args, ws, rank, dev, stream, one)
    value = whole_job_rate(ntr, ws, args.steps, ms_total)
    (nc, rank_tot, tms), km_it, it, res, pred = recs[-1]
    pred_np = pred.cpu().numpy()
    mse = float(np.mean((pred_np - yte_np) ** 2))
    # the dense KRR solution of Eq. (opt) with the exact kernel, for reference (outside the timed region)
    Kd = torch.cdist(xtr, xtr)
    Kd = torch.exp(-0.5 * (Kd / w["ell"]) ** 2)
    Kd.diagonal().add_(w["lam"])
    wd = torch.linalg.solve(Kd, ytr)
    del Kd
    pd = torch.exp(-0.5 * (torch.cdist(xte, xtr) / w["ell"]) ** 2) @ wd
    mse_dense = float(torch.mean((pd - torch.from_numpy(yte_np).to(dev)) ** 2))
    pred_rel = float(torch.linalg.norm(pred - pd) / torch.linalg.norm(pd))
    # Table 1's comparison on the stand-in data: test MSE of the HDF-block model and of the dense
    # exact solve for the four kernels (one untimed fit each)
    yte = torch.from_numpy(yte_np).to(dev)
    table1 = {}
    D_tt, D_qt = torch.cdist(xtr, xtr), torch.cdist(xte, xtr)

    def kfun(kn, D):
        z = D / w["ell"]
        if kn == "gaussian":
            return torch.exp(-0.5 * z * z)
        if kn == "cauchy":
            return 1.0 / (1.0 + z * z)
        if kn == "matern32":
            return (1 + 3 ** 0.5 * z) * torch.exp(-(3 ** 0.5) * z)
        return (1 + 5 ** 0.5 * z + 5.0 / 3.0 * z * z) * torch.exp(-(5 ** 0.5) * z)

    for kn in ("cauchy", "gaussian", "matern32", "matern52"):
        try:
            labels_k, _, _ = hdf.kmeans(xtr, init, stream=stream)
            Kk = hdf.KRR(xtr, labels_k, kn, w["ell"], w["lam"], w["tol"], precision="fp32", p_max=args.p_max,
                         stream=stream)
            wk, itk, _ = Kk.solve(ytr, rtol=rtol, max_iter=max_iter, stream=stream)
            pk = hdf.kernel_matvec(xte, xtr, kn, w["ell"], wk, stream=stream)
            Kk.free()
            Kd = kfun(kn, D_tt)
            Kd.diagonal().add_(w["lam"])
            pdk = kfun(kn, D_qt) @ torch.linalg.solve(Kd, ytr)
            del Kd
            table1[kn] = {"mse_hdf": float(torch.mean((pk - yte) ** 2)), "mse_dense": float(torch.mean((pdk - yte) ** 2)),
                          "cg_iterations": itk}
        except hdf.HdfError as e:
            table1[kn] = {"status": str(e)}
    del D_tt, D_qt
    # roofline of the direct kernel evaluation (the off-diagonal blocks in every CG product and
    # the predictions): one launch over nte x ntr pairs
    wr = torch.randn(ntr, dtype=torch.float64, device=dev)
    hdf.kernel_matvec(xte, xtr, w["kernel"], w["ell"], wr, stream=stream)
    a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    a0.record(stream)
    for _ in range(10):
        hdf.kernel_matvec(xte, xtr, w["kernel"], w["ell"], wr, stream=stream)
    a1.record(stream)
    torch.cuda.synchronize()
    km_ms = a0.elapsed_time(a1) / 10
    pairs = nte * ntr
    flops = pairs * (3 * d + 8)
    peak_alu = NSM * FP32_LANES_PER_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12
    roof = {"kernel": "k_direct_kernel (K(x*, x) w, 6,880 x 13,760 pairs)", "bound": "alu",
            "achieved": flops / (km_ms / 1e3) / 1e12, "peak": peak_alu, "unit": "TFLOP/s",
            "peak_source": "FP32 FMA: 152 SMs x 128 lanes x 2 x 2070 MHz (no measured FP32 peak)",
            "traffic": None, "algorithmic_flops": flops, "flops_per_pair": 3 * d + 8, "ms_per_launch": km_ms,
            "pairs_per_s": pairs / (km_ms / 1e3)}
    roof["frac"] = roof["achieved"] / roof["peak"]
    # end to end from pinned host buffers: H2D of the training and test data, the whole fit,
    # D2H of the predictions
    hx, hy, hq = (torch.from_numpy(a).pin_memory() for a in (xtr_np, ytr_np, xte_np))
    ph = torch.empty(nte, dtype=torch.float64).pin_memory()
    xd, yd, qd = torch.empty_like(xtr), torch.empty_like(ytr), torch.empty_like(xte)
    torch.cuda.synchronize()
    b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    b0.record(stream)
    xd.copy_(hx, non_blocking=True); yd.copy_(hy, non_blocking=True); qd.copy_(hq, non_blocking=True)
    K, _, _, _, pr2 = fit_predict(xd, yd, qd)
    ph.copy_(pr2, non_blocking=True)
    b1.record(stream)
    torch.cuda.synchronize()
    K.free()
    e2e_ms = b0.elapsed_time(b1)
    e2e = {"value": ws * ntr / (e2e_ms / 1e3), "unit": "points/s",
           "h2d_bytes_per_step": (ntr + nte) * d * 8 + ntr * 8, "d2h_bytes_per_step": nte * 8, "ms_per_step": e2e_ms}
    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu:
        from oracle import krr as okrr
        xs, ys, xq, _, init_s = W.krr_data(args.workload, n=min(args.cpu_n, 3000))
        t = time.perf_counter()
        lab, _, _ = okrr.kmeans(xs, init_s)
        wo, _, _, _ = okrr.krr_fit(xs, ys, lab, w["kernel"], w["ell"], w["lam"], w["tol"], rtol=rtol)
        okrr.kernel_matvec(xq, xs, w["kernel"], w["ell"], wo)
        ts_ = time.perf_counter() - t
        cpu = {"value": len(xs) / ts_, "unit": "points/s", "cores": blas_threads() or os.cpu_count(), "kind": "oracle",
               "sample": f"the same recipe at {len(xs)} training points (k-means, oracle HDF blocks, PCG, "
                         f"predictions), FP64 numpy"}
    if rank == 0:
        line = {"metric": METRICS[args.workload], "value": value, "unit": "points/s", "n_gpus": ws,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_total / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                "config": {"workload": args.workload, "n_train": ntr, "n_test": nte, "d": d, "kernel": w["kernel"],
                           "lengthscale": w["ell"], "lambda": w["lam"], "tol": w["tol"], "clusters": w["clusters"],
                           "cg_rtol": rtol, "bulk": "fp32", "parallelism": f"replicas{ws}",
                           "l2": "L2 flushed by a 256 MB write at the start of every step (inside the timed region)"},
                "e2e": e2e, "roofline": roof, "cpu_baseline": cpu, "clocks": clocks, "gpu_launches": launches,
                "detail": {"kmeans_passes": km_it, "cg_iterations": it, "cg_relres": res, "clusters": nc,
                           "rank_total": rank_tot, "factor_ms": tms[0], "precond_ms": tms[1],
                           "test_mse": mse, "test_mse_dense_exact": mse_dense,
                           "pred_rel_diff_vs_dense": pred_rel, "target_variance": float(np.var(yte_np)),
                           "table1_mse_by_kernel": table1}}
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def main():
    args = parse()
    if args.oracle_once:
        return oracle_once(args)
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "ball3_gauss":
        return bench_plain(args)
    if args.workload == "cube4_gauss":
        return bench_adjoint(args)
    if args.workload == "normal5_cauchy":
        return bench_mfree(args)
    if args.workload == "batch512_gauss":
        return bench_batch(args)
    if args.workload == "cross3_gauss":
        return bench_cross(args)
    if args.workload == "fig1_cauchy":
        return bench_fig1(args)
    if args.workload == "krr8_clusters":
        return bench_krr(args)
    if args.workload == "fig3_rank5":
        return bench_fig3(args)
    import numpy as np
    import torch
    from paper_2202_03655_gb300 import hdf, workloads as W

    ws, rank, local = dist()
    if ws > 1:
        import torch.distributed as tdist
        torch.cuda.set_device(local)
        tdist.init_process_group("nccl")
    dev = torch.device("cuda", local if ws > 1 else 0)
    torch.cuda.set_device(dev)
    w = workload_params(args)
    n, c, d = w["n"], w["ncols"], w["d"]
    x_np = W.points(args.workload, n=n)
    V_np = np.asfortranarray(W.rng(w["idx"] + 100).standard_normal((n, c)).astype(np.float32))
    x = torch.from_numpy(x_np).to(dev)
    Vc = torch.from_numpy(np.ascontiguousarray(V_np.T)).to(dev)      # (c, n) = column-major n x c
    Yc = torch.empty_like(Vc)
    stream = torch.cuda.current_stream(dev)

    def step(prec, Vblk, Yblk, keep=False):
        f = hdf.build(x, w["kernel"], w["ell"], w["tol"], precision=prec, p_max=args.p_max, stream=stream)
        f.matvec_ptr(Vblk.data_ptr(), n, c, Yblk.data_ptr(), n, stream=stream)
        info = (f.info.t_ms[5], f.matvec_timings() if keep else None)
        return f, info

    def barrier():
        if ws > 1:
            torch.distributed.barrier()

    # ---- warm-up
    for _ in range(max(args.warmup, 0)):
        f, _ = step("fp32", Vc, Yc)
        f.free()
    torch.cuda.synchronize()

    # ---- timed region (FP32 bulk)
    sampler = ClockSampler(dev.index) if rank == 0 else None
    barrier()
    torch.cuda.synchronize()
    if sampler:
        sampler.start()
    l0 = hdf.launch_count()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    uw_ms, mv_ms, infos = [], [], []
    e0.record(stream)
    for _ in range(args.steps):
        f, _ = step("fp32", Vc, Yc)
        uw_ms.append(f.info.t_ms[5])
        infos.append(f.info)
        mv_ms.append(f.matvec_timings())
        f.free()
    e1.record(stream)
    torch.cuda.synchronize()
    barrier()
    launches = hdf.launch_count() - l0
    clocks = sampler.stop() if sampler else None
    ms_total = max_over_ranks(e0.elapsed_time(e1), ws, dev)
    ms_step = ms_total / args.steps
    value = whole_job_rate(n, ws, args.steps, ms_total)

    # ---- accuracy of the benchmarked factor (outside the timed region)
    info = infos[-1]
    f, _ = step("fp32", Vc, Yc)
    rows = np.sort(W.rng(7).choice(n, 512, replace=False))
    exact = exact_rows_matvec(x, w["kernel"], w["ell"], Vc[0].double(), rows)
    approx = Yc[0][torch.from_numpy(rows).to(dev)].double().cpu().numpy()
    rel_err = float(np.linalg.norm(approx - exact) / np.linalg.norm(exact))
    f.free()

    # ---- roofline of the dominant kernel
    peaks, peak_src = load_peaks()
    r, ldu = info.rank, info.ldu
    nF = sum(info.s_k[k] for k in range(info.L + 1))
    # algorithmic bytes count the true rank r; U is stored with zero padding columns up to ldu
    # (rows padded to whole sectors, blocks narrower than 16 bytes widened), which the kernels
    # also move
    uw_bytes = n * r * 4 + n * d * 8 + n * nF * 4
    mv = np.array(mv_ms).mean(axis=0)            # utv, reduce, uw (first 64-column group)
    utv_bytes = n * r * 4 + n * c * 4
    uwm_bytes = n * r * 4 + n * c * 4
    tc = c >= 9          # FP32 column groups of 9..64 run on the tensor cores (tcgen05, 3xTF32)
    kernels = {
        "k_uwriter": (float(np.mean(uw_ms)), uw_bytes),
        ("k_tc_utv" if tc else "k_utv_tile"): (float(mv[0]), utv_bytes),
        ("k_tc_uw" if tc else "k_uw_tile"): (float(mv[2]), uwm_bytes),
    }
    dom = max(kernels, key=lambda k: kernels[k][0])
    t_dom, b_dom = kernels[dom]
    hbm = float(peaks.get("hbm_gbs", PEAKS_FALLBACK["hbm_gbs"]))
    if dom == "k_uwriter" or tc:
        roof = {"kernel": dom, "bound": "hbm", "achieved": b_dom / (t_dom / 1e3) / 1e9, "peak": hbm,
                "unit": "GB/s", "peak_source": peak_src + " copy bandwidth (burst)"}
        if tc and dom != "k_uwriter":
            flops = 3 * 2.0 * n * ldu * (16 * ((c + 15) // 16))
            roof["tensor_tflops"] = flops / (t_dom / 1e3) / 1e12
    else:
        flops = 2.0 * n * r * c
        peak_alu = NSM * FP32_LANES_PER_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12
        roof = {"kernel": dom, "bound": "alu", "achieved": flops / (t_dom / 1e3) / 1e12, "peak": peak_alu,
                "unit": "TFLOP/s", "peak_source": "FP32 FMA: 152 SMs x 128 lanes x 2 x 2070 MHz",
                "hbm_achieved_gbs": b_dom / (t_dom / 1e3) / 1e9}
    roof["frac"] = roof["achieved"] / roof["peak"]
    tpe = TRAFFIC_PER_U_ELEMENT.get(dom)
    roof["traffic"] = (tpe * n * ldu) if tpe else None
    roof["traffic_source"] = "ncu dram bytes per U element at n = 1,000,000, times n * ldU" if tpe else None
    roof["algorithmic_bytes"] = b_dom
    roof["ms_per_launch"] = t_dom
    kv_bytes = 2 * n * r * 4 + n * c * 8
    kv_ms = float(mv.sum())

    # ---- end to end through the C ABI from pinned host buffers
    xh = torch.from_numpy(x_np).pin_memory()
    Vh = torch.from_numpy(np.ascontiguousarray(V_np.T)).pin_memory()
    Yh = torch.empty_like(Vh).pin_memory()
    xd = torch.empty_like(x)
    torch.cuda.synchronize()
    b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e2e_steps = max(1, min(args.steps, 3))
    marks = []

    def e2e_step():
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(5)]
        ev[0].record(stream)
        xd.copy_(xh, non_blocking=True)
        Vc.copy_(Vh, non_blocking=True)
        ev[1].record(stream)
        f = hdf.build(xd, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
        ev[2].record(stream)
        f.matvec_ptr(Vc.data_ptr(), n, c, Yc.data_ptr(), n, stream=stream)
        ev[3].record(stream)
        Yh.copy_(Yc, non_blocking=True)
        ev[4].record(stream)
        f.free()
        marks.append(ev)

    e2e_step()              # one untimed step
    torch.cuda.synchronize()
    marks.clear()
    b0.record(stream)
    for _ in range(e2e_steps):
        e2e_step()
    b1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = b0.elapsed_time(b1) / e2e_steps
    e2e = {"value": ws * n / (e2e_ms / 1e3), "unit": "points/s", "h2d_bytes_per_step": n * d * 8 + n * c * 4,
           "d2h_bytes_per_step": n * c * 4, "ms_per_step": e2e_ms}
    # where a step's time went: a slow spell of the host link shows in the copies, memory that U has
    # to be mapped into anew in the build
    e2e["parts_ms"] = {k: [ev[i].elapsed_time(ev[i + 1]) for ev in marks]
                       for i, k in enumerate(("h2d", "build", "kv", "d2h"))}

    # ---- the solve on the benchmarked factor (outside the timed region): U^T U on the tensor
    # cores and the LU of the core lambda S^-1 + U^T U on the first call, the device triangular
    # solves and one refinement step on every call; lambda grows with n as in kernel ridge
    # regression
    solve = None
    if not args.no_solve:
        f = hdf.build(x, w["kernel"], w["ell"], w["tol"], precision="fp32", p_max=args.p_max, stream=stream)
        lam = 1e-4 * n
        b = Vc[0]
        torch.cuda.synchronize()
        s0 = time.perf_counter()
        xs = f.solve(lam, b, refine_steps=1)
        torch.cuda.synchronize()
        first = 1e3 * (time.perf_counter() - s0)
        s0 = time.perf_counter()
        xs = f.solve(lam, b, refine_steps=1)
        torch.cuda.synchronize()
        again = 1e3 * (time.perf_counter() - s0)
        res = lam * xs.double() + f.matvec(xs).double() - b.double()
        ldu_s = f.info.ldu
        pk, _ = load_peaks()
        tf32_peak = float(pk.get("bf16_tflops", PEAKS_FALLBACK["bf16_tflops"])) * 1.1 / 2.25
        gram_ms = float(f.info.t_ms[6])
        gram_flops = 3 * 2.0 * n * ldu_s * ldu_s
        solve = {"lambda": lam, "ldu": ldu_s, "first_ms": first, "again_ms": again, "gram_ms": gram_ms,
                 "lu_ms": float(f.info.lu_ms), "lu_fp64_tflops": (2.0 / 3.0) * ldu_s ** 3 / (f.info.lu_ms / 1e3) / 1e12
                 if f.info.lu_ms > 0 else None,
                 "gram_tensor_frac_of_tf32": gram_flops / (gram_ms / 1e3) / 1e12 / tf32_peak if gram_ms > 0 else None,
                 "residual": float(torch.linalg.norm(res) / torch.linalg.norm(b.double()))}
        f.free()
        del xs, res

    # ---- FP64 form of the same step
    fp64 = None
    if not args.no_fp64:
        V64 = Vc.double()
        Y64 = torch.empty_like(V64)
        f, _ = step("fp64", V64, Y64)
        f.free()
        torch.cuda.synchronize()
        a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a0.record(stream)
        f, _ = step("fp64", V64, Y64)
        a1.record(stream)
        torch.cuda.synchronize()
        t64 = a0.elapsed_time(a1)
        mv64 = f.matvec_timings()
        approx64 = Y64[0][torch.from_numpy(rows).to(dev)].cpu().numpy()
        fp64 = {"ms_per_step": t64, "points_per_s": n / (t64 / 1e3), "build_ms": f.info.t_ms[7],
                "kv_ms": float(mv64.sum()), "kv_gbs": (2 * n * f.info.ldu * 8 + n * c * 16) / (float(mv64.sum()) / 1e3) / 1e9,
                "rank": f.info.rank, "rel_err_sampled": float(np.linalg.norm(approx64 - exact) / np.linalg.norm(exact))}
        f.free()
        del V64, Y64

    # ---- CPU oracle baseline on a bounded sample (rank 0, N = 1)
    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu:
        ns = min(args.cpu_n, n)
        xs = x_np[:ns]
        Vs = V_np[:ns].astype(np.float64)
        ts = cpu_oracle_step(xs, w, Vs, args.p_max)
        cpu = cpu_baseline_line(ns / ts, f"first {ns} of the {n} points, one full step (build + K~V, {c} columns), "
                                         "FP64 numpy", args, args.workload)

    if rank == 0:
        line = {
            "metric": METRICS[args.workload],
            "value": value, "unit": "points/s", "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic",
            "config": {"workload": args.workload, "n": n, "d": d, "kernel": w["kernel"], "lengthscale": w["ell"],
                       "tol": w["tol"], "ncols": c, "p_max": args.p_max, "p": info.p, "reached": bool(info.reached),
                       "rank": r, "ldu": ldu, "U_bytes": n * ldu * 4, "parallelism": f"replicas{ws}",
                       "l2": "inputs larger than L2 (U alone is ~40 GB)"},
            "e2e": e2e,
            "roofline": roof,
            "cpu_baseline": cpu,
            "clocks": clocks,
            "gpu_launches": launches,
            "detail": {
                "rel_err_sampled_vs_exact": rel_err, "err_bound": info.err_bound, "cheb_tail": info.cheb_tail,
                "build_ms": float(np.mean([i.t_ms[7] for i in infos])),
                "build_phase_ms": [float(np.mean([i.t_ms[q] for i in infos])) for q in range(8)],
                "build_points_per_s": n / (np.mean([i.t_ms[7] for i in infos]) / 1e3),
                "kv_ms": kv_ms, "kv_gbs": kv_bytes / (kv_ms / 1e3) / 1e9,
                "kernel_ms": {k: v[0] for k, v in kernels.items()},
                "solve": solve,
                "fp64": fp64,
            },
        }
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())

"""Benchmark: Wilson-loop k-points per second on the BBH quadrupole 60 x 60 workload.

One step = the whole hot path over the 60 x 60 grid of the BBH model (gamma = 0.5,
lambda = 1, p = 2): Bloch Hamiltonians, eigensolve (FP32 + FP64 refinement in the
mixed path, FP64 in the plain path), overlaps, ordered loop products, eigenphases,
and the nested loop on the lower Wannier band at every base point.

  value   device time of captured-graph replays (inputs resident), L2 flushed
          between steps, mixed precision (the fp64 path is reported beside it);
  e2e     the public Python API on host inputs, including the upload of the hopping
          list and the read-back of the phases, wall clock per step;
  --impl reference   the FP64 CPU oracle on the same workload.

Prints one JSON line on rank 0.  Under torchrun every rank runs its own copy of the
workload (independent problems, no data-path collective): weak scaling.

The CPU oracle (``oracle/``, test infrastructure) runs only in the bench's CPU leg,
never inside a timed GPU region: the ``cpu_baseline`` measurement, the reference arm,
and the parity of the timed outputs against it (``phase_err_rad`` keys), each after
the GPU timing of its block.
"""
from __future__ import annotations

import argparse
import json
import os
import platform
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "Wilson-loop k-points/sec (eigh+overlap+phases) mixed vs FP64 at ≤1e-6 rad; p50/p99 latency"
UNIT = "k-points/s"
WORKLOAD = "bbh_quadrupole_60x60_nested (gamma=0.5, lambda=1, n=4, p=2, m=1, N=N_t=60)"
FP64_NOMINAL_TFLOPS = 1.25     # GB300 dense FP64, NVIDIA's figure
FP32_NOMINAL_TFLOPS = 152 * 128 * 2 * 2.07e9 / 1e12   # SMs x FP32 lanes x FMA x max clock: 80.5
CSRC = os.path.join(ROOT, "paper_2312_13051_gb300", "csrc")
PROFILES = os.path.join(ROOT, "profiles")


def log(*a):
    print(*a, file=sys.stderr, flush=True)


# ------------------------------------------------------------------ distributed helpers
def dist_env():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)), \
        int(os.environ.get("LOCAL_RANK", 0))


def dist_init(backend: str):
    import torch.distributed as dist
    if not dist.is_initialized():
        dist.init_process_group(backend=backend)
    return dist


def reduce_max(value: float, device=None) -> float:
    """Max of a float over all ranks (identity without a process group)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()):
        return value
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def barrier(device=None):
    import torch.distributed as dist
    if dist.is_available() and dist.is_initialized():
        if device is not None and device.type == "cuda":
            dist.barrier(device_ids=[device.index])
        else:
            dist.barrier()


def weak_scaling_value(units_per_rank: float, steps: int, world: int, max_seconds: float) -> float:
    """Whole-job throughput: all ranks' units over the slowest rank's time."""
    return units_per_rank * steps * world / max_seconds


# ------------------------------------------------------------------ peaks and traffic
def measure_peaks(dev):
    """FP64 and FP32 (SIMT, TF32 off) pipe peaks measured in this run: cuBLAS DGEMM and
    SGEMM on square matrices, best of 5 timed with CUDA events (2 n^3 flops each)."""
    import torch
    out = {}
    tf32 = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = False
    try:
        for name, dt, n in (("fp64", torch.float64, 4096), ("fp32", torch.float32, 8192)):
            a = torch.randn(n, n, dtype=dt, device=dev)
            b = torch.randn(n, n, dtype=dt, device=dev)
            for _ in range(2):
                torch.matmul(a, b)
            best = float("inf")
            for _ in range(5):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                torch.matmul(a, b)
                e1.record()
                e1.synchronize()
                best = min(best, e0.elapsed_time(e1))
            out[name] = 2.0 * n ** 3 / (best * 1e-3) / 1e12
            del a, b
    finally:
        torch.backends.cuda.matmul.allow_tf32 = tf32
    torch.cuda.empty_cache()
    return out


def sources_sha256(names) -> str:
    import hashlib
    h = hashlib.sha256()
    for nm in names:
        with open(os.path.join(CSRC, nm), "rb") as f:
            h.update(nm.encode() + b"\0" + f.read())
    return h.hexdigest()


def committed_traffic(kernel: str, workload: str):
    """DRAM bytes per launch of `kernel` on `workload` from the ncu summaries under
    profiles/: a line `traffic: kernel=K workload=W dram_bytes_per_launch=B
    sources=a.cu,b.cuh sha256=H`.  Returns (bytes, summary file), or (None, reason) when
    no capture exists or the kernel's sources changed since it was taken."""
    import glob
    for path in sorted(glob.glob(os.path.join(PROFILES, "*.md"))):
        for line in open(path):
            if not line.startswith("traffic:"):
                continue
            kv = dict(x.split("=", 1) for x in line.split()[1:] if "=" in x)
            if kv.get("kernel") != kernel or kv.get("workload") != workload:
                continue
            if sources_sha256(kv["sources"].split(",")) != kv.get("sha256"):
                return None, f"{os.path.basename(path)}: sources changed since the capture"
            return int(kv["dram_bytes_per_launch"]), os.path.basename(path)
    return None, "no ncu capture of this kernel and workload under profiles/"


# ------------------------------------------------------------------ algorithmic work
def algorithmic_flops(n, p, N, Nt, m, nhop):
    """Real flops per launch of each kernel (complex MAC = 8 flops)."""
    K = N * Nt
    return {
        "states": K * (16.0 / 3.0 * n ** 3 + 8.0 * n * n * p + 8.0 * nhop),
        "overlaps": K * 8.0 * n * p * p,
        "loops": Nt * (N * 8.0 * p ** 3 + 10.0 * p ** 3 + N * (8.0 * n * p * m + 8.0 * p * p * m)),
        "nested": N * (Nt * (8.0 * n * m * m + 8.0 * m ** 3) + 10.0 * m ** 3),
    }


# ------------------------------------------------------------------ clocks
class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        # raw samples go to BW_CLOCKS_DIR when set (kept for inspection), else to a
        # temporary directory; the JSON line carries their summary either way
        d = os.environ.get("BW_CLOCKS_DIR") or tempfile.gettempdir()
        self.path = os.path.join(d, f"berrywl_clocks_rank{index}.csv")

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}",
                                          f"--query-gpu={self.QUERY}", "--format=csv,noheader,nounits",
                                          "-lms", "100"], stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception as e:       # no nvidia-smi: report nothing
            log("clock sampling unavailable:", e)
            self.proc = None

    def stop(self):
        if not self.proc:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        self.proc.terminate()
        self.proc.wait(timeout=10)
        self.f.close()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax),
                "reasons": sorted(reasons), "samples": len(sm)}


# ------------------------------------------------------------------ CPU oracle
_BLAS_VARS = ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS")


def cpu_model() -> str:
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.lower().startswith("model name"):
                return line.split(":", 1)[1].strip()
    except Exception:
        pass
    return platform.processor() or platform.machine()


class OraclePool:
    """The oracle's per-row work spread over host processes (started with spawn, so it
    is safe after CUDA has been initialised), one BLAS thread per worker: the per-k
    multiprocessing mode of the CPU baseline.  Workers are started eagerly so that the
    single-thread setting reaches every one of them."""

    def __init__(self, workers: int):
        import concurrent.futures as cf
        import multiprocessing as mp
        self.workers = workers
        saved = {k: os.environ.get(k) for k in _BLAS_VARS}
        os.environ.update({k: "1" for k in _BLAS_VARS})
        try:
            self.ex = cf.ProcessPoolExecutor(max_workers=workers, mp_context=mp.get_context("spawn"))
            fs = [self.ex.submit(time.sleep, 0.2) for _ in range(workers)]
            for f in fs:
                f.result(timeout=120)
        finally:
            for k, v in saved.items():
                if v is None:
                    os.environ.pop(k, None)
                else:
                    os.environ[k] = v

    def row_map(self, fn, tasks):
        return self.ex.map(fn, list(tasks), chunksize=1, timeout=600)

    def close(self):
        self.ex.shutdown(cancel_futures=True)


def run_oracle_once(wl, pool=None):
    import oracle
    kw = {"row_map": pool.row_map} if pool is not None else {}
    return oracle.nested_wilson_loop(wl.model, wl.plane, wl.p, m=wl.nested_m, **kw)


def _time_runs(wl, pool, min_seconds):
    runs, t0 = 0, time.perf_counter()
    while True:
        run_oracle_once(wl, pool)
        runs += 1
        el = time.perf_counter() - t0
        if el >= min_seconds:
            return runs, el


def cpu_baseline(wl, min_seconds: float = 10.0):
    """The oracle on the host cores, in both modes the measurement plan names, the better
    one reported: (a) one process, LAPACK threaded by the BLAS library (at n = 4 nothing
    threads, so it runs on one core); (b) the transverse rows of each run spread over
    all cores by a process pool, one BLAS thread each.  A sample = repeated full runs of
    the workload for at least min_seconds per mode."""
    K = wl.plane.N * wl.plane.N_t
    ncpu = os.cpu_count() or 1
    modes = {}
    run_oracle_once(wl)
    runs, el = _time_runs(wl, None, min_seconds / 3)
    modes["threaded_lapack"] = {"value": K * runs / el, "cores": 1, "runs": runs, "seconds": el}
    pool = OraclePool(min(ncpu, wl.plane.N_t))
    try:
        run_oracle_once(wl, pool)
        runs, el = _time_runs(wl, pool, min_seconds)
    finally:
        pool.close()
    modes["per_row_processes"] = {"value": K * runs / el, "cores": pool.workers, "runs": runs,
                                  "seconds": el}
    best = max(modes, key=lambda m: modes[m]["value"])
    b = modes[best]
    return {"value": b["value"], "unit": UNIT, "cores": b["cores"], "kind": "oracle",
            "mode": best, "nproc": ncpu, "cpu_model": cpu_model(), "machine": platform.machine(),
            "sample": f"{b['runs']} full runs of the 60x60 BBH nested workload (numpy FP64) in "
                      f"{b['seconds']:.1f} s, mode {best}",
            "modes": modes}


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    from paper_2312_13051_gb300 import inputs as I
    wl = I.config_bbh()
    K = wl.plane.N * wl.plane.N_t
    ncpu = os.cpu_count() or 1
    pool = OraclePool(min(ncpu, wl.plane.N_t))
    try:
        for _ in range(args.warmup):
            run_oracle_once(wl, pool)
        times = []
        for _ in range(args.steps):
            t0 = time.perf_counter()
            run_oracle_once(wl, pool)
            times.append(time.perf_counter() - t0)
    finally:
        pool.close()
    total = sum(times)
    value = K * args.steps / total
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": WORKLOAD, "precision": "fp64 (CPU oracle)"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": pool.workers, "kind": "oracle",
                             "nproc": ncpu, "cpu_model": cpu_model(),
                             "sample": "each step: the full 60x60 BBH nested workload, numpy FP64, "
                                       f"rows spread over {pool.workers} processes (one BLAS thread "
                                       "each)"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "latency_ms": {"p50": 1e3 * float(np.percentile(times, 50)),
                           "p99": 1e3 * float(np.percentile(times, 99))}}
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------------ GPU path
def time_call_graph(ctx, call, out, steps, warmup, flush, dev, soak_s=0.5, profile_steps=None):
    """Captured-graph replays of `call` timed with CUDA events on the replay stream, L2
    flushed (a 256 MB write) before every timed step.  Returns (total device ms,
    per-kernel ms totals over the profiled replays, kernels per call, outputs as numpy,
    per-step ms).  The timed graph carries no timing marks; a second capture with
    per-kernel CUDA-event marks gives the breakdown (profile_steps replays)."""
    import torch
    s = torch.cuda.Stream(device=dev)
    with torch.cuda.stream(s):
        for _ in range(max(min(warmup, 3), 1)):
            call()
    ctx.status(s)

    def replay_steps(g, n, per_kernel):
        with torch.cuda.stream(s):
            for _ in range(min(warmup, 3)):
                g.replay()
            t_end = time.perf_counter() + soak_s          # untimed soak so clocks settle
            while time.perf_counter() < t_end:
                g.replay()
        torch.cuda.synchronize(dev)
        ev0 = [torch.cuda.Event(enable_timing=True) for _ in range(n)]
        ev1 = [torch.cuda.Event(enable_timing=True) for _ in range(n)]
        barrier(dev)
        torch.cuda.synchronize(dev)
        with torch.cuda.stream(s):
            for k in range(n):
                flush.add_(1)                              # write > L2 between steps
                ev0[k].record(s)
                g.replay()
                ev1[k].record(s)
                if per_kernel is not None:
                    ev1[k].synchronize()
                    for name, ms in ctx.profile_read():
                        per_kernel[name] = per_kernel.get(name, 0.0) + ms
        torch.cuda.synchronize(dev)
        barrier(dev)
        return [a.elapsed_time(b) for a, b in zip(ev0, ev1)]

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        call()
    ctx.status(s)
    per_step = replay_steps(g, steps, None)
    total = sum(per_step)
    ctx.status(s)
    outs = [o.cpu().numpy() for o in out]
    del g
    ctx.set_profiling(True)
    gp = torch.cuda.CUDAGraph()
    with torch.cuda.graph(gp, stream=s):
        call()
    ctx.status(s)
    per_kernel = {}
    replay_steps(gp, profile_steps or steps, per_kernel)
    ctx.status(s)
    ctx.set_profiling(False)
    launches = len(per_kernel)
    del gp
    return total, per_kernel, launches, outs, per_step


def time_graph(lib, ctx, wl, precision, steps, warmup, flush, dev, nested=True):
    """The headline call (BBH nested, or the plain loop) under time_call_graph."""
    import torch
    if nested:
        out = (torch.empty((wl.plane.N_t, wl.p), dtype=torch.float64, device=dev),
               torch.empty((wl.plane.N, wl.nested_m), dtype=torch.float64, device=dev),
               torch.empty((wl.plane.N_t,), dtype=torch.float64, device=dev),
               torch.empty((wl.plane.N_t,), dtype=torch.float64, device=dev))
        call = lambda: lib.nested_wilson_loop(wl.model, wl.plane, wl.p, m=wl.nested_m,
                                              precision=precision, ctx=ctx, check=False, out=out)
    else:
        out = (torch.empty((wl.plane.N_t, wl.p), dtype=torch.float64, device=dev),
               torch.empty((wl.plane.N_t,), dtype=torch.float64, device=dev))
        call = lambda: lib.wilson_loop(wl.model, wl.plane, wl.p, precision=precision, ctx=ctx,
                                       check=False, out=out)
    return time_call_graph(ctx, call, out, steps, warmup, flush, dev)


def _eig_frac(fl, st, peak):
    """Algorithmic eigensolve flops (16/3 n^3 + 8 n^2 nbt per k-point) over the time of
    the eigensolve stages (tridiagonalisation, bisection, inverse iteration,
    back-transform), as a fraction of `peak` TFLOP/s."""
    ms = sum(st.get(k, 0.0) for k in ("lg_tridiag", "lg_bisect", "lg_invit", "lg_backtransform"))
    if ms <= 0.0:
        return None
    return (fl["lg_tridiag"] + fl["lg_backtransform"]) / (ms * 1e-3) / 1e12 / peak


def stage_pipe(stage, mixed, polished, p):
    """The pipe ("fp32" or "fp64") that an n > 32 stage runs on.  The eigensolve stages run in
    FP32 in the mixed request and in an FP64 request that starts from an FP32 solve
    (polished: the call has an lg_polish stage, whose own products are FP64); overlaps, loop
    products and, from 128 bands on, eigenphases of the mixed request are double-float on
    the FP32 pipe."""
    if stage == "lg_polish":
        return "fp64"
    if stage.startswith("lg_"):
        return "fp32" if mixed or polished else "fp64"
    if stage == "eigenphases" and p < 128:
        return "fp64"
    return "fp32" if mixed else "fp64"


PIPE_SOURCE = {"fp32": "measured cuBLAS SGEMM 8192^3, TF32 off (the FP32 pipe the stage runs on)",
               "fp64": "measured cuBLAS DGEMM 4096^3 (FP64 pipe)"}


def manyband_stage_flops(n, p, N, Nt, nnz_groups, mixed, n_ent=None, polished=False):
    """Algorithmic flops of each stage of the n > 32 Wilson-loop call over K = N Nt
    k-points (complex multiply-add = 8 flops): Bloch sum 8 per hopping group,
    Householder tridiagonalisation 16/3 n^3, back-transform of nbt vectors 8 n^2 nbt,
    refinement 8 n_ent p (H Q from the n_ent assembled entries of H) + 16 n (n - p) p +
    16 n p^2 (mixed, and polished FP64 requests), the polish's FP64 products 8 n_ent p +
    16 n p^2 (H Q, Q^dag H Q and the Gram matrix by half, Q G), overlaps 8 n p^2, loop
    products 8 p^3 per step plus ~10 p^3 for the eigenphases of each loop; bisection and
    inverse iteration are O(n p)."""
    n_ent = n * n if n_ent is None else n_ent
    K = N * Nt
    nbt = min(n, p + 1) if mixed or polished else p
    # keys: the stage names the library's per-kernel timing marks carry
    fl = {"lg_tridiag": K * 16.0 / 3.0 * n ** 3, "lg_backtransform": K * 8.0 * n * n * nbt,
          "overlaps": K * 8.0 * n * p * p, "loops": Nt * (N * 8.0 * p ** 3 + 10.0 * p ** 3),
          "lg_build": K * 8.0 * nnz_groups}
    if mixed or polished:
        fl["lg_refine"] = K * (8.0 * n_ent * p + 16.0 * n * (n - p) * p + 16.0 * n * p * p)
    if polished:
        fl["lg_polish"] = K * (8.0 * n_ent * p + 16.0 * n * p * p)
    return fl


def time_e2e(lib, ctx, wl, precision, steps, warmup, dev):
    """Public API on host inputs: upload of the hopping list inside the call, results
    copied back to pinned host memory, wall clock per step."""
    import torch
    # the four outputs are views of one device buffer, read back by one copy
    shapes = ((wl.plane.N_t, wl.p), (wl.plane.N, wl.nested_m), (wl.plane.N_t,), (wl.plane.N_t,))
    sizes = [int(np.prod(sh)) for sh in shapes]
    dbuf = torch.empty(sum(sizes), dtype=torch.float64, device=dev)
    out = tuple(v.view(sh) for v, sh in zip(torch.split(dbuf, sizes), shapes))
    host = torch.empty(sum(sizes), dtype=torch.float64, pin_memory=True)
    s = torch.cuda.current_stream(dev)

    def step():
        lib.nested_wilson_loop(wl.model, wl.plane, wl.p, m=wl.nested_m, precision=precision,
                               ctx=ctx, check=False, out=out)
        host.copy_(dbuf, non_blocking=True)
        s.synchronize()

    for _ in range(max(warmup, 3)):
        step()
    ctx.status()
    lat = []
    barrier(dev)
    torch.cuda.synchronize(dev)
    for _ in range(steps):
        t0 = time.perf_counter()
        step()
        lat.append(time.perf_counter() - t0)
    barrier(dev)
    ctx.status()
    m = wl.model
    h2d = int(m.R.nbytes + m.i.nbytes + m.j.nbytes + m.t.nbytes)
    d2h = int(host.numel() * host.element_size())
    return sum(lat), lat, h2d, d2h


def run_ours(args):
    import torch
    rank, world, local = dist_env()
    if world > 1:
        dist_init("nccl")
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    from paper_2312_13051_gb300 import build as B
    B.build()
    from paper_2312_13051_gb300 import _lib as lib
    from paper_2312_13051_gb300 import inputs as I
    import oracle

    wl = I.config_bbh()
    K = wl.plane.N * wl.plane.N_t
    ctx = lib.Context(local)
    flush = torch.zeros(256 << 20, dtype=torch.uint8, device=dev)   # 256 MB > 129 MB L2
    peaks = measure_peaks(dev)
    clocks = ClockSampler(local)
    clocks.start()
    res = {}
    for prec in ("mixed", "fp64"):
        total_ms, per_kernel, nker, outs, per_step = time_graph(lib, ctx, wl, prec, args.steps,
                                                                args.warmup, flush, dev)
        res[prec] = dict(total_ms=total_ms, per_kernel=per_kernel, nker=nker, outs=outs,
                         per_step=per_step)
    # saturated batch: the plain Wilson loop of the same model on a 64x finer transverse
    # grid (230 400 k-points, 3840 independent loops per call), which fills every SM
    sat = I.Workload("bbh_60x3840", wl.model, I.Plane(wl.plane.N, 64 * wl.plane.N_t), wl.p)
    sat_res = {}
    if not args.no_saturated:
        for prec in ("mixed", "fp64"):
            t, pk, nk, outs, _ = time_graph(lib, ctx, sat, prec, max(3, args.steps // 4),
                                            args.warmup, flush, dev, nested=False)
            sat_res[prec] = dict(total_ms=t, per_kernel=pk, nker=nk, steps=max(3, args.steps // 4),
                                 phases=outs[0])
    # many-band model (n = 256, p = 64, 101 x 101): where the mixed path pays off;
    # graph replays of the whole call, L2 flushed between steps, per-stage marks
    mb_res = {}
    if not args.no_manyband:
        mb = I.config_manyband()
        for prec in ("mixed", "fp64"):
            out = (torch.empty((mb.plane.N_t, mb.p), dtype=torch.float64, device=dev),
                   torch.empty((mb.plane.N_t,), dtype=torch.float64, device=dev))
            call = (lambda prec=prec, out=out:
                    lib.wilson_loop(mb.model, mb.plane, mb.p, precision=prec, ctx=ctx, check=False,
                                    out=out))
            t, pk, nk, outs, per_step = time_call_graph(ctx, call, out, args.manyband_steps, 1, flush,
                                                        dev, soak_s=0.0, profile_steps=1)
            mb_res[prec] = dict(total_ms=t, steps=args.manyband_steps, stages=pk, nker=nk,
                                phases=outs[0], per_step=per_step)
        # the spin-resolved (C_down sector) and nested (lower Wannier band) loops of the
        # same plane, mixed request, one profiled call each
        kinds = [k for k in args.manyband_kinds.split(",") if k in ("spin", "nested")]
        for kind in kinds:
            if kind == "spin":
                call = lambda: lib.spin_resolved_wilson_loop(mb.model, mb.plane, mb.p, mb.spin_op, -1,
                                                             precision="mixed", ctx=ctx, want_pso=False)
            else:
                call = lambda: lib.nested_wilson_loop(mb.model, mb.plane, mb.p, m=mb.nested_m,
                                                      precision="mixed", ctx=ctx)
            call()
            ctx.status()
            ctx.set_profiling(True)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize(dev)
            e0.record()
            call()
            e1.record()
            e1.synchronize()
            stages = dict(ctx.profile_read())
            ctx.set_profiling(False)
            ctx.status()
            mb_res[kind + "_mixed"] = dict(ms=e0.elapsed_time(e1), stages=stages)
    # disordered spin-Hall supercells (L x L cells of the config-0 model, W = 2, 16 x 16
    # supercell k-grid, half filling): seeded realisations, one graph replay of the whole
    # call per realisation and precision, L2 flushed before it, per-stage marks
    sc_res = {}
    if not args.no_supercell:
        for Ls in [int(x) for x in args.supercell_sides.split(",") if x]:
            for prec in ("mixed", "fp64"):
                acc = dict(total_ms=0.0, stages={}, phases=[], per_call=[])
                for seed in range(args.supercell_realisations):
                    msc = I.supercell(I.spin_hall(1.0), Ls, W=2.0, seed=seed)
                    psc, plsc = msc.n // 2, I.Plane(16, 16)
                    out = (torch.empty((plsc.N_t, psc), dtype=torch.float64, device=dev),
                           torch.empty((plsc.N_t,), dtype=torch.float64, device=dev))
                    call = (lambda m_=msc, pl_=plsc, p_=psc, prec=prec, out=out:
                            lib.wilson_loop(m_, pl_, p_, precision=prec, ctx=ctx, check=False, out=out))
                    t, pk, _, outs, _ = time_call_graph(ctx, call, out, 1, 1, flush, dev, soak_s=0.0,
                                                        profile_steps=1)
                    acc["total_ms"] += t
                    acc["per_call"].append(t)
                    for k, v in pk.items():
                        acc["stages"][k] = acc["stages"].get(k, 0.0) + v
                    acc["phases"].append(outs[0])
                sc_res[(Ls, prec)] = acc
    clk = clocks.stop()
    e2e_s, lat, h2d, d2h = time_e2e(lib, ctx, wl, "mixed", args.steps, args.warmup, dev)

    # parity of the timed outputs against the oracle (rank 0 computes the reference)
    err = {}
    if rank == 0:
        ref_ph, ref_n, _, _ = oracle.nested_wilson_loop(wl.model, wl.plane, wl.p, m=wl.nested_m)
        for prec in res:
            ph, nest = res[prec]["outs"][0], res[prec]["outs"][1]
            err[prec] = max(max(oracle.circular_match_error(ph[r], ref_ph[r]) for r in range(ph.shape[0])),
                            max(oracle.circular_match_error(nest[j], ref_n[j]) for j in range(nest.shape[0])))
        if mb_res:              # one transverse row of the many-band plane vs the oracle
            row = 37
            plr = I.Plane(mb.plane.N, 1, origin=tuple(np.array(mb.plane.trans_dir) * row / mb.plane.N_t))
            ref_mb, _ = oracle.wilson_loop(mb.model, plr, mb.p)
            for prec in ("mixed", "fp64"):
                mb_res[prec]["phase_err_rad"] = oracle.circular_match_error(mb_res[prec]["phases"][row], ref_mb[0])
        for Ls in sorted({k[0] for k in sc_res}):   # one transverse row of realisation 0
            row = 5
            msc = I.supercell(I.spin_hall(1.0), Ls, W=2.0, seed=0)
            plr = I.Plane(16, 1, origin=(0.0, row / 16.0, 0.0))
            t0 = time.perf_counter()
            ref_sc, _ = oracle.wilson_loop(msc, plr, msc.n // 2)
            t_row = time.perf_counter() - t0
            for prec in ("mixed", "fp64"):
                sc_res[(Ls, prec)]["phase_err_rad"] = oracle.circular_match_error(
                    sc_res[(Ls, prec)]["phases"][0][row], ref_sc[0])
            sc_res[(Ls, "cpu")] = dict(seconds=t_row, k_points=16)
        for prec in sat_res:   # rows 64 i of the fine grid are the k-points of row i
            ph = sat_res[prec]["phases"]
            sat_res[prec]["phase_err_rad"] = max(
                oracle.circular_match_error(ph[64 * r], ref_ph[r]) for r in range(ref_ph.shape[0]))

    max_s = {p: reduce_max(res[p]["total_ms"] / 1e3, dev) for p in res}
    max_e2e = reduce_max(e2e_s, dev)
    if rank != 0:
        return 0
    value = weak_scaling_value(K, args.steps, world, max_s["mixed"])
    fp64_value = weak_scaling_value(K, args.steps, world, max_s["fp64"])
    hop_groups = len(np.unique(np.stack([wl.model.i, wl.model.j,
                                         wl.model.R[:, 0], wl.model.R[:, 1], wl.model.R[:, 2]], 1), axis=0))
    flops = algorithmic_flops(wl.model.n, wl.p, wl.plane.N, wl.plane.N_t, wl.nested_m, hop_groups)
    pk = res["mixed"]["per_kernel"]
    if "overlaps" not in pk:      # formed inside the loop kernel
        flops["loops"] += flops["overlaps"]
    if "states" not in pk:        # solved inside the loop kernel
        flops["loops"] += flops["states"]
    if "nested" not in pk:        # nested loops in the same (cooperative) launch
        flops["loops"] += flops["nested"]
    dom = max(pk, key=pk.get)
    avg_ms = pk[dom] / args.steps
    achieved = flops[dom] / (avg_ms * 1e-3) / 1e12
    peak = peaks["fp64"]
    shares = {k: v / sum(pk.values()) for k, v in pk.items()}
    fused = dom == "loops" and "states" not in pk
    traffic, traffic_src = (committed_traffic("k_loops_fused_df", "bbh_60x60_nested") if fused
                            else (None, "no capture of this kernel"))
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": res["mixed"]["total_ms"] / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "df32+f64",
        "data": "synthetic",
        "config": {"workload": WORKLOAD,
                   "precision": "mixed request: at n = 4, p = 2 states, overlaps and loop products "
                                "in double-float (pairs of FP32, ~48-bit) on the FP32 pipe (FP32 "
                                "Jacobi + double-float Newton refinement), phase tables, Bloch "
                                "factors and eigenphases in double-float, one cooperative kernel "
                                "with the plan in its parameters; FP32 solve + "
                                "FP64-grade refinement for larger n (manyband block)",
                   "timing": "CUDA-graph replay of the whole call, CUDA events per step",
                   "l2": "flushed between steps (256 MB write)",
                   "parallelism": f"replicas x{world}"},
        "fp64": {"value": fp64_value, "ms_per_step": res["fp64"]["total_ms"] / args.steps,
                 "dtype": "f64", "phase_err_rad": err.get("fp64"),
                 "kernel_ms_per_step": {k: v / args.steps for k, v in res["fp64"]["per_kernel"].items()}},
        "mixed_over_fp64": fp64_value and value / fp64_value,
        "phase_err_rad": err.get("mixed"),
        "kernel_ms_per_step": {k: v / args.steps for k, v in pk.items()},
        "roofline": {"kernel": "k_loops_fused_df" if fused else dom, "bound": "alu",
                     "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
                     "traffic": traffic, "traffic_source": traffic_src,
                     "peak_source": "measured in this run: cuBLAS DGEMM 4096^3, best of 5 (the "
                                    "FP64-grade arithmetic the path delivers, computed in "
                                    "double-float on the FP32 pipe)",
                     "frac_of_nominal_fp64": achieved / FP64_NOMINAL_TFLOPS,
                     "fp32_pipe_frac_of_measured_sgemm": achieved / peaks["fp32"],
                     "algorithmic_flops_per_launch": flops[dom], "share": shares[dom],
                     "note": "latency-bound at 3600 k-points: 60 loops, one CTA each, on 60 of "
                             "152 SMs (the saturated block fills the SMs)"},
        "peaks_measured_tflops": peaks,
        "latency_ms": {"p50": 1e3 * float(np.percentile(lat, 50)),
                       "p99": 1e3 * float(np.percentile(lat, 99))},
        "e2e": {"value": weak_scaling_value(K, args.steps, world, max_e2e), "unit": UNIT,
                "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
        "gpu_launches": res["mixed"]["nker"] * args.steps,
        "clocks": clk,
    }
    if sat_res:
        Ks = sat.plane.N * sat.plane.N_t
        fl_s = algorithmic_flops(wl.model.n, wl.p, sat.plane.N, sat.plane.N_t, 0, hop_groups)
        blk = {"workload": "bbh_quadrupole_60x3840 plain Wilson loop (same model, 64x finer "
                           "transverse grid: 3840 independent loops)",
               "k_points_per_call": Ks}
        if "overlaps" not in sat_res["mixed"]["per_kernel"]:
            fl_s["loops"] += fl_s["overlaps"]
        if "states" not in sat_res["mixed"]["per_kernel"]:
            fl_s["loops"] += fl_s["states"]
        for prec, r in sat_res.items():
            pks = r["per_kernel"]
            d = max(pks, key=pks.get)
            ach = fl_s[d] / (pks[d] / r["steps"] * 1e-3) / 1e12
            blk[prec] = {"value": weak_scaling_value(Ks, r["steps"], world, reduce_max(r["total_ms"] / 1e3, dev)),
                         "ms_per_step": r["total_ms"] / r["steps"], "phase_err_rad": r.get("phase_err_rad"),
                         "kernel_ms_per_step": {k: v / r["steps"] for k, v in pks.items()},
                         "roofline": {"kernel": d, "bound": "alu", "achieved": ach, "peak": peak,
                                      "unit": "TFLOP/s", "frac": ach / peak,
                                      "peak_source": "measured cuBLAS DGEMM (FP64-grade work)",
                                      "fp32_pipe_frac_of_measured_sgemm": ach / peaks["fp32"]}}
        line["saturated"] = blk
    if mb_res:
        Km = mb.plane.N * mb.plane.N_t
        nnz_groups = len(np.unique(np.stack([mb.model.i, mb.model.j, mb.model.R[:, 0], mb.model.R[:, 1],
                                             mb.model.R[:, 2]], 1), axis=0))
        n_ent = len(np.unique(np.stack([mb.model.i, mb.model.j], 1), axis=0))
        blk = {"workload": f"manyband n=256 p=64 101x101 plain Wilson loop ({args.manyband_steps} "
                           "graph replays per precision, L2 flushed between them)",
               "k_points_per_call": Km}
        for prec in ("mixed", "fp64"):
            r = mb_res[prec]
            ms = r["total_ms"] / r["steps"]
            st = r["stages"]
            polished = "lg_polish" in st
            fl = manyband_stage_flops(mb.model.n, mb.p, mb.plane.N, mb.plane.N_t, nnz_groups,
                                      prec == "mixed", n_ent, polished)
            if "eigenphases" in st:         # a stage of its own
                fl["eigenphases"] = mb.plane.N_t * 10.0 * mb.p ** 3
                fl["loops"] -= fl["eigenphases"]
            d = max((k for k in st if k in fl), key=st.get)
            ach = fl[d] / (st[d] * 1e-3) / 1e12
            pipe = stage_pipe(d, prec == "mixed", polished, mb.p)
            pk_ = peaks[pipe]
            blk[prec] = {"value": weak_scaling_value(Km, r["steps"], world,
                                                     reduce_max(r["total_ms"] / 1e3, dev)),
                         "ms_per_call": ms, "dtype": "f32+df32" if prec == "mixed" else "f64",
                         "per_step_ms": [round(x, 3) for x in r["per_step"]],
                         "stage_ms": {k: round(v, 3) for k, v in st.items()},
                         "roofline": {"kernel": d, "bound": "alu", "achieved": ach, "peak": pk_,
                                      "unit": "TFLOP/s", "frac": ach / pk_,
                                      "algorithmic_flops_per_call": fl[d],
                                      "peak_source": PIPE_SOURCE[pipe],
                                      "eigensolve_frac": _eig_frac(
                                          fl, st, peaks[stage_pipe("lg_tridiag", prec == "mixed", polished, mb.p)])}}
            if "phase_err_rad" in r:
                blk[prec]["phase_err_rad_sampled_row"] = r["phase_err_rad"]
        for kind in ("spin_mixed", "nested_mixed"):
            if kind in mb_res:
                blk[kind] = {"ms_per_call": mb_res[kind]["ms"],
                             "stage_ms": {k: round(v, 3) for k, v in mb_res[kind]["stages"].items()}}
        blk["mixed_over_fp64"] = blk["mixed"]["value"] / blk["fp64"]["value"]
        line["manyband"] = blk
    if sc_res:
        blk = {"workload": "disordered spin-Hall supercells (L x L cells of the 4-band model, n = 4 L^2, "
                           "p = n/2), on-site disorder U[-W/2, W/2] with W = 2, 16 x 16 supercell "
                           f"k-grid, {args.supercell_realisations} seeded realisations per L; plain "
                           "Wilson loop, one CUDA-graph replay per realisation, L2 flushed before each"}
        for Ls in sorted({k[0] for k in sc_res}):
            msc = I.supercell(I.spin_hall(1.0), Ls, W=2.0, seed=0)
            n_, p_ = msc.n, msc.n // 2
            groups = len(np.unique(np.stack([msc.i, msc.j, msc.R[:, 0], msc.R[:, 1], msc.R[:, 2]], 1), axis=0))
            n_ent = len(np.unique(np.stack([msc.i, msc.j], 1), axis=0))
            Kc = 16 * 16
            sub = {"n": n_, "p": p_, "k_points_per_call": Kc}
            for prec in ("mixed", "fp64"):
                r = sc_res[(Ls, prec)]
                calls = len(r["per_call"])
                st = {k: v / calls for k, v in r["stages"].items()}
                polished = "lg_polish" in st
                fl = manyband_stage_flops(n_, p_, 16, 16, groups, prec == "mixed", n_ent, polished)
                fl["loops"] = 16 * 15 * 8.0 * p_ ** 3       # N - 1 products of p x p per loop
                fl["eigenphases"] = 16 * 10.0 * p_ ** 3    # Hessenberg + QR per loop
                d = max((k for k in st if k in fl), key=st.get)
                ach = fl[d] / (st[d] * 1e-3) / 1e12
                pipe = stage_pipe(d, prec == "mixed", polished, p_)
                pk_ = peaks[pipe]
                sub[prec] = {"value": Kc * calls / (r["total_ms"] * 1e-3), "unit": UNIT,
                             "ms_per_call": r["total_ms"] / calls,
                             "per_call_ms": [round(x, 2) for x in r["per_call"]],
                             "stage_ms_per_call": {k: round(v, 2) for k, v in st.items()},
                             "phase_err_rad_sampled_row": r.get("phase_err_rad"),
                             "roofline": {"kernel": d, "bound": "alu", "achieved": ach, "peak": pk_,
                                          "unit": "TFLOP/s", "frac": ach / pk_,
                                          "algorithmic_flops_per_call": fl[d],
                                          "peak_source": PIPE_SOURCE[pipe]}}
            cpu = sc_res.get((Ls, "cpu"))
            if cpu:
                sub["cpu_baseline"] = {"value": cpu["k_points"] / cpu["seconds"], "unit": UNIT,
                                       "cores": os.cpu_count(), "kind": "oracle",
                                       "sample": f"one transverse row (16 of 256 k-points) of realisation 0, "
                                                 f"numpy FP64 with threaded LAPACK, {cpu['seconds']:.2f} s; "
                                                 "the rate is extrapolated to the whole call"}
            sub["mixed_over_fp64"] = sub["mixed"]["value"] / sub["fp64"]["value"]
            blk[f"L{Ls}"] = sub
        line["supercell"] = blk
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(wl, args.cpu_seconds)
    print(json.dumps(line), flush=True)
    return 0


def run_serving(args):
    """Config-4 serving stream through the request server (continuous batching).

    Poisson arrivals (seeded) of Wilson-loop requests on flux-threaded, disordered
    spin-Hall supercells (L from --sides, W ~ U[0, 4], nk x nk grid, p = n/2), each
    submitted at its arrival time; the server admits them as slots and device memory
    free up.  Reports achieved throughput and p50/p99 latency (submit -> results in
    host memory) for the mixed and the FP64 path, and the phase error of sampled
    requests against the oracle.
    """
    import torch
    torch.cuda.set_device(0)
    from paper_2312_13051_gb300 import build as B
    B.build()
    from paper_2312_13051_gb300 import _lib as lib
    from paper_2312_13051_gb300 import inputs as I
    import oracle

    sides = tuple(int(x) for x in args.sides.split(","))
    reqs = I.serving_requests(args.requests, rate=args.rate, sides=sides,
                              nk_range=(args.nk_min, args.nk_max))
    models = [I.serving_model(r) for r in reqs]
    planes = [I.Plane(r["nk"], r["nk"]) for r in reqs]
    clocks = ClockSampler(0)
    out = {}
    clocks.start()
    for prec in ("mixed", "fp64"):
        srv = lib.Server(0, max_slots=args.slots)
        # warm-up: one small request per precision (library load, first launches)
        w = srv.submit(I.spin_hall(1.0), I.Plane(4, 4), 2, prec)
        srv.wait(w)
        done, results = {}, {}
        t0 = time.perf_counter()
        nxt = 0
        while len(done) < len(reqs):
            now = time.perf_counter() - t0
            while nxt < len(reqs) and reqs[nxt]["arrival"] <= now:
                m = models[nxt]
                rid = srv.submit(m, planes[nxt], m.n // 2, prec)
                results[rid] = nxt
                nxt += 1
            for rid, info, ph, gap in srv.poll():
                done[results[rid]] = (info, ph)
            if nxt < len(reqs):
                time.sleep(max(0.0, min(0.002, reqs[nxt]["arrival"] - (time.perf_counter() - t0))))
            else:
                time.sleep(0.0005)
        wall = time.perf_counter() - t0
        srv.close()
        lat = np.array([done[i][0]["latency_ms"] for i in range(len(reqs))])
        ok = [i for i in range(len(reqs)) if done[i][0]["status"] == "OK"]
        kpts = sum(reqs[i]["nk"] ** 2 for i in ok)
        failed = {}
        for i in range(len(reqs)):
            st = done[i][0]["status"]
            if st != "OK":
                failed[st] = failed.get(st, 0) + 1
        out[prec] = dict(wall_s=wall, requests_per_s=len(reqs) / wall, kpoints_per_s=kpts / wall,
                         p50_ms=float(np.percentile(lat, 50)), p99_ms=float(np.percentile(lat, 99)),
                         ok=len(ok), failed=failed,
                         device_ms_sum=float(sum(done[i][0]["device_ms"] for i in range(len(reqs)))))
        # parity on the smallest successful requests (one transverse row each, oracle FP64)
        errs = []
        for i in sorted(ok, key=lambda i: models[i].n * reqs[i]["nk"])[:args.parity_samples]:
            pl = planes[i]
            row = 1 % pl.N_t
            plr = I.Plane(pl.N, 1, origin=tuple(np.array(pl.trans_dir) * row / pl.N_t))
            ref, _ = oracle.wilson_loop(models[i], plr, models[i].n // 2)
            errs.append(oracle.circular_match_error(done[i][1][row], ref[0]))
        out[prec]["phase_err_rad"] = max(errs) if errs else None
        out[prec]["parity_samples"] = len(errs)
    clk = clocks.stop()
    line = {
        "metric": "Wilson-loop serving: k-points/s and p50/p99 latency (submit -> host results)",
        "value": out["mixed"]["kpoints_per_s"], "unit": UNIT, "n_gpus": 1,
        "higher_is_better": True, "dtype": "f32+f64", "data": "synthetic",
        "config": {"workload": "serving stream: flux-threaded disordered spin-Hall supercells",
                   "requests": len(reqs), "rate_per_s": args.rate, "sides": list(sides),
                   "nk_range": [args.nk_min, args.nk_max], "slots": args.slots, "p": "n/2"},
        "mixed": out["mixed"], "fp64": out["fp64"],
        "mixed_over_fp64": out["mixed"]["kpoints_per_s"] / max(out["fp64"]["kpoints_per_s"], 1e-30),
        "clocks": clk,
    }
    print(json.dumps(line), flush=True)
    return 0


def run_profile_case(args):
    """A few uncaptured calls of one workload, for ncu captures (no timing printed)."""
    import torch
    torch.cuda.set_device(0)
    from paper_2312_13051_gb300 import build as B
    B.build()
    from paper_2312_13051_gb300 import _lib as lib
    from paper_2312_13051_gb300 import inputs as I
    ctx = lib.Context(0)
    wl = I.config_bbh()
    case = args.profile_case
    prec = args.profile_precision
    for _ in range(args.warmup):
        if case == "bench":
            lib.nested_wilson_loop(wl.model, wl.plane, wl.p, m=wl.nested_m, precision=prec, ctx=ctx)
        elif case == "saturated":
            lib.wilson_loop(wl.model, I.Plane(60, 3840), wl.p, precision=prec, ctx=ctx)
        elif case == "manyband":
            mb = I.config_manyband(N=24)
            lib.wilson_loop(mb.model, mb.plane, mb.p, precision=prec, ctx=ctx)
        elif case == "supercell":
            m10 = I.supercell(I.spin_hall(1.0), 10, W=2.0, seed=5)
            lib.wilson_loop(m10, I.Plane(16, 16), 200, precision=prec, ctx=ctx)
        elif case == "plaquette":   # past 64 bands: link GEMMs and determinant LU
            lib.plaquette_flux(I.supercell(I.chern_eq4(1.5), 9), I.Plane(6, 5), 81, precision=prec,
                               ctx=ctx)
    torch.cuda.synchronize()
    ctx.status()
    print("profile case done:", case, flush=True)
    return 0


def main(argv=None):
    ap = argparse.ArgumentParser(description=__doc__)
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--cpu-seconds", type=float, default=10.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--serving", action="store_true",
                    help="run the serving stream (request server) instead of the step bench")
    ap.add_argument("--requests", type=int, default=24)
    ap.add_argument("--rate", type=float, default=200.0)
    ap.add_argument("--sides", default="8,12,16")
    ap.add_argument("--nk-min", type=int, default=8)
    ap.add_argument("--nk-max", type=int, default=24)
    ap.add_argument("--slots", type=int, default=4)
    ap.add_argument("--parity-samples", type=int, default=3)
    ap.add_argument("--no-manyband", action="store_true",
                    help="skip the many-band (n = 256) mixed-vs-FP64 measurement")
    ap.add_argument("--manyband-steps", type=int, default=10,
                    help="timed graph replays of the many-band call per precision")
    ap.add_argument("--manyband-kinds", default="wilson",
                    help="comma list of many-band loops to time: wilson (always), spin, nested")
    ap.add_argument("--profile-precision", choices=["mixed", "fp64"], default="mixed",
                    help="precision of the --profile-case calls")
    ap.add_argument("--no-supercell", action="store_true",
                    help="skip the disordered-supercell block (config 2)")
    ap.add_argument("--supercell-sides", default="10",
                    help="supercell sides L of the disordered-supercell block (n = 4 L^2)")
    ap.add_argument("--supercell-realisations", type=int, default=4)
    ap.add_argument("--no-saturated", action="store_true",
                    help="skip the saturated-batch measurement (230 400 k-points per call)")
    ap.add_argument("--profile-case", choices=["bench", "saturated", "manyband", "supercell", "plaquette"],
                    help="run --warmup uncaptured calls of one workload and exit (for ncu)")
    args = ap.parse_args(argv)
    if args.warmup < 3:
        log("warmup raised to 3")
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    if args.serving:
        return run_serving(args)
    if args.profile_case:
        return run_profile_case(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())

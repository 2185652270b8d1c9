#!/usr/bin/env python
"""Benchmark: grid points per second of the 3D Helmholtz inverse at 256^3.

Workload: 256^3 cell grid on [0,1]^3, tanh stretching factor 1.5 in every
direction, Dirichlet walls, lambda = dt/Re = 1e3/1000 = 1, eigen transforms in
x and y with the Thomas algorithm along z (TPT), right-hand side i.i.d.
uniform[-1, 1] (seed 0 + rank).  One step = one complete solve
(I - lambda*Delta) u = f to the path's residual tolerance, including every
refinement step and the final residual check.

Arms: the plain FP64 path (tolerance 1e-11) and, when available, the mixed
path (split tensor-core transforms, tolerance 1e-10).  `value` is the faster
arm that met its tolerance.  The field is 134 MB and the working set several
times larger than the 129 MB L2, so no extra L2 flush is needed between steps.

Multi-GPU: the solves are independent problems, so N GPUs run N replicas
("scaling": "weak"), one per rank, with no data-path collective; value is the
points solved by all ranks divided by the slowest rank's time.

`--impl reference` times the FP64 CPU oracle (NumPy TPT) on the host cores on
the same workload instead.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import workloads  # noqa: E402

N_DEFAULT = 256
BETA = 1.5
LAM = 1e3 / 1000.0
METRIC = "grid-pts/s per Helmholtz solve at 256^3"
FP64_PEAK_GFLOPS = 152 * 2 * 2 * 2.07  # SMs x FP64 FMA/clk/SM x 2 flop x GHz (about 1.26 TFLOP/s)


def load_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return json.load(fh), "measured"
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}, "fallback"


def dram_traffic(kernel):
    """DRAM bytes per launch of `kernel` from the committed ncu summary
    (profiles/dram_traffic_256cube.json), or None when there is no entry or the
    kernel's sources changed since the counters were taken."""
    try:
        with open(os.path.join(ROOT, "profiles", "dram_traffic_256cube.json")) as fh:
            table = json.load(fh)
        e = table[kernel]
        h = hashlib.sha256()
        for f in e["sources"]:
            with open(os.path.join(ROOT, "paper_1107_2461_gb300", "csrc", f), "rb") as fh:
                h.update(fh.read())
        if h.hexdigest() != e["sha256"]:
            return None
        return float(e["dram_read_bytes"] + e["dram_write_bytes"])
    except Exception:
        return None


class ClockSampler:
    """nvidia-smi clock / throttle sampling during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "25"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def slowest_rank(values, device, world):
    """Element-wise maximum of per-rank timings over all ranks (the job's time
    is its slowest replica's); identity on one rank."""
    import torch
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    if world > 1:
        import torch.distributed as dist
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t]


def whole_job_rate(world, points, steps, seconds):
    """Whole-job throughput of `world` replicas that each solved `steps`
    problems of `points` grid points in (at most) `seconds`."""
    return world * points * steps / seconds


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def oracle_tpt_time(n, seed=0):
    """Time one FP64 oracle TPT solve (NumPy) on the host cores."""
    from oracle import assembled as asm
    from oracle import decomposition as dec
    faces = workloads.box_faces(n, BETA)
    ops = asm.cell_ops(faces, (0, 0, 0), (0, 0, 0))
    f = workloads.rhs_uniform(n[::-1], seed)
    t0 = time.perf_counter()
    dec.tpt_solve(f, ops, LAM)
    return time.perf_counter() - t0


def oracle_tpt_time_one_thread(n, timeout=180):
    """The same oracle solve in a child process limited to one BLAS / OpenMP
    thread (seconds; None if it could not be timed)."""
    env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1")
    code = f"import sys; sys.path.insert(0, {ROOT!r}); import bench; print(bench.oracle_tpt_time({tuple(n)!r}))"
    try:
        out = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=timeout)
        return float(out.stdout.strip().splitlines()[-1])
    except Exception:
        return None


def blas_threads():
    try:
        from threadpoolctl import threadpool_info
        info = threadpool_info()
        if info:
            return max(int(i.get("num_threads", 1)) for i in info)
    except Exception:
        pass
    return os.cpu_count() or 1


def kernel_model(name, n, steps, K):
    """(bound, algorithmic units per launch, unit kind, useful launches in K solves).

    Algorithmic work: a transform along direction d costs 36 digit products = 72
    n_d flop per point (FP64 path) or 3 split products = 6 n_d flop per point
    (mixed path) on the tensor cores; the bytes are one read of the input and one write of the
    output field (FP32 intermediates, FP64 user arrays, 8-byte double-float
    solution).  Refinement rounds after convergence return at once and are not
    counted as useful launches."""
    P = float(n[0] * n[1] * n[2])
    rounds = 1 + steps
    t = {
        # FP64 path: fwd and back transform of a direction share a name (digit
        # products on the tensor cores, FP64 fields in and out)
        "transform_x_f64": ("hbm", 16.0 * P, "byte", 2 * rounds * K),
        "transform_y_f64": ("hbm", 16.0 * P, "byte", 2 * rounds * K),
        "thomas_z_f64": ("hbm", 16.0 * P, "byte", rounds * K),
        "residual_f64": ("hbm", 24.0 * P, "byte", rounds * K),
        # mixed path (bytes; the tensor flops are reported beside them)
        "transform_xf_tc": ("hbm", 8.0 * P, "byte", rounds * K),
        "transform_yf_tc": ("hbm", 8.0 * P, "byte", rounds * K),
        "transform_yb_tc": ("hbm", 8.0 * P, "byte", rounds * K),
        "transform_xb_set_tc": ("hbm", 8.0 * P, "byte", K),
        "transform_xb_corr_tc": ("hbm", 8.0 * P, "byte", min(steps, 1) * K),
        "transform_xb_add_tc": ("hbm", 12.0 * P, "byte", max(steps - 1, 0) * K),
        "thomas_z_f32": ("hbm", 8.0 * P, "byte", rounds * K),
        # first check r_1 = b - A H: H and b read, r_1 written as two FP32 planes
        "residual_df": ("hbm", 20.0 * P, "byte", K),
        # later checks r = r_1 - A L: r_1 planes, L and H read, r and the FP64 output written
        "residual_corr": ("hbm", 28.0 * P, "byte", steps * K),
        "residual_df_init": ("hbm", 12.0 * P, "byte", K),
        # converts the output only when no refinement round ran
        "finalize_out": ("hbm", 12.0 * P, "byte", K if steps == 0 else 0),
    }
    return t.get(name)


def tensor_flops(name, n):
    P = float(n[0] * n[1] * n[2])
    d = {"x": 0, "y": 1, "z": 2}.get(name[len("transform_"):][:1], 1)
    if name in ("transform_x_f64", "transform_y_f64"):
        return 72.0 * P * n[d]  # 36 digit products
    return 6.0 * P * n[d] if name.endswith("_tc") else None


def run_arm(fdi, torch, prec, n, K, W, dev, rank, stream, thomas_axis=2, refine_tol=None, thomas_config=None):
    faces = workloads.box_faces(n, BETA)
    plan = fdi.plan_create(faces, n, prec=prec, thomas_axis=thomas_axis)
    if thomas_config is not None and prec != fdi.PREC_FP64:
        fdi.set_thomas_config(plan, thomas_config)
    if refine_tol is not None:
        plan.set_tolerances(refine_tol, 3)
    f = workloads.rhs_uniform(n[::-1], rank)
    rhs = torch.from_numpy(f).to(dev)
    out = torch.empty_like(rhs)
    with torch.cuda.stream(stream):
        for _ in range(W):
            fdi.helmholtz_solve(plan, LAM, rhs, out, stream)
    torch.cuda.synchronize()
    _, steps, rel, st = fdi.last_result(plan)
    launches_per = fdi.last_launch_count(plan)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    if torch.distributed.is_initialized():
        torch.distributed.barrier()
    torch.cuda.synchronize()
    with ClockSampler(torch.cuda.current_device()) as clk:
        e0.record(stream)
        for _ in range(K):
            fdi.helmholtz_solve(plan, LAM, rhs, out, stream)
        e1.record(stream)
        torch.cuda.synchronize()
    if torch.distributed.is_initialized():
        torch.distributed.barrier()
    ms = e0.elapsed_time(e1)
    _, steps, rel, st = fdi.last_result(plan)
    # per-kernel times from a separate pass with CUDA events around every launch
    # (kept out of the timed region above: the events add gaps between kernels)
    fdi.enable_timing(plan, True)
    fdi.reset_kernel_times(plan)
    with torch.cuda.stream(stream):
        for _ in range(K):
            fdi.helmholtz_solve(plan, LAM, rhs, out, stream)
    torch.cuda.synchronize()
    ktimes = fdi.kernel_times(plan)
    fdi.enable_timing(plan, False)
    # end to end through the C ABI with host buffers (fdi_field_solve_host):
    # every step copies its right-hand side from pinned host memory to the
    # device and its solution back; the library pipelines the copies of
    # neighbouring steps with the solves.  Two distinct right-hand sides and
    # two result arrays alternate.
    h_in = [torch.from_numpy(f).pin_memory(),
            torch.from_numpy(workloads.rhs_uniform(n[::-1], rank + 1000)).pin_memory()]
    h_out = [torch.empty(h_in[0].shape, dtype=torch.float64).pin_memory() for _ in range(2)]
    rhs_seq = [h_in[i % 2] for i in range(K)]
    out_seq = [h_out[i % 2] for i in range(K)]
    fdi.field_solve_host(plan, fdi.FIELD_CELL, 1.0, LAM, rhs_seq[:4], out_seq[:4], stream)  # warm-up
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    rel_host = fdi.field_solve_host(plan, fdi.FIELD_CELL, 1.0, LAM, rhs_seq, out_seq, stream)
    e2e_s = time.perf_counter() - t0
    # the same without overlap: copy in, solve, copy out, one step after another
    d_in = torch.empty_like(rhs)
    d_out = torch.empty_like(rhs)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    with torch.cuda.stream(stream):
        for i in range(K):
            d_in.copy_(h_in[i % 2], non_blocking=True)
            fdi.helmholtz_solve(plan, LAM, d_in, d_out, stream)
            h_out[i % 2].copy_(d_out, non_blocking=True)
    stream.synchronize()
    e2e_serial_s = time.perf_counter() - t0
    plan.destroy()
    return {"ms": ms, "steps": steps, "rel": rel, "status": st, "ktimes": ktimes, "launches_per": launches_per,
            "e2e_s": e2e_s, "e2e_serial_s": e2e_serial_s, "e2e_max_rel": max(rel_host), "h2d": f.nbytes,
            "d2h": f.nbytes, "clocks": clk.summary()}


def run_stokes(fdi, torch, prec, n, reps, warm, stream, krylov=0, resident=False):
    """Stokes-inverse latency on the staggered n^3 no-slip box (tanh 1.5, Re 1000,
    dt in {1e-2, 1e3}, Gaussian forcing seeds 0-2): p50 / p99 of the wall time of
    complete solves (each call ends with the stream synchronised).  resident:
    the Helmholtz solves as resident launches (fdi_plan_set_resident)."""
    faces = workloads.box_faces((n, n, n), BETA)
    plan = fdi.plan_create(faces, (n, n, n), grid=fdi.GRID_MAC, prec=prec)
    fdi.set_krylov(plan, krylov)
    fdi.set_resident(plan, resident)
    shapes = workloads.mac_shapes((n, n, n))
    f = [torch.from_numpy(workloads.rhs_gaussian(shapes[c], i)).cuda() for i, c in enumerate("uvw")]
    u = [torch.empty_like(t) for t in f]
    p = torch.empty(shapes["p"], dtype=torch.float64, device="cuda")
    out = {}
    for dt in (1e-2, 1e3):
        for _ in range(warm):
            fdi.stokes_solve(plan, dt, 1000.0, f, u, p, stream)
        stream.synchronize()
        lat = []
        for _ in range(reps):
            t0 = time.perf_counter()
            fdi.stokes_solve(plan, dt, 1000.0, f, u, p, stream)
            stream.synchronize()
            lat.append(1e3 * (time.perf_counter() - t0))
        it, _, rel, st = fdi.last_result(plan)
        lat.sort()
        out[f"dt={dt:g}"] = {"p50_ms": lat[len(lat) // 2], "p99_ms": lat[min(len(lat) - 1, int(0.99 * len(lat)))],
                             "krylov_iters": it, "rel_residual": rel, "status": st, "reps": reps,
                             "launches_per_solve": fdi.last_launch_count(plan)}
    plan.destroy()
    return out


def run_batch(fdi, torch, prec, count, reps, stream):
    """Batched Helmholtz solves over uneven stretched grids (shapes from
    {32..160} with aspect up to 1:4, beta ~ U[1,2], lambda log-uniform in
    [1e-4, 1], seed 0; RHS seeds 1..count): grid-points/s of whole batches
    (concurrent plans, one graph launch per batch after the first two calls)."""
    probs = workloads.mixed_shape_batch(count, 0)
    plans, lams, rhs, outs = [], [], [], []
    for q, (nn, beta, lam) in enumerate(probs):
        faces = [workloads.tanh_faces(nn[d], beta) for d in range(3)]
        plans.append(fdi.plan_create(faces, nn, prec=prec))
        rhs.append(torch.from_numpy(workloads.rhs_uniform(nn[::-1], q + 1)).cuda())
        outs.append(torch.empty_like(rhs[-1]))
        lams.append(lam)
    pts = float(sum(np.prod(nn) for nn, _, _ in probs))
    with torch.cuda.stream(stream):
        for _ in range(3):
            fdi.helmholtz_solve_batched(plans, lams, rhs, outs, stream)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    with torch.cuda.stream(stream):
        for _ in range(reps):
            fdi.helmholtz_solve_batched(plans, lams, rhs, outs, stream)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / reps
    worst = max(fdi.last_result(pl)[2] for pl in plans)
    ok = all(fdi.last_result(pl)[3] == 0 for pl in plans)
    for pl in plans:
        pl.destroy()
    return {"value": pts / (ms * 1e-3), "unit": "grid-pts/s", "ms_per_batch": ms, "solves": count,
            "points": pts, "worst_rel_residual": worst, "all_converged": ok, "reps": reps}


def pct(v, q):
    v = sorted(v)
    return v[min(len(v) - 1, int(q * len(v)))] if v else None


def run_serving(fdi, torch, prec, count, rate_hz, max_n, slots):
    """Serving trace: Poisson arrivals (rate_hz, seed 0) of Stokes-inverse
    requests on stretched no-slip boxes (beta 1.5), cubic n uniform over
    {48, 64, 96, 128, 160, 192, 256} up to max_n, dt log-uniform in [1e-2, 1e3],
    Re in {100, 1000, 5000}; pinned host arrays in and out, submitted at their
    arrival times into a server with `slots` workers and a 160 GB device budget.
    Host memory stays bounded: the Gaussian forcing is one seeded set per grid
    size, shared read-only by that size's requests, and the outputs come from a
    pool of buffers per size; a request whose pool buffer is still held by an
    unfinished request waits for it before submission (counted).  Reported:
    end-to-end latency (arrival to completion), queueing delay (arrival to
    start) and service latency (start to completion), overall and per size,
    and the completion rate over the trace (the sustainable rate when the
    arrivals exceed it)."""
    rng = np.random.default_rng(0)
    sizes = [v for v in (48, 64, 96, 128, 160, 192, 256) if v <= max_n]
    arrivals = workloads.poisson_arrivals(count, rate_hz, 0)
    draws = [(int(rng.choice(sizes)), float(10.0 ** rng.uniform(-2.0, 3.0)), float(rng.choice([100.0, 1000.0, 5000.0])))
             for _ in range(count)]
    pool_len = {256: 6, 192: 8, 160: 12, 128: 16}
    forcing, pools, owner, used = {}, {}, {}, {}

    def pinned(shape, src=None):
        # page-locked host array (a client next to the GPU keeps its buffers
        # pinned, so the request copies run at the host link's rate)
        t = torch.empty(tuple(shape), dtype=torch.float64, pin_memory=True)
        a = t.numpy()
        a[...] = 0.0 if src is None else src
        keep.append(t)
        return a

    keep = []
    for nn in sorted({d[0] for d in draws}):
        sh = workloads.mac_shapes((nn, nn, nn))
        forcing[nn] = [pinned(sh[c], workloads.rhs_gaussian(sh[c], 1000 * nn + i)) for i, c in enumerate("uvw")]
        pools[nn] = [([pinned(sh[c]) for c in "uvw"], pinned(sh["p"])) for _ in range(pool_len.get(nn, 32))]
        used[nn] = 0
    srv = fdi.Server(160 << 30, slots)
    t0 = time.perf_counter()
    tickets, waits = [], 0
    for q, (nn, dt, Re) in enumerate(draws):
        wait = arrivals[q] - (time.perf_counter() - t0)
        if wait > 0:
            time.sleep(wait)
        k = used[nn] % len(pools[nn])
        used[nn] += 1
        prev = owner.get((nn, k))
        if prev is not None and srv.poll(prev)["state"] != 2:
            srv.poll(prev, wait=True)
            waits += 1
        u, p = pools[nn][k]
        t = srv.submit((nn, nn, nn), 1.5, dt, Re, forcing[nn], u, p, prec=prec)
        owner[(nn, k)] = t
        tickets.append(t)
    srv.drain()
    wall = time.perf_counter() - t0
    res = [srv.poll(t) for t in tickets]
    st = srv.stats()
    srv.close()
    lat = [r["latency_ms"] for r in res]
    que = [r["queue_ms"] for r in res]
    svc = [r["latency_ms"] - r["queue_ms"] for r in res]
    per = {}
    for nn in sorted(forcing):
        s_n = [svc[q] for q in range(count) if draws[q][0] == nn]
        per[f"{nn}^3"] = {"requests": len(s_n), "service_p50_ms": pct(s_n, 0.5), "service_p99_ms": pct(s_n, 0.99)}
    return {"completed": st["completed"], "all_converged": all(r["status"] == 0 for r in res),
            "worst_rel_residual": max(r["rel_residual"] for r in res),
            "latency_p50_ms": pct(lat, 0.5), "latency_p99_ms": pct(lat, 0.99),
            "queue_p50_ms": pct(que, 0.5), "queue_p99_ms": pct(que, 0.99),
            "service_p50_ms": pct(svc, 0.5), "service_p99_ms": pct(svc, 0.99),
            "completion_rate_rps": st["throughput_rps"], "offered_rate_rps": rate_hz, "trace_s": wall,
            "submissions_waiting_for_a_buffer": waits, "per_size": per, "plans_created": st["plans_created"],
            "peak_gb": st["peak_bytes"] / 1e9}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="fdi", choices=["fdi", "reference"])
    ap.add_argument("--n", type=int, default=N_DEFAULT)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--arms", default="fp64,mixed")
    ap.add_argument("--no-tpf", action="store_true", help="skip the FP64 TPF arm")
    ap.add_argument("--no-fp64tol", action="store_true", help="skip the mixed arm refined to 1e-11")
    ap.add_argument("--stokes-n", type=int, default=64, help="Stokes latency grid (0: skip)")
    ap.add_argument("--stokes-reps", type=int, default=10)
    ap.add_argument("--batch", type=int, default=64, help="batched uneven-grid solves per batch (0: skip)")
    ap.add_argument("--serve", type=int, default=2000, help="serving-trace requests, mixed precision (0: skip)")
    ap.add_argument("--serve-fp64", type=int, default=60,
                    help="serving-trace requests of the FP64 arm (the first ones of the same trace; 0: skip)")
    ap.add_argument("--serve-max-n", type=int, default=256, help="largest cubic grid in the serving trace")
    ap.add_argument("--serve-slots", type=int, default=4)
    ap.add_argument("--thomas-config", type=int, default=None,
                    help="FP32 Thomas configuration of the mixed arms (fdi_plan_set_thomas_config)")
    args = ap.parse_args()
    n = (args.n, args.n, args.n)
    P = n[0] * n[1] * n[2]
    K, W = args.steps, max(args.warmup, 3)
    rank, world, local = dist_env()
    workload = {"workload": f"helmholtz_tpt_{args.n}^3_tanh{BETA}_dirichlet_lambda{LAM:g}", "n": list(n),
                "beta": BETA, "lambda": LAM, "bc": "dirichlet", "method": "TPT (eigen x,y; Thomas z)",
                "rhs": "uniform[-1,1] seed 0+rank", "l2": "inputs+workspace larger than L2 (134 MB field)"}

    if args.impl == "reference":
        if rank != 0:
            return 0
        os.environ.setdefault("OMP_NUM_THREADS", str(os.cpu_count() or 1))
        # W untimed warm-up solves (the first pays for page faults and BLAS
        # start-up), within a minute
        t, t_warm = [], time.perf_counter()
        for _ in range(W):
            t.append(oracle_tpt_time(n))
            if time.perf_counter() - t_warm > 60.0:
                break
        times = []
        budget = 150.0
        t_start = time.perf_counter()
        for k in range(K):
            times.append(oracle_tpt_time(n, seed=k))
            if time.perf_counter() - t_start > budget:
                break
        v = P * len(times) / sum(times)
        line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "grid-pts/s", "n_gpus": args.gpus,
                "steps": len(times), "warmup": len(t), "ms_per_step": 1e3 * sum(times) / len(times),
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
                "data": "synthetic", "config": workload,
                "cpu_baseline": {"value": v, "unit": "grid-pts/s", "cores": blas_threads(), "kind": "oracle",
                                 "sample": f"{len(times)} full {args.n}^3 TPT solves by the NumPy FP64 oracle"},
                "e2e": {"value": v, "unit": "grid-pts/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(line))
        return 0

    import torch
    import torch.distributed as dist
    if world > 1:
        dist.init_process_group("nccl", init_method="env://")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    from paper_1107_2461_gb300 import build as _b
    _b.build()
    import paper_1107_2461_gb300 as fdi
    stream = torch.cuda.Stream()

    arms = {}
    precs = {"fp64": (fdi.PREC_FP64, 1e-11), "mixed": (fdi.PREC_MIXED_F16, 1e-10)}
    # the TPF variant (eigen transforms in all three directions, Eq. 29) runs on the FP64 path
    # mixed_fp64tol: the mixed path refined to the FP64 path's tolerance
    helm_arms = {"fp64": (fdi.PREC_FP64, 1e-11, 2), "mixed": (fdi.PREC_MIXED_F16, 1e-10, 2),
                 "fp64_tpf": (fdi.PREC_FP64, 1e-11, -1), "mixed_tpf": (fdi.PREC_MIXED_F16, 1e-10, -1),
                 "mixed_fp64tol": (fdi.PREC_MIXED_F16, 1e-11, 2)}
    helm_names = args.arms.split(",")
    if not args.no_tpf:
        helm_names += [a + "_tpf" for a in ("fp64", "mixed") if a in helm_names]
    if "mixed" in helm_names and not args.no_fp64tol:
        helm_names.append("mixed_fp64tol")
    for name in helm_names:
        prec, tol, taxis = helm_arms[name]
        try:
            slow = name == "fp64_tpf"  # FP64-pipe bound: fewer solves
            arms[name] = run_arm(fdi, torch, prec, n, max(3, K // 10) if slow else K, W, dev, rank, stream,
                                 thomas_axis=taxis, thomas_config=args.thomas_config,
                                 refine_tol=tol if name == "mixed_fp64tol" else None)
            if slow:
                arms[name]["K"] = max(3, K // 10)
            arms[name]["tol"] = tol
            arms[name]["prec"] = prec
        except fdi.FdiError as e:
            if e.status == fdi.fdi.ERR_UNSUPPORTED:
                continue
            raise
    # slowest rank
    for a in arms.values():
        a["ms_max"], a["e2e_max"], a["e2e_serial_max"] = slowest_rank([a["ms"], a["e2e_s"], a["e2e_serial_s"]],
                                                                      dev, world)
        a["value"] = whole_job_rate(world, P, a.get("K", K), a["ms_max"] * 1e-3)
        a["ok"] = a["status"] == 0 and a["rel"] <= a["tol"]
    best_name = max((k for k in arms if arms[k]["ok"]), key=lambda k: arms[k]["value"], default=None)
    if best_name is None:
        best_name = next(iter(arms))
    best = arms[best_name]

    # roofline of the dominant kernel of the reported arm
    peaks, peak_kind = load_peaks()
    roof = None
    per_kernel = {}
    for name, (tot_ms, cnt) in best["ktimes"].items():
        km = kernel_model(name, n, best["steps"], K)
        if km is None:
            continue
        bound, units, kind, useful = km
        if useful <= 0:
            continue  # launched but returned at once
        useful = max(1, min(cnt, useful))
        avg_s = tot_ms * 1e-3 / useful
        if kind == "flop":
            achieved, peak, unit = units / avg_s / 1e9, FP64_PEAK_GFLOPS, "GFLOP/s"
            src = "FP64 pipe: 152 SMs x 2 FMA/clk x 2 flop x 2.07 GHz (derived)"
        else:
            achieved, peak, unit = units / avg_s / 1e9, peaks["hbm_gbs"], "GB/s"
            src = f"MEASURED_PEAKS.json hbm_gbs ({peak_kind})"
        e = {"kernel": name, "bound": bound, "achieved": achieved, "peak": peak, "unit": unit,
             "frac": achieved / peak, "traffic": None, "avg_launch_ms": tot_ms / useful, "launches": useful,
             "total_ms": tot_ms, "peak_source": src}
        tf = tensor_flops(name, n)
        if tf is not None:
            e["tensor_tflops"] = tf / avg_s / 1e12
            e["tensor_frac"] = e["tensor_tflops"] / peaks["bf16_tflops"]
            e["tensor_peak_source"] = "MEASURED_PEAKS.json bf16_tflops (fp16 dense rate = bf16 rate)"
        per_kernel[name] = e
    if per_kernel:
        # the transform roles are launches of one kernel (k_tc_transform, as
        # the ncu launch list counts it): grouped when choosing the dominant one
        cand = {k: e for k, e in per_kernel.items() if not k.endswith("_tc")}
        tc = [e for k, e in per_kernel.items() if k.endswith("_tc")]
        if tc:
            tot_ms = sum(e["total_ms"] for e in tc)
            launches = sum(e["launches"] for e in tc)
            work = sum(e["achieved"] * 1e9 * e["avg_launch_ms"] * 1e-3 * e["launches"] for e in tc)
            g = {"kernel": "k_tc_transform", "roles": sorted(k for k in per_kernel if k.endswith("_tc")),
                 "bound": "hbm", "achieved": work / (tot_ms * 1e-3) / 1e9, "peak": tc[0]["peak"], "unit": "GB/s",
                 "traffic": None, "avg_launch_ms": tot_ms / launches, "launches": launches, "total_ms": tot_ms,
                 "peak_source": tc[0]["peak_source"]}
            g["frac"] = g["achieved"] / g["peak"]
            tfl = sum(e.get("tensor_tflops", 0.0) * 1e12 * e["avg_launch_ms"] * 1e-3 * e["launches"] for e in tc)
            g["tensor_tflops"] = tfl / (tot_ms * 1e-3) / 1e12
            g["tensor_frac"] = g["tensor_tflops"] / peaks["bf16_tflops"]
            g["tensor_peak_source"] = tc[0].get("tensor_peak_source")
            cand["k_tc_transform"] = g
        roof = dict(max(cand.values(), key=lambda e: e["total_ms"]))
        if tuple(n) == (256, 256, 256):
            if roof["kernel"] == "k_tc_transform":
                tr = [dram_traffic(k) for k in roof["roles"]]
                tr = [t for t in tr if t is not None]
                roof["traffic"] = sum(tr) / len(tr) if tr else None
            else:
                roof["traffic"] = dram_traffic(roof["kernel"])
    stokes = None
    if args.stokes_n > 0:
        stokes = {}
        for name in args.arms.split(","):
            prec = precs[name][0]
            variants = [("", 0, False), ("/bicgstab2", 1, False), ("/cg", 2, False)]
            if prec != fdi.PREC_FP64:
                variants += [("/resident", 0, True), ("/cg/resident", 2, True)]
            for kname, kry, res in variants:
                try:
                    stokes[name + kname] = run_stokes(fdi, torch, prec, args.stokes_n, args.stokes_reps, 2, stream,
                                                      krylov=kry, resident=res)
                except fdi.FdiError as e:
                    stokes[name + kname] = {"error": str(e)}
    batch = None
    if args.batch > 0:
        batch = {"config": f"{args.batch} Helmholtz solves, grids from {{32,48,64,96,128,160}}^3 with aspect <= 4, "
                           "beta ~ U[1,2], lambda log-uniform [1e-4, 1], seed 0"}
        for name in args.arms.split(","):
            try:
                batch[name] = run_batch(fdi, torch, precs[name][0], args.batch, 5, stream)
            except fdi.FdiError as e:
                batch[name] = {"error": str(e)}
    serving = None
    if args.serve > 0:
        serving = {"config": f"Stokes-inverse requests ({args.serve} mixed, the first {args.serve_fp64} of the "
                             f"same trace FP64), Poisson arrivals at 200/s (seed 0), cubic n from {{48..256}} up to "
                             f"{args.serve_max_n}, dt log-uniform [1e-2,1e3], Re in {{100,1000,5000}}, beta 1.5, "
                             f"{args.serve_slots} slots, 160 GB budget, tolerance 1e-10 (mixed) / 1e-11 (FP64)"}
        for name in args.arms.split(","):
            count = args.serve if name == "mixed" else args.serve_fp64
            if count <= 0:
                continue
            try:
                serving[name] = run_serving(fdi, torch, precs[name][0], count, 200.0, args.serve_max_n,
                                            args.serve_slots)
            except fdi.FdiError as e:
                serving[name] = {"error": str(e)}
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        t = oracle_tpt_time(n)
        t1 = oracle_tpt_time_one_thread(n)
        cpu = {"value": P / t, "unit": "grid-pts/s", "cores": blas_threads(), "kind": "oracle",
               "sample": f"one full {args.n}^3 TPT solve by the NumPy FP64 oracle ({t:.2f} s)",
               "one_thread": ({"value": P / t1, "seconds": t1} if t1 else None)}
    if rank != 0:
        return 0
    line = {
        "metric": METRIC, "value": best["value"], "unit": "grid-pts/s", "n_gpus": world, "steps": K, "warmup": W,
        "ms_per_step": best["ms_max"] / best.get("K", K), "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f64" if best_name == "fp64" else "f16-split/f32-acc + f64 refinement",
        "data": "synthetic", "config": dict(workload, arm=best_name, parallelism=f"replicas x{world}"),
        "e2e": {"value": whole_job_rate(world, P, best.get("K", K), best["e2e_max"]), "unit": "grid-pts/s",
                "h2d_bytes_per_step": best["h2d"], "d2h_bytes_per_step": best["d2h"],
                "api": "fdi_field_solve_host (host FP64 arrays in and out, copies pipelined with the solves)",
                "max_rel_residual": best["e2e_max_rel"],
                "serial_value": whole_job_rate(world, P, best.get("K", K), best["e2e_serial_max"]),
                "serial": "copy in, solve, copy out per step on one stream, no overlap"},
        "gpu_launches": best["launches_per"] * K,
        "roofline": roof,
        "cpu_baseline": cpu,
        "clocks": best["clocks"],
        "stokes_latency": ({"config": f"MAC {args.stokes_n}^3, tanh {BETA}, no-slip, Re 1000, Gaussian forcing; "
                                      "BiCGstab (default), BiCGstab(2) (/bicgstab2; iterations are outer ones) and "
                                      "volume-weighted CG (/cg; one C-product per iteration); /resident: the "
                                      "Helmholtz solves as resident launches (one cooperative launch per solve, "
                                      "the three velocity solves sharing one)",
                            **stokes} if stokes is not None else None),
        "batched": batch,
        "serving": serving,
        "kernels": {k: {kk: round(vv, 4) if isinstance(vv, float) else vv for kk, vv in e.items()
                        if kk in ("achieved", "unit", "frac", "avg_launch_ms", "launches", "tensor_frac")}
                    for k, e in per_kernel.items()},
        "arms": {k: {"value": a["value"], "ms_per_solve": a["ms_max"] / a.get("K", K), "rel_residual": a["rel"],
                     "refine_steps": a["steps"], "tol": a["tol"], "met_tol": a["ok"],
                     "kernels": {kn: {"ms_total": v[0], "launches": v[1]} for kn, v in a["ktimes"].items()}}
                 for k, a in arms.items()},
    }
    print(json.dumps(line))
    if world > 1:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())

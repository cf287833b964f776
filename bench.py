"""Benchmark: sustained CG Gflops of the mixed-precision domain-wall solve on GB300.

Workload: one full solve D psi = eta on a 16^3 x 32 lattice, Ns = 16, weights
omega_s = sigma_s = 1 + 0.5 cos(pi (s - 1/2) / Ns), m0 = 1.8, mq = 0.02, links exp(0.5 i H)
(seed 2), complex Gaussian source (seed 2); FP32 inner CG with FP64 reliable updates to a
true relative residual of 1e-10.  One step = one whole solve (source preparation, inner
CG, FP64 restarts, reconstruction, final FP64 residual check).

value: counted flops (fixed per-site counts) / device time, inputs resident in HBM.
e2e:   the same metric through dwf_solve with pinned host buffers (H2D of eta and D2H of
       psi inside the timed region).
The working set (~1.5 GB) is larger than L2, so no flush is needed between steps.

--impl reference times the FP64 CPU oracle on this machine's host cores instead (one
C C^dagger application on the same lattice per step: a bounded sample of the workload).
Multi-GPU (torchrun): every rank solves its own replica (no data-path collective);
value = all ranks' flops / max time over ranks.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

DIMS, NS, M0, MQ, EPS, SEED = (16, 16, 16, 32), 16, 1.8, 0.02, 0.5, 2
WORKLOAD = "dwf_full_solve_16x16x16x32_Ns16_cosine_mq0.02_tol1e-10"
METRIC = "CG Gflops & % HBM roofline (16^3x32,Ns16); served solves/s, p99 latency"
PAPER_BEST_GFLOPS = 233.0  # GTX 480, CG (mixed), same lattice (Table 1): other hardware, context

# ncu DRAM traffic (dram__bytes_read.sum + dram__bytes_write.sum) per launch, bytes, of the
# FP32 kernel classes at this workload, from one ncu capture of the kernels as they stand
# (summarised under profiles/).  Valid only for the kernel source it was captured on: empty
# (traffic reported as null) until the kernels are captured again after a change.
NCU_TRAFFIC = {"hop_m5": 152075008 + 70445312, "hop_xpay": 252933120 + 74510848,
               "hop_update": 353506304 + 76856064, "smix_p": 302014976 + 238914816}


def flops_ccdag(n, ns):
    return n * (5232.0 + 192.0 * ns)


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if not self.proc:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
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
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None, "reasons": sorted(reasons),
                "samples": len(sm)}


def aggregate_over_ranks(ms, flops, device=None):
    """Whole-job numbers of independent replicas: the slowest rank's time and the sum of the
    work of all ranks (no data-path collective; only these two scalars are reduced)."""
    import torch
    import torch.distributed as tdist
    if not (tdist.is_available() and tdist.is_initialized()) or tdist.get_world_size() == 1:
        return ms, flops
    t = torch.tensor([float(ms)], dtype=torch.float64, device=device)
    f = torch.tensor([float(flops)], dtype=torch.float64, device=device)
    tdist.all_reduce(t, op=tdist.ReduceOp.MAX)
    tdist.all_reduce(f, op=tdist.ReduceOp.SUM)
    return float(t.item()), float(f.item())


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def host_cores():
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


def _oracle_replica(dims, ns, warmup, reps, barrier, q):
    """One host core: the oracle's FP64 C C^dagger on its own copy of the workload's input."""
    import oracle
    from paper_1101_0423_gb300 import inputs
    om, sg = inputs.weights("cosine", ns)
    U = inputs.gauge_field(dims, EPS, seed=SEED)
    x = inputs.gaussian_source(dims, ns, seed=SEED, parity=1)
    mp, mm = oracle.m5(ns, M0, MQ, om, sg)
    for _ in range(warmup):
        oracle.ccdag_op(dims, ns, U, mp, mm, 1, x)
    barrier.wait()
    t0 = time.perf_counter()
    for _ in range(reps):
        oracle.ccdag_op(dims, ns, U, mp, mm, 1, x)
    q.put((t0, time.perf_counter()))


def oracle_on_all_cores(dims, ns, warmup, reps, cores=None):
    """The oracle as it stands, one process per host core (spawned: no state shared with a
    CUDA context), each applying C C^dagger to its own input; all start together behind a
    barrier.  Returns (aggregate GFLOP/s, wall seconds of the timed region, cores)."""
    import multiprocessing as mp_
    import oracle
    oracle.build()
    cores = cores or host_cores()
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ[k] = "1"  # one thread per replica, inherited by the spawned processes
    ctx = mp_.get_context("spawn")
    barrier, q = ctx.Barrier(cores), ctx.Queue()
    procs = [ctx.Process(target=_oracle_replica, args=(dims, ns, warmup, reps, barrier, q)) for _ in range(cores)]
    for pr in procs:
        pr.start()
    spans = [q.get() for _ in procs]
    for pr in procs:
        pr.join()
    wall = max(t for _, t in spans) - min(t for t, _ in spans)
    n = dims[0] * dims[1] * dims[2] * dims[3] // 2 * ns
    return cores * reps * flops_ccdag(n, ns) / wall / 1e9, wall, cores


def run_reference(args):
    """The oracle, as it stands, on all host cores: each step is one FP64 C C^dag application
    per core (independent replicas, the CPU analogue of the replica scaling on GPUs)."""
    world, rank, _ = dist_env()
    if rank != 0:
        return
    gf, wall, cores = oracle_on_all_cores(DIMS, NS, args.warmup, args.steps)
    sample = (f"{args.steps} FP64 C C^dagger applications on 16^3x32x16 per host core, "
              f"{cores} cores in parallel (oracle, one thread each)")
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": gf, "unit": "GFLOP/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": wall / args.steps * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": {"workload": WORKLOAD, "sample": "C C^dagger application"},
        "cpu_baseline": {"value": gf, "unit": "GFLOP/s", "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": gf, "unit": "GFLOP/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


def cpu_baseline_sample(gpu_iters, gpu_restarts):
    """The oracle on the host cores, bounded samples: one FP64 C C^dagger application on one
    core (the line's value) and on every core at once; the whole 4^4x8 normal-equation solve;
    and the 16^3x32x16 solve time extrapolated from the C C^dagger cost and the GPU solve's
    iteration and restart counts (one C C^dagger each; labelled as extrapolated)."""
    import oracle
    from paper_1101_0423_gb300 import inputs
    oracle.build()
    om, sg = inputs.weights("cosine", NS)
    U = inputs.gauge_field(DIMS, EPS, seed=SEED)
    x = inputs.gaussian_source(DIMS, NS, seed=SEED, parity=1)
    mp, mm = oracle.m5(NS, M0, MQ, om, sg)
    n = DIMS[0] * DIMS[1] * DIMS[2] * DIMS[3] // 2 * NS
    t0 = time.perf_counter()
    oracle.ccdag_op(DIMS, NS, U, mp, mm, 1, x)
    dt = time.perf_counter() - t0
    gf_all, wall_all, cores = oracle_on_all_cores(DIMS, NS, 0, 1)
    # 4^4 x 8 Shamir normal equations on even sites (the small workload), solved whole
    d0, ns0 = (4, 4, 4, 4), 8
    om0, sg0 = inputs.weights("shamir", ns0)
    mp0, mm0 = oracle.m5(ns0, M0, 0.05, om0, sg0)
    U0 = inputs.gauge_field(d0, 0.3, seed=1)
    b0 = inputs.gaussian_source(d0, ns0, seed=1, parity=0)
    t1 = time.perf_counter()
    _, it0, res0 = oracle.cg(d0, ns0, U0, mp0, mm0, 0, b0, tol=1e-10)
    dt0 = time.perf_counter() - t1
    ops = gpu_iters + gpu_restarts
    return {"value": flops_ccdag(n, NS) / dt / 1e9, "unit": "GFLOP/s", "cores": 1, "kind": "oracle",
            "sample": "one FP64 C C^dagger application on 16^3x32x16 (single thread), "
                      f"{dt:.1f} s; same flop count as the GPU's CG iterations",
            "all_cores": {"value": gf_all, "unit": "GFLOP/s", "cores": cores,
                          "sample": f"one FP64 C C^dagger per core, {cores} cores at once, {wall_all:.1f} s"},
            "small_solve": {"seconds": dt0, "iters": it0, "true_res": res0,
                            "sample": "4^4x8 Shamir normal equations, FP64 CG to 1e-10 (single thread)"},
            "extrapolated_solve_s": {"one_core": ops * dt, "all_cores": ops * flops_ccdag(n, NS) / (gf_all * 1e9),
                                     "basis": f"{gpu_iters} iterations + {gpu_restarts} restarts of the GPU solve, "
                                              "one C C^dagger each (extrapolated, not run)"}}


# ---------------------------------------------------------------- served workload

SERVE_LATTICES_FULL = [(8, 8, 8, 8), (12, 12, 12, 24), (16, 16, 16, 32), (24, 24, 24, 48)]
SERVE_NS = [8, 16, 24, 32]
SERVE_WEIGHTS = ["shamir", "borici", "cosine"]


def serve_requests(n, lattices, seed=77):
    """n requests drawn uniformly from lattice x Ns x mq ~ U[0.005, 0.1] x weight set."""
    from paper_1101_0423_gb300 import inputs
    u = inputs.uniforms(seed, inputs.TAG_MISC, 4 * n)
    reqs = []
    for i in range(n):
        reqs.append(dict(dims=lattices[int(u[4 * i] * len(lattices))], Ns=SERVE_NS[int(u[4 * i + 1] * 4)],
                         mq=0.005 + 0.095 * u[4 * i + 2], weights=SERVE_WEIGHTS[int(u[4 * i + 3] * 3)],
                         rhs_seed=1000 + i))
    return reqs


def serve_run(reqs, lam, gauges_np, inner_prec, max_inflight=4, budget_gb=150.0, seed=78):
    """Submit reqs at Poisson arrival rate lam (1/s), poll until all finish; server stats."""
    import numpy as np
    from paper_1101_0423_gb300 import dwf, inputs
    srv = dwf.dwf_server_create(hbm_budget_gb=budget_gb, max_inflight=max_inflight)
    try:
        handles = {d: dwf.dwf_server_add_gauge(srv, d, U) for d, U in gauges_np.items()}
        gaps = -np.log(1.0 - inputs.uniforms(seed, inputs.TAG_ARRIVALS, len(reqs))) / lam
        rhs = [inputs.gaussian_source(r["dims"], r["Ns"], seed=r["rhs_seed"]) for r in reqs]
        pending, statuses, escalated = [], [], 0
        t0 = time.perf_counter()
        next_t = t0
        for r, g, b in zip(reqs, gaps, rhs):
            next_t += g
            while time.perf_counter() < next_t:
                time.sleep(min(0.002, max(0.0, next_t - time.perf_counter())))
            om, sg = inputs.weights(r["weights"], r["Ns"])
            pending.append(dwf.dwf_submit(srv, r["dims"], r["Ns"], M0, r["mq"], om, sg, handles[r["dims"]], b,
                                          inner_prec=inner_prec, tol=1e-10))
        while pending:
            left = []
            for t in pending:
                res = dwf.dwf_poll(srv, t)
                if res is None:
                    left.append(t)
                else:
                    statuses.append(res[1]["status"])
                    escalated += res[1]["stats"]["escalations"] > 0
            pending = left
            time.sleep(0.002)
        st = dwf.dwf_server_get_stats(srv)
        st["ok"] = sum(1 for x in statuses if x == dwf.DWF_OK)
        # 16-bit solves in AUTO mode that switched to FP32 inner iterations partway
        st["escalated_to_f32"] = escalated
        return st
    finally:
        dwf.dwf_server_destroy(srv)


def serve_measure(n, lattices, inner_prec, fractions, progress=False):
    """Capacity from the requests solved one after another, then Poisson runs at each
    fraction.  A run at fraction f lasts about n / (f x capacity) seconds."""
    from paper_1101_0423_gb300 import inputs
    reqs = serve_requests(n, lattices)
    gauges_np = {d: inputs.gauge_field(d, EPS, seed=10 + i) for i, d in enumerate(SERVE_LATTICES_FULL)
                 if d in {r["dims"] for r in reqs}}
    seq = serve_run(reqs, 1e9, gauges_np, inner_prec, max_inflight=1)   # back to back, one at a time
    capacity = seq["solves_per_s"]
    if progress:
        est = sum(n / (f * capacity) for f in fractions)
        print(f"serve: capacity {capacity:.3f} solves/s; the {len(fractions)} arrival-rate runs take about "
              f"{est / 60:.0f} min", file=sys.stderr, flush=True)
    for f in fractions:
        if progress:
            print(f"serve: lambda = {f} x capacity ({n} requests)", file=sys.stderr, flush=True)
        st = serve_run(reqs, f * capacity, gauges_np, inner_prec)
        yield {"lambda_fraction": f, "lambda_per_s": f * capacity, "capacity_per_s": capacity,
               "solves_per_s": st["solves_per_s"], "p50_ms": st["p50_ms"], "p99_ms": st["p99_ms"],
               "mean_ms": st["mean_ms"], "completed": st["completed"], "ok": st["ok"],
               "batched": st["batched"], "escalated_to_f32": st["escalated_to_f32"]}


def odwf_measure(repeats=3):
    """The optimal domain-wall operator: sigma = omega = the optimal weights for |H_w| in
    [0.05, 6.2] (dwf_optimal_weights), on the 16^3 x 32 x 16 lattice, source, gauge and
    mass of the default line, against the cosine weights of that line.  FP32 inner, 1e-10."""
    import torch
    from paper_1101_0423_gb300 import dwf, inputs
    lmin, lmax = 0.05, 6.2
    om_opt, delta = dwf.dwf_optimal_weights(NS, lmin, lmax)
    U = inputs.gauge_field(DIMS, EPS, seed=SEED)
    eta = inputs.gaussian_source(DIMS, NS, seed=SEED)
    stream = torch.cuda.current_stream()
    rows = {}
    for name, (om, sg) in {"optimal": (om_opt, om_opt), "cosine": inputs.weights("cosine", NS)}.items():
        with dwf.Context(DIMS, NS, M0, MQ, om, sg, U) as ctx:
            d_eta = torch.from_numpy(eta).cuda()
            d_psi = torch.empty_like(d_eta)
            dwf.dwf_solve_dev(ctx.h, d_eta, d_psi, stream=stream)  # warm-up
            times, st = [], None
            for _ in range(repeats):
                st = dwf.dwf_solve_dev(ctx.h, d_eta, d_psi, stream=stream)
                times.append(st["time_ms"])
            ms = statistics.median(times)
            rows[name] = {"solve_ms": ms, "gflops": st["flops"] / (ms * 1e-3) / 1e9, "iters": st["iters"],
                          "restarts": st["restarts"], "true_res_full": st["true_res_full"]}
    return {"workload": "optimal domain-wall weights (sigma = omega, |H_w| in [0.05, 6.2]), 16^3x32xNs16, "
                        "mq 0.02, fp32 inner, tol 1e-10", "delta": delta, "omega": [float(w) for w in om_opt],
            **rows}


def batch_measure():
    """12 spin-colour point sources on 24^3 x 48 x 16 Shamir (mq = 0.01): one batched solve
    against the same 12 solved one after another; and a ragged set of 8 right-hand sides on
    16^3 x 32 with Ns in {8,12,16,20,24,32,12,16} and masses 0.005..0.1 (different operators),
    served concurrently, solved one after another, and as one ragged solve; and 8 sources of one operator on
    8^4 x 16 and 12^3 x 24 x 16, single FP32 solves against batches in FP32, fp16 and bf16.
    FP64 restarts, 1e-10."""
    import numpy as np
    import torch
    from paper_1101_0423_gb300 import dwf, inputs
    out = []
    dims, ns, mq = (24, 24, 24, 48), 16, 0.01
    om, sg = inputs.weights("shamir", ns)
    U = inputs.gauge_field(dims, EPS, seed=3)
    src = np.stack([inputs.point_source(dims, ns, spin, col) for spin in range(4) for col in range(3)])
    stream = torch.cuda.current_stream()
    with dwf.Context(dims, ns, M0, mq, om, sg, U) as ctx:
        d_rhs = torch.from_numpy(src).cuda()
        d_sol = torch.empty_like(d_rhs)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        st_b = dwf.dwf_solve_batch_dev(ctx.h, 12, d_rhs, d_sol, stream=stream)
        torch.cuda.synchronize()
        tb = time.perf_counter() - t0
        t0 = time.perf_counter()
        st_s = [dwf.dwf_solve_dev(ctx.h, d_rhs[k], d_sol[k], stream=stream) for k in range(12)]
        torch.cuda.synchronize()
        ts = time.perf_counter() - t0
    fl_b = sum(x["flops"] for x in st_b)
    fl_s = sum(x["flops"] for x in st_s)
    out.append({"workload": "12 point sources, 24^3x48xNs16 Shamir mq=0.01, fp32 inner",
                "batched": {"solves_per_s": 12 / tb, "seconds": tb, "gflops": fl_b / tb / 1e9,
                            "iters": [x["iters"] for x in st_b],
                            "max_true_res_full": max(x["true_res_full"] for x in st_b)},
                "sequential": {"solves_per_s": 12 / ts, "seconds": ts, "gflops": fl_s / ts / 1e9,
                               "iters": [x["iters"] for x in st_s],
                               "max_true_res_full": max(x["true_res_full"] for x in st_s)}})
    # ragged set: different operators, served concurrently vs one after another
    dims = (16, 16, 16, 32)
    Ur = inputs.gauge_field(dims, EPS, seed=4)
    nss = [8, 12, 16, 20, 24, 32, 12, 16]
    masses = list(np.geomspace(0.005, 0.1, 8))
    rhs = [inputs.gaussian_source(dims, n, seed=200 + i) for i, n in enumerate(nss)]
    om_sg = [inputs.weights("shamir", n) for n in nss]
    t0 = time.perf_counter()
    seq_ok = 0
    for n, m, b, (om, sg) in zip(nss, masses, rhs, om_sg):
        with dwf.Context(dims, n, M0, m, om, sg, Ur) as ctx:
            _, st = dwf.dwf_solve(ctx.h, b)
            seq_ok += st["converged"]
    ts = time.perf_counter() - t0
    srv = dwf.dwf_server_create(hbm_budget_gb=150.0, max_inflight=8)
    try:
        g = dwf.dwf_server_add_gauge(srv, dims, Ur)
        t0 = time.perf_counter()
        tickets = [dwf.dwf_submit(srv, dims, n, M0, m, om, sg, g, b)
                   for n, m, b, (om, sg) in zip(nss, masses, rhs, om_sg)]
        ok = 0
        while tickets:
            left = []
            for t in tickets:
                r = dwf.dwf_poll(srv, t)
                if r is None:
                    left.append(t)
                else:
                    ok += r[1]["status"] == dwf.DWF_OK
            tickets = left
            time.sleep(0.002)
        tc = time.perf_counter() - t0
    finally:
        dwf.dwf_server_destroy(srv)
    # the same set on eight resident contexts sharing one gauge field: one after another, and
    # as one ragged solve (every interval of inner iterations of all eight one CUDA graph)
    gh = dwf.dwf_gauge_create(dims, Ur)
    ctxs = [dwf.Context(dims, n, M0, m, om, sg, gauge=gh) for n, m, (om, sg) in zip(nss, masses, om_sg)]
    dwf.dwf_gauge_release(gh)
    try:
        d_rhs = [torch.from_numpy(b).cuda() for b in rhs]
        d_seq = [torch.empty_like(b) for b in d_rhs]
        d_rag = [torch.empty_like(b) for b in d_rhs]
        for c, b, x in zip(ctxs, d_rhs, d_seq):   # warm-up: builds the gauge forms, tunes shapes
            dwf.dwf_solve_dev(c.h, b, x, stream=stream)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        st_seq = [dwf.dwf_solve_dev(c.h, b, x, stream=stream) for c, b, x in zip(ctxs, d_rhs, d_seq)]
        torch.cuda.synchronize()
        tr_seq = time.perf_counter() - t0
        t0 = time.perf_counter()
        st_rag = dwf.dwf_solve_ragged_dev([c.h for c in ctxs], d_rhs, d_rag, stream=stream)
        torch.cuda.synchronize()
        tr_rag = time.perf_counter() - t0
        same = all(bool(torch.equal(a, b)) for a, b in zip(d_seq, d_rag))
    finally:
        for c in ctxs:
            c.close()
    out.append({"workload": "ragged 8 rhs, 16^3x32, Ns {8,12,16,20,24,32,12,16}, mq 0.005..0.1, fp32 inner",
                "served_concurrently": {"solves_per_s": 8 / tc, "seconds": tc, "ok": ok,
                                        "note": "includes building each context"},
                "sequential": {"solves_per_s": 8 / ts, "seconds": ts, "ok": seq_ok,
                               "note": "includes building each context"},
                "resident_sequential": {"solves_per_s": 8 / tr_seq, "seconds": tr_seq,
                                        "iters": [x["iters"] for x in st_seq],
                                        "max_true_res_full": max(x["true_res_full"] for x in st_seq)},
                "ragged_one_graph": {"solves_per_s": 8 / tr_rag, "seconds": tr_rag,
                                     "iters": [x["iters"] for x in st_rag],
                                     "max_true_res_full": max(x["true_res_full"] for x in st_rag),
                                     "identical_to_sequential": same}})
    # small volumes, where one right-hand side leaves most of the GPU idle: 8 sources of one
    # operator on 8^4 x 16 and 12^3 x 24 x 16 (cosine, mq 0.02), single FP32 solves one after
    # another against batches in FP32, fp16 and bf16 inner precision (all to 1e-10)
    for dims in ((8, 8, 8, 8), (12, 12, 12, 24)):
        om, sg = inputs.weights("cosine", NS)
        Us = inputs.gauge_field(dims, EPS, seed=5)
        src = np.stack([inputs.gaussian_source(dims, NS, seed=400 + k) for k in range(8)])
        row = {"workload": f"8 sources of one operator, {'x'.join(map(str, dims))}x16 cosine mq 0.02"}
        with dwf.Context(dims, NS, M0, MQ, om, sg, Us) as ctx:
            d_rhs = torch.from_numpy(src).cuda()
            d_sol = torch.empty_like(d_rhs)
            dwf.dwf_solve_dev(ctx.h, d_rhs[0], d_sol[0], stream=stream)   # warm-up (tunes shapes)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            st = [dwf.dwf_solve_dev(ctx.h, d_rhs[k], d_sol[k], stream=stream) for k in range(8)]
            torch.cuda.synchronize()
            ts = time.perf_counter() - t0
            row["single_f32_sequential"] = {"solves_per_s": 8 / ts, "iters": st[0]["iters"],
                                            "max_true_res_full": max(x["true_res_full"] for x in st)}
            for name, prec in (("batch_f32", dwf.PREC_F32), ("batch_fp16", dwf.PREC_F16), ("batch_bf16", dwf.PREC_BF16)):
                dwf.dwf_solve_batch_dev(ctx.h, 8, d_rhs, d_sol, stream=stream, inner_prec=prec)  # warm-up
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                st = dwf.dwf_solve_batch_dev(ctx.h, 8, d_rhs, d_sol, stream=stream, inner_prec=prec)
                torch.cuda.synchronize()
                tb = time.perf_counter() - t0
                row[name] = {"solves_per_s": 8 / tb, "iters": max(x["iters"] for x in st),
                             "max_true_res_full": max(x["true_res_full"] for x in st)}
        out.append(row)
    return out


def _oracle_residual_worker(args):
    """|eta - D psi| / |eta| by the FP64 oracle, one solution (spawned process)."""
    import numpy as np
    import oracle
    from paper_1101_0423_gb300 import inputs
    dims, ns, eps, gseed, mq, kind, eta, psi = args
    om, sg = inputs.weights(kind, ns)
    U = inputs.gauge_field(dims, eps, seed=gseed)
    return float(np.linalg.norm(eta - oracle.dfull(dims, ns, U, M0, mq, om, sg, psi)) / np.linalg.norm(eta))


def configs_measure():
    """Every workload configuration solved on the GPU at its real size, its true residual
    recomputed by the FP64 oracle on the host cores (a spawned pool, one solution per core):
    4^4x8 Shamir normal equations; 16^3x32x16 cosine and Borici; the cosine solve with FP32,
    bf16 and fp16 inner iterations; the 12 point sources on 24^3x48x16 as one batch; the
    ragged set of 8 right-hand sides (Ns 8..32, masses 0.005..0.1) on 16^3x32."""
    import multiprocessing as mp_
    import numpy as np
    import torch
    import oracle
    from paper_1101_0423_gb300 import dwf, inputs
    oracle.build()
    pool = mp_.get_context("spawn").Pool(min(12, host_cores()))
    rows, jobs = [], []
    stream = torch.cuda.current_stream()

    def solve(dims, ns, kind, mq, eps, gseed, eta, **kw):
        om, sg = inputs.weights(kind, ns)
        with dwf.Context(dims, ns, M0, mq, om, sg, inputs.gauge_field(dims, eps, seed=gseed)) as ctx:
            d_eta = torch.from_numpy(eta).cuda()
            d_psi = torch.empty_like(d_eta)
            st = dwf.dwf_solve_dev(ctx.h, d_eta, d_psi, stream=stream, **kw)
            return d_psi.cpu().numpy(), st

    # 4^4 x 8 normal equations (the small workload): the oracle's C C^dag residual inline
    d0, ns0 = (4, 4, 4, 4), 8
    om0, sg0 = inputs.weights("shamir", ns0)
    U0 = inputs.gauge_field(d0, 0.3, seed=1)
    b0 = inputs.gaussian_source(d0, ns0, seed=1, parity=0)
    x0, st0 = solve(d0, ns0, "shamir", 0.05, 0.3, 1, b0, system=dwf.SYS_NORMAL, schur_parity=0)
    mp, mm = oracle.m5(ns0, M0, 0.05, om0, sg0)
    r0 = np.linalg.norm(b0 - oracle.ccdag_op(d0, ns0, U0, mp, mm, 0, x0)) / np.linalg.norm(b0)
    rows.append({"config": "4^4x8 Shamir mq 0.05, normal equations on even sites", "inner": "f32",
                 "iters": st0["iters"], "restarts": st0["restarts"], "solve_ms": st0["time_ms"],
                 "true_res_library": st0["true_res"], "true_res_oracle": float(r0)})
    eta16 = inputs.gaussian_source(DIMS, NS, seed=SEED)
    sols = {}
    for kind, inner in (("cosine", "f32"), ("cosine", "bf16"), ("cosine", "f16"), ("borici", "f32")):
        prec = {"f32": dwf.PREC_F32, "bf16": dwf.PREC_BF16, "f16": dwf.PREC_F16}[inner]
        # reliable updates throughout: every inner iteration in the precision named
        psi, st = solve(DIMS, NS, kind, MQ, EPS, SEED, eta16, inner_prec=prec, mode=dwf.MODE_RELIABLE)
        if kind == "cosine":
            sols[inner] = psi
        rows.append({"config": f"16^3x32x16 {kind} mq 0.02", "inner": inner, "mode": "reliable",
                     "delta": 0.3 if inner == "f16" else 0.01, "iters": st["iters"],
                     "restarts": st["restarts"], "escalations": st["escalations"], "solve_ms": st["time_ms"],
                     "true_res_library": st["true_res_full"]})
        jobs.append((len(rows) - 1, (DIMS, NS, EPS, SEED, MQ, kind, eta16, psi)))
    for inner in ("bf16", "f16"):
        rows[[r["inner"] for r in rows].index(inner)]["rel_diff_vs_f32"] = float(
            np.linalg.norm(sols[inner] - sols["f32"]) / np.linalg.norm(sols["f32"]))
    # 12 point sources, 24^3 x 48 x 16 Shamir, one batch
    d3 = (24, 24, 24, 48)
    om3, sg3 = inputs.weights("shamir", NS)
    src = np.stack([inputs.point_source(d3, NS, spin, col) for spin in range(4) for col in range(3)])
    with dwf.Context(d3, NS, M0, 0.01, om3, sg3, inputs.gauge_field(d3, EPS, seed=3)) as ctx:
        d_rhs = torch.from_numpy(src).cuda()
        d_sol = torch.empty_like(d_rhs)
        st3 = dwf.dwf_solve_batch_dev(ctx.h, 12, d_rhs, d_sol, stream=stream)
        sol3 = d_sol.cpu().numpy()
    for k in range(12):
        rows.append({"config": f"24^3x48x16 Shamir mq 0.01, point source {k} (spin {k // 3}, colour {k % 3}), "
                               "batch of 12", "inner": "f32", "iters": st3[k]["iters"],
                     "restarts": st3[k]["restarts"], "solve_ms": st3[k]["time_ms"],
                     "true_res_library": st3[k]["true_res_full"]})
        jobs.append((len(rows) - 1, (d3, NS, EPS, 3, 0.01, "shamir", src[k], sol3[k])))
    del d_rhs, d_sol
    # the ragged set: 8 operators on 16^3 x 32
    for i, (n, m) in enumerate(zip([8, 12, 16, 20, 24, 32, 12, 16], np.geomspace(0.005, 0.1, 8))):
        eta = inputs.gaussian_source(DIMS, n, seed=200 + i)
        psi, st = solve(DIMS, n, "shamir", float(m), EPS, 4, eta)
        rows.append({"config": f"16^3x32 Shamir, ragged set member {i}: Ns {n}, mq {m:.4f}", "inner": "f32",
                     "iters": st["iters"], "restarts": st["restarts"], "solve_ms": st["time_ms"],
                     "true_res_library": st["true_res_full"]})
        jobs.append((len(rows) - 1, (DIMS, n, EPS, 4, float(m), "shamir", eta, psi)))
    for (i, _), res in zip(jobs, pool.imap(_oracle_residual_worker, [j for _, j in jobs])):
        rows[i]["true_res_oracle"] = res
    pool.close()
    pool.join()
    return rows


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--inner", default="f32", choices=["f32", "f16", "bf16", "f64"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-serve", action="store_true")
    ap.add_argument("--batch", action="store_true",
                    help="only the batched workloads: 12 point sources on 24^3x48x16, ragged 8-rhs set")
    ap.add_argument("--serve", action="store_true",
                    help="only the served sweep: 40 requests over all four lattices at 0.2..0.95 of capacity")
    ap.add_argument("--serve-requests", type=int, default=40,
                    help="requests per arrival-rate run of --serve (the sweep lasts about 12.5 x this / capacity)")
    ap.add_argument("--serve-prec", choices=("bf16", "f16", "f32"), default="bf16",
                    help="inner precision of the served solves (the served workload names bf16)")
    ap.add_argument("--serve-fractions", default="0.2,0.4,0.6,0.8,0.95",
                    help="arrival rates of --serve as fractions of the measured capacity")
    ap.add_argument("--odwf", action="store_true",
                    help="only the optimal-weights solve on 16^3x32x16 against the cosine weights")
    ap.add_argument("--apply-ccdag", type=int, default=0, metavar="N",
                    help="only N applications of C C^dagger on the benchmark's lattice, inputs and "
                         "launch configuration (a short program for profiler captures): one solve first "
                         "picks the tuned launch shapes, then the applications run inside a profiler "
                         "range (capture with ncu --profile-from-start off)")
    ap.add_argument("--apply-prec", choices=("f32", "f16", "bf16", "f64"), default="f32",
                    help="arithmetic form of --apply-ccdag")
    ap.add_argument("--configs", action="store_true",
                    help="only the per-configuration table: every workload at its real size, iterations, "
                         "restarts and the oracle-recomputed true residual")
    args = ap.parse_args()
    if args.impl == "reference":
        return run_reference(args)
    if args.batch:
        from paper_1101_0423_gb300 import build as _b
        _b.build()
        for row in batch_measure():
            print(json.dumps(row))
        return
    if args.apply_ccdag:
        import torch
        from paper_1101_0423_gb300 import build as _b, dwf, inputs
        _b.build()
        om, sg = inputs.weights("cosine", NS)
        x = torch.from_numpy(inputs.gaussian_source(DIMS, NS, seed=9, parity=1)).cuda()
        y = torch.empty_like(x)
        with dwf.Context(DIMS, NS, M0, MQ, om, sg, inputs.gauge_field(DIMS, EPS, seed=SEED)) as ctx:
            stream = torch.cuda.current_stream()
            prec = {"f32": dwf.PREC_F32, "f16": dwf.PREC_F16, "bf16": dwf.PREC_BF16,
                    "f64": dwf.PREC_F64}[args.apply_prec]
            # the benchmark's solve tunes the launch shapes the applications then use (FP64 has
            # one shape, its solve runs in FP32)
            eta = torch.from_numpy(inputs.gaussian_source(DIMS, NS, seed=SEED)).cuda()
            dwf.dwf_solve_dev(ctx.h, eta, torch.empty_like(eta), stream=stream,
                              inner_prec=dwf.PREC_F32 if prec == dwf.PREC_F64 else prec, mode=dwf.MODE_RELIABLE)
            stream.synchronize()
            torch.cuda.profiler.start()
            for _ in range(args.apply_ccdag):
                dwf.dwf_apply_eo_dev(ctx.h, dwf.OP_CCDAG, prec, 1, x, y, stream=stream)
            stream.synchronize()
            torch.cuda.profiler.stop()
        print(json.dumps({"applied": "C C^dagger " + args.apply_prec, "times": args.apply_ccdag,
                          "max_abs": float(y.abs().max())}))
        return
    if args.configs:
        from paper_1101_0423_gb300 import build as _b
        _b.build()
        for row in configs_measure():
            print(json.dumps(row), flush=True)
        return
    if args.odwf:
        from paper_1101_0423_gb300 import build as _b
        _b.build()
        print(json.dumps(odwf_measure()))
        return
    if args.serve:
        from paper_1101_0423_gb300 import build as _b, dwf
        _b.build()
        prec = {"bf16": dwf.PREC_BF16, "f16": dwf.PREC_F16, "f32": dwf.PREC_F32}[args.serve_prec]
        fractions = [float(f) for f in args.serve_fractions.split(",")]
        for row in serve_measure(args.serve_requests, SERVE_LATTICES_FULL, prec, fractions, progress=True):
            print(json.dumps({"metric": "served solves/s, p99 latency", "config": {
                "workload": "served: uniform lattice {8^4,12^3x24,16^3x32,24^3x48} x Ns {8,16,24,32} x "
                            f"mq U[0.005,0.1] x {{shamir,borici,cosine}}, {args.serve_prec} inner, tol 1e-10, "
                            "150 GB budget", "requests": args.serve_requests}, **row}), flush=True)
        return

    import numpy as np
    import torch
    import torch.distributed as tdist

    from paper_1101_0423_gb300 import build as _build
    from paper_1101_0423_gb300 import dwf, inputs

    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    if world > 1:
        tdist.init_process_group("nccl", device_id=torch.device("cuda", local))
    if rank == 0:
        _build.build()
    if world > 1:
        tdist.barrier()
    dwf.load()
    prec = {"f32": dwf.PREC_F32, "f16": dwf.PREC_F16, "bf16": dwf.PREC_BF16, "f64": dwf.PREC_F64}[args.inner]

    om, sg = inputs.weights("cosine", NS)
    U = inputs.gauge_field(DIMS, EPS, seed=SEED)
    eta = inputs.gaussian_source(DIMS, NS, seed=SEED)
    stream = torch.cuda.current_stream()
    ctx = dwf.Context(DIMS, NS, M0, MQ, om, sg, U)
    d_eta = torch.from_numpy(eta).cuda()
    d_psi = torch.empty_like(d_eta)
    params = dwf.dwf_solve_params_default()
    params.tol = 1e-10
    params.inner_prec = prec

    def step(profile=0):
        params.profile = profile
        return dwf.dwf_solve_dev(ctx.h, d_eta, d_psi, params=params, stream=stream)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()

    def barrier():
        if world > 1:
            tdist.barrier()
        torch.cuda.synchronize()

    # ---- timed region: device-resident inputs
    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)
    barrier()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    stats = [step() for _ in range(args.steps)]
    e1.record(stream)
    barrier()
    clocks = sampler.stop()
    ms = e0.elapsed_time(e1)
    flops = sum(s["flops"] for s in stats)
    launches = sum(s["kernel_launches"] for s in stats)
    t_max, flops_all = aggregate_over_ranks(ms, flops, device="cuda")
    value = flops_all / (t_max * 1e-3) / 1e9

    # ---- e2e: through dwf_solve with pinned host buffers, copies inside the timed region
    h_eta = torch.from_numpy(eta).pin_memory()
    h_psi = torch.empty_like(h_eta).pin_memory()
    import ctypes
    lib = dwf.load()
    P = ctypes.POINTER(ctypes.c_double)
    pe = ctypes.cast(h_eta.data_ptr(), P)
    pp = ctypes.cast(h_psi.data_ptr(), P)
    params.profile = 0
    barrier()
    t0 = time.perf_counter()
    e2e_flops, e2e_dev_ms, e2e_walls = 0.0, 0.0, []
    for _ in range(args.steps):
        st = dwf.SolveStats()
        tw = time.perf_counter()
        rc = lib.dwf_solve(ctx.h, pe, pp, ctypes.byref(params), ctypes.byref(st))
        e2e_walls.append(1e3 * (time.perf_counter() - tw))
        if rc != 0:
            raise dwf.DwfError(rc, dwf.dwf_last_error(ctx.h))
        e2e_flops += st.flops
        e2e_dev_ms += st.time_ms
    barrier()
    e2e_s = time.perf_counter() - t0
    e2e_s, e2e_flops = aggregate_over_ranks(e2e_s, e2e_flops, device="cuda")
    e2e_value = e2e_flops / e2e_s / 1e9
    nbytes = eta.nbytes

    # ---- roofline of the dominant kernel class: CUDA events around each launch on the
    # library's launch stream, over profiled steps of the same workload
    prof = [step(profile=1) for _ in range(max(1, min(args.steps, 2)))]
    torch.cuda.synchronize()
    n = DIMS[0] * DIMS[1] * DIMS[2] * DIMS[3] // 2 * NS
    S = {0: 192, 1: 96, 2: 52, 3: 52}[prec]
    G = {0: 144, 1: 72, 2: 24, 3: 24}[prec]
    alg = {"hop_m5": 2 * S + 8 * G / NS, "hop_xpay": 3 * S + 8 * G / NS, "hop_update": 4 * S + 8 * G / NS,
           "smix_p": 6 * S}
    cls_ms = {k: sum(p["class_ms"][k] for p in prof) for k in dwf.KC_NAMES}
    cls_n = {k: sum(p["class_launches"][k] for p in prof) for k in dwf.KC_NAMES}
    total = sum(cls_ms.values())
    dom = max(alg, key=lambda k: cls_ms[k])
    avg_ms = cls_ms[dom] / max(cls_n[dom], 1)
    achieved = alg[dom] * n / (avg_ms * 1e-3) / 1e9
    peak, peak_kind = measured_peaks()
    traffic = NCU_TRAFFIC.get(dom)
    roofline = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                "traffic": traffic, "kernel": f"k_hop ({dom})", "peak_source": peak_kind,
                "bytes_per_launch": alg[dom] * n, "avg_launch_us": avg_ms * 1e3,
                "class_share": {k: cls_ms[k] / total for k in cls_ms},
                "class_frac": {k: (alg[k] * n / (cls_ms[k] / max(cls_n[k], 1) * 1e-3) / 1e9) / peak
                               for k in alg if cls_n[k]}}
    # the launch shapes the autotuner chose in this process for the timed solves
    shapes = {}
    for name, kc in (("hop_m5", dwf.KC_HOP_M5), ("hop_xpay", dwf.KC_HOP_XPAY), ("hop_update", dwf.KC_HOP_UPDATE)):
        try:
            t, pers, tuned = dwf.dwf_tuned_shape(ctx.h, prec, kc)
            shapes[name] = {"threads": t, "persistent": bool(pers), "tuned": bool(tuned)}
        except Exception:  # a shape report must not cost the line
            pass
    roofline["launch_shapes"] = shapes

    if rank != 0:
        if world > 1:
            tdist.destroy_process_group()
        return
    s0 = stats[-1]
    out = {
        "metric": METRIC, "value": value, "unit": "GFLOP/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": t_max / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": value / PAPER_BEST_GFLOPS,
        "dtype": {0: "f64", 1: "f32", 2: "f16", 3: "bf16"}[prec] + "+f64-restarts",
        "data": "synthetic",
        "config": {"workload": WORKLOAD, "lattice": "16x16x16x32", "Ns": NS, "weights": "cosine omega=sigma",
                   "inner_prec": args.inner, "tol": 1e-10, "parallelism": f"replicas{world}",
                   "l2": "working set > L2 (no flush needed)",
                   "iters": s0["iters"], "restarts": s0["restarts"], "true_res": s0["true_res"],
                   "true_res_full": s0["true_res_full"],
                   "solves_per_s": world * args.steps / (t_max * 1e-3)},
        "e2e": {"value": e2e_value, "unit": "GFLOP/s", "h2d_bytes_per_step": nbytes, "d2h_bytes_per_step": nbytes,
                "wall_ms_per_step": e2e_walls, "solve_device_ms_per_step": e2e_dev_ms / args.steps},
        "gpu_launches": launches,
        "roofline": roofline,
        "clocks": clocks,
        "vs_baseline_note": "value / 233 Gflops (paper Table 1, GTX 480, same lattice): other hardware, context",
    }
    if world == 1 and not args.no_serve:
        # bounded served sample: 12 Poisson-arriving requests at 0.8 of the measured capacity,
        # lattices up to 16^3x32 (the full sweep over all four lattices is `bench.py --serve`)
        row = next(serve_measure(12, SERVE_LATTICES_FULL[:3], dwf.PREC_BF16, [0.8]))
        out["served"] = {"solves_per_s": row["solves_per_s"], "p50_ms": row["p50_ms"], "p99_ms": row["p99_ms"],
                         "lambda_per_s": row["lambda_per_s"], "capacity_per_s": row["capacity_per_s"],
                         "requests": row["completed"], "ok": row["ok"],
                         "escalated_to_f32": row["escalated_to_f32"],
                         "sample": "12 requests, uniform lattice {8^4,12^3x24,16^3x32} x Ns {8,16,24,32} x "
                                   "mq U[0.005,0.1] x {shamir,borici,cosine}, bf16 inner (AUTO mode: a "
                                   "solve whose bf16 cycles fail continues in FP32), tol 1e-10, "
                                   "Poisson arrivals at 0.8 x single-stream capacity, 4 slots, 150 GB budget"}
    if world == 1 and not args.no_cpu_baseline:
        out["cpu_baseline"] = cpu_baseline_sample(s0["iters"], s0["restarts"])
    print(json.dumps(out))
    ctx.close()
    if world > 1:
        tdist.destroy_process_group()


if __name__ == "__main__":
    main()

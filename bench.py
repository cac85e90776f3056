#!/usr/bin/env python3
"""Benchmark: QP solves/s of the GB300 OSQP path, batched vs plain.

Default workload: 4096 ragged MPC QPs (App. A.3 generator) solved cold in
one persistent batched launch, FP32-mixed, ε_abs = ε_rel = 1e-3.  One step
= one cold solve of every problem of the batch (Ruiz scaling, ρ vector and
Jacobi diagonal, the ADMM iterations with PCG linear solves, termination,
unscaling), timed on the device (CUDA events on the solver's stream); the
batch's data (GBs) exceed L2, so no flush is needed.  The same line carries
the plain single-problem FP64 form (the 20000 × 200 Lasso QP, one solve per
step, L2 flushed between steps) under "plain", so batched and plain come
from one run.

``--workload`` selects any other workload alone.  ``--impl reference``
times the FP64 CPU oracle on the same workload instead (rank 0 only).
Multi-GPU: the batched workload is one problem set of 4096·N problems
partitioned across the N ranks by longest-processing-time on estimated work
(weak scaling, no collective on the data path); single problems run as
replicas.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_1711_08013_gb300 import problems as pb  # noqa: E402

METRIC = "QP solves/s at eps 1e-3 (batched vs plain); ADMM iter/s; p50/p99 solve latency"
UNIT = "QP solves/s"
WORKLOADS = {
    "lasso": (1, "Lasso QP: data matrix 20000x200 at 15% N(0,1), lambda=0.2*|Ad^T b|_inf; "
                 "variables (x,y,t) n=20400, rows m=20400"),
    "random": (0, "random QP n=50 m=500, P=MM^T+1e-2 I, A at 15% N(0,1)"),
    "portfolio": (2, "portfolio QP n=10000 assets k=100 factors, F at 50% N(0,1); "
                     "variables (x,y) n=10100, rows m=10101"),
    "mpc_batch": (3, "4096 ragged MPC QPs per GPU, nx~U{4..32}, nu=nx/2, T~U{10..30}, one "
                     "persistent launch (cold: scaling + ADMM per problem)"),
    "serve": (4, "serving: Poisson arrivals at RATE req/s over a pool of 256 random-QP (m=10n) and "
                 "256 Huber (100n x n) problem IDs, n~logU[10,NMAX], warm-started perturbed q/l/u"),
    "svm": (None, "SVM QP (App. A.7): 100 features, 10000 points at 15% density, labels split in half; "
                  "variables (x,t) n=10100, rows m=20000"),
    "eqqp": (None, "equality-constrained QP (App. A.2): n=1000, m=500, P=MM^T+1e-2 I, A at 15%"),
    "lasso_path": (None, "Lasso regularisation path: the 20000x200 Lasso QP, 100 lambda values "
                         "log-spaced from |Ad^T b|_inf to 0.01 of it, q updated in place, warm start"),
    "mpc_loop": (None, "MPC closed loop: nx=80, nu=40, T=10 (App. A.3 instance ranges, DARE terminal "
                       "cost), 100 simulation steps, l/u of the initial-state rows updated, warm start"),
    "portfolio_bt": (None, "portfolio back test: n=10000 assets, k=100 factors, 960 trading days, daily "
                           "mu update, monthly D/F value update (same pattern), warm start"),
}
PARAM_LEN = {"lasso_path": 100, "mpc_loop": 100, "portfolio_bt": 960}
# DRAM bytes (dram__bytes_read.sum + dram__bytes_write.sum) of one launch of
# the dominant kernel, from one single-pass ncu capture of the same command
# with the kernels as they are now; for the batch, the capture of the first 608
# problems scaled by the problems of the launch.  Absent: not captured
# since the kernels last changed.  The single-problem figure holds for the
# row partitions it was captured with (group widths of Kn and Ā).
TRAFFIC = {("lasso", "fp64"): 21.120000e6}
TRAFFIC_GROUPS = {("lasso", "fp64"): (2, 2)}
TRAFFIC_BATCH_PER_PROBLEM = {"fp32": 3.025579776e9 / 608}
# Mean time per QP and mean iterations per QP that the paper reports for the
# same sequences (OSQP direct method on a CPU; context only)
PARAM_PAPER = {
    "lasso_path": {"dim": 200, "ws_s": 0.149, "nows_s": 2.089, "ws_iter": 26.0, "nows_iter": 281.75},
    "mpc_loop": {"dim": 80, "ws_s": 0.0217, "nows_s": 0.0668, "ws_iter": 31.75, "nows_iter": 32.0},
    "portfolio_bt": {"dim": 100, "ws_s": 0.0305, "nows_s": 0.177, "ws_iter": 25.4, "nows_iter": 93.3},
}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["gb300", "reference"], default="gb300")
    ap.add_argument("--workload", choices=sorted(WORKLOADS), default="mpc_batch")
    ap.add_argument("--precision", choices=["fp64", "fp32"], default=None,
                    help="default: fp32 (mixed) for mpc_batch, fp64 otherwise")
    ap.add_argument("--autotune", type=int, choices=[0, 1], default=1,
                    help="1: row partitions chosen by timing at setup; 0: the row-length rule")
    ap.add_argument("--launch", type=int, choices=[0, 1, 2, 3], default=0,
                    help="single problems: 0 the library's rule, 1 one CTA, 2 whole-GPU grid, "
                         "3 one 8-CTA cluster")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-plain", action="store_true",
                    help="mpc_batch: skip the plain single-problem FP64 Lasso measurement")
    ap.add_argument("--duration", type=float, default=60.0, help="serve: seconds of arrivals")
    ap.add_argument("--rate", type=float, default=2000.0, help="serve: requests per second")
    ap.add_argument("--nmax", type=int, default=500, help="serve: largest problem dimension n")
    ap.add_argument("--large-slots", type=int, default=16,
                    help="serve: launch slots that large (cluster) requests may hold at once")
    ap.add_argument("--rates", type=lambda v: [float(x) for x in v.split(",")], default=None,
                    help="serve: comma-separated offered rates to sweep before the headline run")
    ap.add_argument("--seq-len", type=int, default=None,
                    help="parametric workloads: QPs of the sequence (default: the paper's length)")
    args = ap.parse_args()
    if args.precision is None:
        args.precision = "fp32" if args.workload == "mpc_batch" else "fp64"
    return args


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


# ----------------------------------------------------------------------------
# clocks sampled while the timed region runs
# ----------------------------------------------------------------------------
class ClockSampler:
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            f = [a.strip() for a in line.split(",")]
            if len(f) < 9:
                continue
            try:
                rows.append((float(f[1]), float(f[2]), f[5:9]))
            except ValueError:
                continue
        os.remove(self.path)
        if not rows:
            return None
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for _, _, r in rows for i, v in enumerate(r) if v == "Active"})
        return {"sm_mhz": statistics.median(r[0] for r in rows),
                "sm_max_mhz": max(r[1] for r in rows), "reasons": reasons, "samples": len(rows)}


# ----------------------------------------------------------------------------
# algorithmic bytes of one ADMM launch (stages of the ADMM kernel, each array
# read or written once per stage; matrix values + column indices once per
# sparse product, plus one index per row for the row structure; layout
# padding is not counted)
# ----------------------------------------------------------------------------
def admm_bytes(n, m, nnz_kn, nnz_a, sv, K, J, C):
    """Algorithmic bytes of one solve of K ADMM iterations, J PCG iterations
    and C checks: every matrix pass streams its values (sv bytes each), int32
    column indices and int32 row pointers once, and every vector a stage
    touches is read or written once (d = 8 bytes for FP64 vectors, sv for
    working-precision ones); gathers are counted once per stage, as if the
    vector were cached.  Stages: R (Kn pass, first PCG residual and b), A0
    (first Ā pass, M⁻¹r), U (Algorithm 1 steps 5-7); per PCG iteration the Kn
    pass B (w = Ku) and the elementwise updates and inner products Cc, and
    the Ā pass A for every PCG iteration after the first of its ADMM
    iteration; per check K1 (the FP64 products) and K2 (the norms).  A PCG
    iteration thus streams (nnz(P) + 2·nnz(A))·(sv + 4) matrix bytes, with
    nnz_kn = nnz(P full) + nnz(A)."""
    d = 8
    kn = nnz_kn * (sv + 4) + 4 * (n + 1)
    am = nnz_a * (sv + 4) + 4 * (m + 1)
    R = kn + n * (2 * d + sv) + m * 2 * sv + n * 2 * sv
    A0 = am + n * 3 * sv + m * d + n * 2 * sv + m * sv
    B = kn + n * sv + m * sv + n * sv
    Cc = n * 5 * sv + n * 3 * sv + m * (2 * sv + d) + m * sv
    A = am + n * 2 * sv + m * d + n * sv + m * sv
    U = n * (sv + d) + n * 2 * d + m * (sv + 6 * d) + m * (3 * d + 2 * sv)
    K1 = kn + am + n * (2 * d + sv) + m * (2 * d + 1) + n * 4 * d + m * 3 * d
    K2 = m * (9 * d + 1) + m * 2 * sv + n * 8 * d
    a_phases = max(J - K, 0)
    return K * (R + A0 + U) + J * (B + Cc) + a_phases * A + C * (K1 + K2)


def build_problem(args, rank):
    cfg, desc = WORKLOADS[args.workload]
    if args.workload == "svm":
        return cfg, desc, pb.svm(100, seed=7000 + rank)
    if args.workload == "eqqp":
        return cfg, desc, pb.eq_qp(1000, seed=8000 + rank)
    return cfg, desc, pb.config_problem(cfg, instance=rank)


def param_problem(name, rank=0):
    """The first QP of a parametric sequence and the sequence generator."""
    from paper_1711_08013_gb300 import parametric as pm
    if name == "lasso_path":
        qp = pb.lasso(200, seed=1000 + rank)
        return qp, lambda k: pm.lasso_path(qp, k)
    if name == "mpc_loop":
        qp = pb.mpc_paper(80, T=10, seed=2000 + rank)
        return qp, lambda k: pm.mpc_closed_loop(qp, k)
    qp = pb.portfolio(100, seed=3000 + rank)
    return qp, lambda k: pm.portfolio_backtest(qp, days=k, seed=7 + rank)


def param_oracle(name, k, budget_s=15.0):
    """The oracle replaying the sequence, each solve warm-started from its
    previous solution, until k QPs or about budget_s seconds."""
    from oracle import oracle as O
    from paper_1711_08013_gb300 import parametric as pm
    qp, seq = param_problem(name)
    gen = seq(k)
    cur, x, y, done, iters = qp, None, None, 0, 0
    t0 = time.perf_counter()
    try:
        upd = next(gen)
        while True:
            cur = pm.apply_update(cur, upd)
            r = O.solve(cur, x0=x, y0=y)
            x, y = r.x, r.y
            done += 1
            iters += r.iter
            if done >= k or time.perf_counter() - t0 > budget_s:
                break
            upd = gen.send(r.x)
    except StopIteration:
        pass
    return done, time.perf_counter() - t0, iters


def workload_desc(args, workload):
    """The workload's description with its size and rate parameters filled in."""
    return (WORKLOADS[workload][1].replace("NMAX", str(getattr(args, "nmax", "NMAX")))
            .replace("RATE", f"{getattr(args, 'rate', 0):g}"))


def _reference_line(args, workload, value, steps, dt, iters, sample, cores):
    return {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": steps,
        "warmup": 0, "ms_per_step": 1e3 * dt / max(1, steps), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "impl": "reference", "config": {"workload": workload_desc(args, workload), "precision": "fp64",
                                         "eps": 1e-3},
        "admm_iter_per_s": iters / dt if iters is not None else None,
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }


def run_reference(args, ws, rank):
    if rank != 0:
        return 0
    if args.workload == "mpc_batch":
        # the oracle on rank 0's share of the batch (the whole 4096-problem
        # set at N = 1), one problem per process on all host cores; a step is
        # one pass over it, and the run stops early past about two minutes
        import multiprocessing as mp
        from oracle import oracle as O
        O.build()
        count, spec, weights = batch_spec(ws)
        from paper_1711_08013_gb300 import dist as D
        mine = D.shard(weights, 0, ws)
        qps = [pb.mpc(*spec[i][:2], seed=spec[i][2]) for i in mine]
        cores = os.cpu_count() or 1
        with mp.get_context("spawn").Pool(cores) as pool:
            for _ in range(args.warmup):
                pool.map(_oracle_iters_one, qps, chunksize=4)
            t0 = time.perf_counter()
            steps = iters = 0
            while steps < args.steps:
                iters += sum(pool.map(_oracle_iters_one, qps, chunksize=4))
                steps += 1
                if time.perf_counter() - t0 > 120.0:
                    break
            dt = time.perf_counter() - t0
        value = steps * len(qps) / dt
        line = _reference_line(args, "mpc_batch", value, steps, dt, iters,
                               f"{steps} pass(es) over the {len(qps)} problems of rank 0's share, "
                               f"one problem per process on {cores} cores, {dt:.1f} s", cores)
        line["warmup"] = args.warmup
        print(json.dumps(line), flush=True)
        return 0
    if args.workload == "serve":
        # the oracle solving a bounded sample of the request stream (each
        # request's perturbed QP, warm-started from its problem's previous
        # solution as the server does), single thread
        from oracle import oracle as O
        from paper_1711_08013_gb300.serve import poisson_requests
        qps = serve_pool(args.nmax, seed=4000)
        reqs = poisson_requests(qps, args.rate, args.duration, seed=100)
        last = {}
        t0 = time.perf_counter()
        done = iters = 0
        for r in reqs:
            q = pb._finish("req", qps[r.pid].P, r.q, qps[r.pid].A, r.l, r.u)
            x0, y0 = last.get(r.pid, (None, None))
            res = O.solve(q, x0=x0, y0=y0)
            last[r.pid] = (res.x, res.y)
            done += 1
            iters += res.iter
            if time.perf_counter() - t0 > 20.0:
                break
        dt = time.perf_counter() - t0
        print(json.dumps(_reference_line(args, "serve", done / dt, done, dt, iters,
                                         f"first {done} requests of the stream, warm-started, "
                                         f"single thread, {dt:.1f} s", 1)), flush=True)
        return 0
    if args.workload in PARAM_LEN:
        k = args.seq_len or PARAM_LEN[args.workload]
        done, dt, iters = param_oracle(args.workload, k)
        value = done / dt
        print(json.dumps({
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": done,
            "warmup": 0, "ms_per_step": 1e3 * dt / done, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "impl": "reference", "config": {"workload": workload_desc(args, args.workload),
                                             "precision": "fp64", "eps": 1e-3},
            "admm_iter_per_s": iters / dt,
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                             "sample": f"first {done} QPs of the sequence, warm-started, "
                                       f"single thread, {dt:.1f} s"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        }), flush=True)
        return 0
    from oracle import oracle as O
    cfg, desc, qp = build_problem(args, 0)
    for _ in range(args.warmup):
        O.solve(qp)
    t0 = time.perf_counter()
    iters = 0
    for _ in range(args.steps):
        r = O.solve(qp)
        iters += r.iter
    dt = time.perf_counter() - t0
    value = args.steps / dt
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * dt / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "impl": "reference",
        "config": {"workload": desc, "precision": "fp64", "eps": 1e-3},
        "admm_iter_per_s": iters / dt,
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                         "sample": f"{args.steps} full solves of the workload, single thread"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def result_error(qp, x, y, obj, ox, oobj, eps=1e-3):
    """A GPU result against the oracle's solution of the same QP at the same
    ε (objective and x), with the result's own unscaled residuals of §3.4
    beside their tolerances, all computed on the host in FP64."""
    P = qp.P_full()
    Ax, Px, Aty = qp.A @ x, P @ x, qp.A.T @ y
    viol = np.maximum(Ax - qp.u, 0.0) + np.minimum(Ax - qp.l, 0.0)
    z = np.clip(Ax, qp.l, qp.u)
    amax = lambda v: float(np.max(np.abs(v), initial=0.0))
    return {"obj_rel": abs(obj - oobj) / max(1.0, abs(oobj)),
            "x_rel": amax(x - ox) / max(1.0, amax(ox)),
            "prim_res": amax(viol), "eps_prim": eps + eps * max(amax(Ax), amax(z)),
            "dual_res": amax(Px + qp.q + Aty),
            "eps_dual": eps + eps * max(amax(Px), amax(Aty), amax(qp.q))}


def cpu_baseline(args, qp):
    """The oracle timed on the same instance; also returns its last solution
    for the error statement of the GPU result."""
    from oracle import oracle as O
    O.solve(qp)
    t0 = time.perf_counter()
    k = 0
    while True:
        r = O.solve(qp)
        k += 1
        if time.perf_counter() - t0 > 10.0 or k >= 200:
            break
    dt = time.perf_counter() - t0
    return {"value": k / dt, "unit": UNIT, "cores": 1, "kind": "oracle",
            "sample": f"{k} full solves (setup + ADMM) of the same workload instance, "
                      f"{dt:.1f} s, single thread"}, r


def batch_spec(ws):
    """The global batched problem set: 4096 (OSQP_BATCH_COUNT) problems per
    rank, generated from one specification so that any rank can build any
    problem alone."""
    count = int(os.environ.get("OSQP_BATCH_COUNT", "4096"))
    spec = pb.mpc_batch_spec(count * ws, seed=3000)
    return count, spec, [pb.mpc_spec_work(nx, T) for nx, T, _ in spec]


def batch_main(args, ws, rank, local):
    """Batched workload: a step is one cold solve of every problem of this
    rank's share of the batch (Ruiz scaling + ADMM), timed on the device; the
    data (≈ GBs) exceed L2."""
    import torch
    import torch.distributed as dist
    from paper_1711_08013_gb300 import _binding as B
    from paper_1711_08013_gb300 import dist as D
    from paper_1711_08013_gb300.solver import BatchSolver

    torch.cuda.set_device(local)
    if ws > 1:
        D.init("nccl", torch.device("cuda", local))
    dev = torch.device("cuda", local)
    count, spec, weights = batch_spec(ws)
    prec = B.FP64 if args.precision == "fp64" else B.FP32_MIXED
    stream = torch.cuda.Stream()
    sb = D.ShardedBatch(weights, lambda i: pb.mpc(*spec[i][:2], seed=spec[i][2]),
                        lambda qs: BatchSolver(qs, stream=stream.cuda_stream, precision=prec,
                                               autotune=args.autotune),
                        rank=rank, world=ws)
    qps, bs = sb.problems, sb.solver
    local_count = len(qps)
    h = bs.handle
    for _ in range(args.warmup):
        B.osqp_batch_reset(h)
        B.osqp_batch_solve(h)
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(args.steps)]
    sampler = ClockSampler(torch.cuda.current_device())
    if ws > 1:
        dist.barrier()
    torch.cuda.synchronize()
    sampler.start()
    for k in range(args.steps):
        B.osqp_batch_reset(h)
        evs[k][0].record(stream)
        B.osqp_batch_solve_async(h)
        evs[k][1].record(stream)
        stream.synchronize()
    torch.cuda.synchronize()
    clocks = sampler.stop()
    if ws > 1:
        dist.barrier()
    last = [bs.result(i) for i in range(local_count)]
    step_s = [a.elapsed_time(b) * 1e-3 for a, b in evs]
    total = sum(step_s)
    if any(r.status != B.SOLVED for r in last):
        raise SystemExit("a batched solve did not converge")
    iters = sum(r.iter for r in last)
    lat = sorted(r.solve_time for r in last)
    total_max = D.max_over_ranks(total, device=dev)
    solves_all = D.sum_over_ranks(float(local_count * args.steps), device=dev)
    iters_all = D.sum_over_ranks(float(iters), device=dev)
    sv = 8 if prec == B.FP64 else 4
    bytes_launch = sum(admm_bytes(q.n, q.m, q.P_full().nnz + q.A.nnz, q.A.nnz, sv, r.iter,
                                  r.pcg_iters, (r.iter + 24) // 25) for q, r in zip(qps, last))
    t_launch = statistics.mean(step_s)
    peak, peak_src = hbm_peak()
    # end to end through the public API: new q/l/u of every problem from
    # pinned host memory (one whole-batch transfer per vector), the solve,
    # and x, y of every problem back to pinned host memory
    cat = lambda vs: torch.tensor(np.concatenate(vs)).pin_memory()
    q_all, l_all, u_all = cat([q.q for q in qps]), cat([q.l for q in qps]), cat([q.u for q in qps])
    x_all = torch.empty(sum(q.n for q in qps), dtype=torch.float64).pin_memory()
    y_all = torch.empty(sum(q.m for q in qps), dtype=torch.float64).pin_memory()

    def e2e_step():
        B.osqp_batch_update_all(h, q_all.data_ptr(), l_all.data_ptr(), u_all.data_ptr())
        B.osqp_batch_solve(h)
        B.osqp_batch_get_all(h, x_all.data_ptr(), y_all.data_ptr())

    e2e_step()
    e2e_steps = max(1, min(args.steps, 3))
    if ws > 1:
        dist.barrier()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        B.osqp_batch_reset(h)
        e2e_step()
    e2e_dt = D.max_over_ranks(time.perf_counter() - t0, device=dev)
    traffic = (TRAFFIC_BATCH_PER_PROBLEM[args.precision] * local_count
               if args.precision in TRAFFIC_BATCH_PER_PROBLEM else None)
    # the row partitions in use: per shape class the autotuner's measured
    # choice (or the rule's, autotune = 0), counted over this rank's problems
    table = B.osqp_batch_tuning(h)
    chosen = {}
    for i in range(local_count):
        g = B.osqp_batch_schedule(h, i)
        for kind, name in ((0, "Kn"), (1, "A")):
            key = f"{name}:G{g[kind]}"
            chosen[key] = chosen.get(key, 0) + 1
    row_partition = {"chosen_by": "timing" if table else "rule", "shape_classes": len(table),
                     "problems_per_width": dict(sorted(chosen.items()))}
    line = {
        "metric": METRIC, "value": solves_all / total_max, "unit": UNIT, "n_gpus": ws,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total_max / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f64" if prec == B.FP64 else "f32+f64", "data": "synthetic",
        "config": {"workload": WORKLOADS["mpc_batch"][1].replace("4096", str(count)),
                   "precision": args.precision, "eps": 1e-3,
                   "l2": "inputs larger than L2 (no flush)",
                   "parallelism": (f"one set of {count * ws} problems sharded over {ws} GPUs "
                                   "(LPT on estimated work)") if ws > 1 else "single",
                   "row_partition": row_partition},
        "admm_iter_per_s": iters_all / (total_max / args.steps),
        "p50_ms": 1e3 * lat[len(lat) // 2], "p99_ms": 1e3 * lat[int(0.99 * (len(lat) - 1))],
        "admm_iters_per_solve": iters / local_count,
        "pcg_iters_per_solve": sum(r.pcg_iters for r in last) / local_count,
        "roofline": {"bound": "hbm", "kernel": "k_batch", "achieved": bytes_launch / t_launch / 1e9,
                     "peak": peak, "unit": "GB/s", "frac": bytes_launch / t_launch / 1e9 / peak,
                     "traffic": traffic, "peak_source": peak_src,
                     "algorithmic_bytes_per_launch": bytes_launch},
        "e2e": {"value": D.sum_over_ranks(float(local_count * e2e_steps), device=dev) / e2e_dt,
                "unit": UNIT,
                "h2d_bytes_per_step": 8 * sum(q.n + 2 * q.m for q in qps),
                "d2h_bytes_per_step": 8 * sum(q.n + q.m for q in qps)},
        # k_batch every step, plus k_batch_cluster when heavy problems went to
        # clusters (their results report launch 3; the order repeats each step)
        "gpu_launches": args.steps * (1 + int(any(r.launch == 3 for r in last))),
        "clocks": clocks,
    }
    sb.close()
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"], idx, out = batch_cpu_baseline(qps)
        line["oracle_error"] = batch_error(qps, last, idx, out)
    if not args.no_plain:
        # the plain single-problem FP64 form on the same GPU(s), for the
        # batched-vs-plain comparison of the metric
        import copy
        pa = copy.copy(args)
        pa.workload, pa.precision = "lasso", "fp64"
        plain = single_main(pa, ws, rank, local, init_dist=False)
        keep = ("value", "unit", "ms_per_step", "steps", "warmup", "dtype", "config",
                "admm_iter_per_s", "p50_ms", "p99_ms", "admm_iters_per_solve",
                "pcg_iters_per_solve", "roofline", "e2e", "gpu_launches", "clocks",
                "cpu_baseline", "oracle_error")
        line["plain"] = {k: plain[k] for k in keep if k in plain}
        line["batched_over_plain"] = line["value"] / plain["value"]
    if rank == 0:
        print(json.dumps(line), flush=True)
    if ws > 1:
        dist.destroy_process_group()
    return 0


def hbm_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        return float(json.load(open(path))["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def _oracle_solve_one(qp):
    from oracle import oracle as O
    r = O.solve(qp)
    return r.status, r.x, r.obj_val


def _oracle_iters_one(qp):
    from oracle import oracle as O
    r = O.solve(qp)
    return r.iter


def batch_cpu_baseline(qps, budget_s=12.0, sample=256):
    """The oracle on the batch, one problem per process across all host
    cores (spawned pool: safe after CUDA initialisation), in passes over the
    whole batch until about budget_s seconds of wall time; also returns the
    oracle's solutions of an evenly spaced sample for the error statement."""
    import multiprocessing as mp
    from oracle import oracle as O
    O.build()
    idx = list(range(0, len(qps), max(1, len(qps) // sample)))[:sample]
    cores = os.cpu_count() or 1
    ctx = mp.get_context("spawn")
    with ctx.Pool(cores) as pool:
        pool.map(_oracle_iters_one, qps[:cores])  # warm the workers
        out = pool.map(_oracle_solve_one, [qps[i] for i in idx], chunksize=1)
        t0 = time.perf_counter()
        done = 0
        while True:
            pool.map(_oracle_iters_one, qps, chunksize=4)
            done += len(qps)
            if time.perf_counter() - t0 > budget_s:
                break
        dt = time.perf_counter() - t0
    return {"value": done / dt, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"{done // len(qps)} pass(es) over all {len(qps)} batch problems, one "
                      f"problem per process on {cores} cores, {dt:.1f} s"}, idx, out


def batch_error(qps, results, idx, out):
    """Error statement of the batch results on the oracle's sample: the worst
    and median objective and x differences, and the worst residual as a
    fraction of its tolerance."""
    errs = [result_error(qps[i], results[i].x, results[i].y, results[i].obj_val, ox, oobj)
            for i, (_, ox, oobj) in zip(idx, out)]
    med = lambda v: float(statistics.median(v))
    return {"problems": len(errs), "reference": "oracle (FP64, direct method) at the same eps",
            "obj_rel_max": max(e["obj_rel"] for e in errs),
            "obj_rel_median": med([e["obj_rel"] for e in errs]),
            "x_rel_max": max(e["x_rel"] for e in errs),
            "x_rel_median": med([e["x_rel"] for e in errs]),
            "prim_res_over_eps_max": max(e["prim_res"] / e["eps_prim"] for e in errs),
            "dual_res_over_eps_max": max(e["dual_res"] / e["eps_dual"] for e in errs)}


def serve_spec(nmax, seed=4000, pool=256):
    return pb.serving_pool_spec(seed=seed, pool=pool, n_range=(10, nmax))


def serve_problem(entry):
    cls, n, sd = entry
    return pb.random_qp(n, seed=sd) if cls == "random_qp" else pb.huber(n, seed=sd)


def serve_pool(nmax, seed=4000):
    return [serve_problem(e) for e in serve_spec(nmax, seed)]


def serve_work(entry):
    """Estimated matrix entries of a pool problem (random QP: m = 10n rows at
    15%; Huber: 100n × n data at 15% plus the identity blocks)."""
    cls, n, _ = entry
    return 1.5 * n * n if cls == "random_qp" else 15.0 * n * n + 400.0 * n


def serve_main(args, ws, rank, local):
    """Serving workload: the request stream is the step; value = achieved
    solves/s, with offered load, p50/p99 latency (arrival → result on the host)
    and queueing reported beside it.  One global pool of problem IDs is
    sharded across ranks by LPT on estimated work; each rank serves the
    requests of the global stream that name its IDs.  --rates adds a sweep of
    offered rates (each run for --duration seconds) and the highest of them
    at which fewer than 1% of the requests were dropped."""
    import torch
    from paper_1711_08013_gb300 import _binding as B
    from paper_1711_08013_gb300 import dist as D
    from paper_1711_08013_gb300.serve import Server, poisson_requests, shard_requests
    torch.cuda.set_device(local)
    if ws > 1:
        D.init("nccl", torch.device("cuda", local))
    dev = torch.device("cuda", local)
    spec = serve_spec(args.nmax, seed=4000)
    mine = D.shard([serve_work(e) for e in spec], rank, ws)
    local_of = {g: k for k, g in enumerate(mine)}
    qps = [serve_problem(spec[g]) for g in mine]
    prec = B.FP64 if args.precision == "fp64" else B.FP32_MIXED
    slots, large_slots = 32, args.large_slots
    srv = Server(qps, slots=slots, precision=prec, large_slots=large_slots)

    def stream(rate, duration, seed):
        """The global request stream (identical on every rank: the generator
        draws every request's perturbation from one stream, on the sizes of
        other ranks' IDs too), kept for this rank's IDs."""
        shapes = [qps[local_of[g]] if g in local_of else _shape_qp(spec[g])
                  for g in range(len(spec))]
        return shard_requests(poisson_requests(shapes, rate, duration, seed=seed), mine)

    def one(rate, duration, seed):
        reqs = stream(rate, duration, seed)
        st = srv.run(reqs, deadline=duration)
        served = [r for r in reqs if r.t_done == r.t_done]
        offered = D.sum_over_ranks(float(len(reqs)), device=dev)
        done = D.sum_over_ranks(float(st.requests), device=dev)
        dropped = D.sum_over_ranks(float(st.dropped), device=dev)
        wall = D.max_over_ranks(st.wall, device=dev)
        return st, reqs, served, offered, done, dropped, wall

    one(args.rate, min(2.0, args.duration), 1)  # warm-up stream
    sweep = []
    for rate in (args.rates or []):
        st, reqs, served, offered, done, dropped, wall = one(rate, args.duration, 200 + int(rate))
        sweep.append({"offered_req_per_s": rate, "offered": int(offered), "served": int(done),
                      "dropped": int(dropped), "achieved_req_per_s": done / wall,
                      "p50_ms": st.p50_ms, "p99_ms": st.p99_ms,
                      "drop_frac": dropped / max(1.0, offered)})
    sampler = ClockSampler(torch.cuda.current_device())
    sampler.start()
    st, reqs, served, offered, total, dropped, wall = one(args.rate, args.duration, 100)
    clocks = sampler.stop()
    bad = sum(r.status != B.SOLVED for r in served)
    ok_rates = [w["offered_req_per_s"] for w in sweep if w["drop_frac"] < 0.01]
    line = {
        "metric": METRIC, "value": total / wall, "unit": UNIT, "n_gpus": ws, "steps": 1,
        "warmup": 1, "ms_per_step": 1e3 * wall, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64" if prec == B.FP64 else "f32+f64", "data": "synthetic",
        "config": {"workload": workload_desc(args, "serve"),
                   "offered_req_per_s": args.rate, "duration_s": args.duration,
                   "pool": len(spec), "slots": slots, "large_slots": large_slots,
                   "max_batch": None, "precision": args.precision, "eps": 1e-3,
                   "parallelism": (f"pool of {len(spec)} IDs sharded over {ws} GPUs (LPT on "
                                   "estimated work)") if ws > 1 else "single"},
        "p50_ms": st.p50_ms, "p99_ms": st.p99_ms, "mean_queue_ms": st.mean_queue_ms,
        "launches": st.launches, "not_solved": bad, "offered": int(offered),
        "dropped": int(dropped),
        "host_launch_s": st.host_launch_s, "host_result_s": st.host_result_s,
        "mean_iters": float(np.mean([r.iter for r in served])) if served else 0.0,
        "sweep": sweep,
        "max_rate_under_1pct_drop": max(ok_rates) if ok_rates else None,
        "e2e": {"value": total / wall, "unit": UNIT,
                "h2d_bytes_per_step": int(8 * sum(qps[r.pid].n + 2 * qps[r.pid].m for r in served)),
                "d2h_bytes_per_step": int(8 * sum(qps[r.pid].n + 2 * qps[r.pid].m for r in served))},
        "gpu_launches": st.launches, "clocks": clocks,
    }
    srv.close()
    if rank == 0:
        print(json.dumps(line), flush=True)
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return 0


def _shape_qp(entry):
    """Sizes of a pool problem without its matrices: q, l, u of the right
    lengths (the request generator perturbs those)."""
    cls, n, sd = entry
    import types
    m = 10 * n if cls == "random_qp" else 3 * 100 * n
    nn = n if cls == "random_qp" else n + 3 * 100 * n
    return types.SimpleNamespace(n=nn, m=m, q=np.zeros(nn), l=-np.ones(m), u=np.ones(m))


def param_main(args, ws, rank, local):
    """Parametric sequences (§8.4): a step is one QP of the sequence, solved
    in place on the resident data after its update.  value = QPs / summed
    device solve time of the warm-started pass; e2e = QPs / host wall time of
    the same pass (update copies from host memory, solve, x/y read-back); a
    cold pass (zero iterates, ρ̄ reset) over the first QPs gives the
    warm-start time and iteration ratios of the paper's table."""
    import torch
    from paper_1711_08013_gb300 import _binding as B
    from paper_1711_08013_gb300 import dist as D
    from paper_1711_08013_gb300 import parametric as pm
    torch.cuda.set_device(local)
    if ws > 1:
        D.init("nccl", torch.device("cuda", local))
    dev = torch.device("cuda", local)
    prec = B.FP64 if args.precision == "fp64" else B.FP32_MIXED
    K = args.seq_len or PARAM_LEN[args.workload]
    qp, seq = param_problem(args.workload, rank)
    stream = torch.cuda.Stream()
    # warm-up: the first QPs of the sequence on a throwaway session
    with pm.GpuSession(qp, stream=stream.cuda_stream, precision=prec) as s:
        pm.run(s, seq(max(1, args.warmup)))
    sampler = ClockSampler(torch.cuda.current_device())
    trace = []
    if ws > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    with pm.GpuSession(qp, stream=stream.cuda_stream, precision=prec) as s:
        sampler.start()
        t0 = time.perf_counter()
        steps = pm.run(s, seq(K), trace=trace)
        wall = time.perf_counter() - t0
        clocks = sampler.stop()
    if any(st.status != B.SOLVED for st in steps):
        raise SystemExit("a sequence solve did not converge")
    dev_s = sum(st.solve_time for st in steps)
    kc = min(K, 40 if args.workload == "portfolio_bt" else K)
    with pm.GpuSession(qp, stream=stream.cuda_stream, precision=prec) as s:
        cold = pm.run(s, seq(kc), warm=False)
    cold_s = sum(st.solve_time for st in cold) / len(cold)
    ws_s = dev_s / len(steps)
    it_ws = sum(st.iter for st in steps) / len(steps)
    it_cold = sum(st.iter for st in cold) / len(cold)
    dev_max = D.max_over_ranks(dev_s, device=dev)
    sv = 8 if prec == B.FP64 else 4
    nnz_kn = qp.P_full().nnz + qp.A.nnz
    algo = sum(admm_bytes(qp.n, qp.m, nnz_kn, qp.A.nnz, sv, st.iter, st.pcg_iters,
                          (st.iter + 24) // 25) for st in steps)
    peak = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))["hbm_gbs"] if os.path.exists(
        os.path.join(ROOT, "MEASURED_PEAKS.json")) else 6800.0
    h2d = sum(8 * sum(len(np.asarray(v).ravel()) for v in u.values()) for u in trace) / len(trace)
    kernel = "k_admm_grid" if qp.A.nnz + nnz_kn + qp.n + qp.m > 60000 else "k_admm_block"
    line = {
        "metric": METRIC, "value": ws * len(steps) / dev_max, "unit": UNIT, "n_gpus": ws,
        "steps": len(steps), "warmup": args.warmup, "ms_per_step": 1e3 * dev_max / len(steps),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f64" if prec == B.FP64 else "f32+f64", "data": "synthetic",
        "config": {"workload": WORKLOADS[args.workload][1], "precision": args.precision,
                   "eps": 1e-3, "sequence_len": K, "l2": "no flush: successive QPs reuse the "
                   "resident data, as the sequence does"},
        "admm_iter_per_s": sum(st.iter for st in steps) / dev_s,
        "ws_ms_per_qp": 1e3 * ws_s, "cold_ms_per_qp": 1e3 * cold_s, "cold_qps": len(cold),
        "ws_iter_per_qp": it_ws, "cold_iter_per_qp": it_cold,
        "time_improvement": cold_s / ws_s, "iter_improvement": it_cold / it_ws,
        "paper_context": dict(PARAM_PAPER[args.workload], hardware="MIT SuperCloud node with 16 Intel Xeon E5-2650 cores; OSQP with the single-threaded QDLDL direct solver (paper, Sec. 8)"),
        "roofline": {"bound": "hbm", "kernel": kernel, "achieved": algo / dev_s / 1e9,
                     "peak": peak, "unit": "GB/s", "frac": algo / dev_s / 1e9 / peak,
                     "traffic": None, "algorithmic_bytes_per_launch": algo / len(steps)},
        "e2e": {"value": ws * len(steps) / D.max_over_ranks(wall, device=dev), "unit": UNIT,
                "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": 8 * (qp.n + 2 * qp.m)},
        # per QP: the ADMM launch; a vector update adds the refresh launch, a
        # matrix update the two raw-value gathers and the scaling launch
        "gpu_launches": sum(1 + (1 if any(k in u for k in ("q", "l", "u")) else 0)
                            + (3 if ("P_val" in u or "A_val" in u) else 0) for u in trace),
        "clocks": clocks,
    }
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        done, dt, _ = param_oracle(args.workload, K)
        line["cpu_baseline"] = {"value": done / dt, "unit": UNIT, "cores": 1, "kind": "oracle",
                                "sample": f"first {done} QPs of the sequence, warm-started, "
                                          f"single thread, {dt:.1f} s"}
    if rank == 0:
        print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def single_main(args, ws, rank, local, init_dist=True):
    """Single-problem workloads: a step is one whole solve of one QP (data
    reloaded from HBM, scaling, ADMM), L2 flushed between steps.  Returns the
    JSON line (rank 0 prints it when this is the run's workload)."""
    import torch
    import torch.distributed as dist
    from paper_1711_08013_gb300 import _binding as B
    from paper_1711_08013_gb300.solver import Solver

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device")
    from paper_1711_08013_gb300 import dist as D
    torch.cuda.set_device(local)
    if ws > 1 and init_dist:
        D.init("nccl", torch.device("cuda", local))

    cfg, desc, qp = build_problem(args, rank)
    prec = B.FP64 if args.precision == "fp64" else B.FP32_MIXED
    stream = torch.cuda.Stream()
    s = Solver(qp, stream=stream.cuda_stream, precision=prec, autotune=args.autotune,
               launch=args.launch)
    groups = B.osqp_diag_schedule(s.handle)
    n, m = qp.n, qp.m
    dev = torch.device("cuda", local)
    Pv = torch.tensor(qp.P.data, dtype=torch.float64, device=dev)
    Av = torch.tensor(qp.A.data, dtype=torch.float64, device=dev)
    qd = torch.tensor(qp.q, dtype=torch.float64, device=dev)
    ld = torch.tensor(qp.l, dtype=torch.float64, device=dev)
    ud = torch.tensor(qp.u, dtype=torch.float64, device=dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    h = s.handle

    def step():
        B.osqp_load_data_device(h, Pv.data_ptr(), qd.data_ptr(), Av.data_ptr(), ld.data_ptr(),
                                ud.data_ptr())

    with torch.cuda.stream(stream):
        for _ in range(args.warmup):
            step()
            B.osqp_solve_async(h)
        stream.synchronize()
        res = s.result()
        if res.status != B.SOLVED:
            raise SystemExit(f"warm-up solve did not converge: status {res.status}")

        evs = [[torch.cuda.Event(enable_timing=True) for _ in range(3)] for _ in range(args.steps)]
        infos = []
        sampler = ClockSampler(torch.cuda.current_device())
        if ws > 1:
            dist.barrier()
        torch.cuda.synchronize()
        sampler.start()
        for k in range(args.steps):
            flush.fill_(float(k))
            e0, e1, e2 = evs[k]
            e0.record(stream)
            step()
            e1.record(stream)
            B.osqp_solve_async(h)
            e2.record(stream)
            stream.synchronize()
            infos.append(s.result())
        torch.cuda.synchronize()
        clocks = sampler.stop()
        if ws > 1:
            dist.barrier()
    step_s = [evs[k][0].elapsed_time(evs[k][2]) * 1e-3 for k in range(args.steps)]
    admm_s = [evs[k][1].elapsed_time(evs[k][2]) * 1e-3 for k in range(args.steps)]
    total = sum(step_s)
    iters = sum(r.iter for r in infos)
    pcg = sum(r.pcg_iters for r in infos)
    if any(r.status != B.SOLVED for r in infos):
        raise SystemExit("a timed solve did not converge")
    total_max = D.max_over_ranks(total, device=dev)
    iters_all = D.sum_over_ranks(float(iters), device=dev)

    # end to end through the public C ABI with host buffers: pinned host →
    # device copies of every input, the solve, and a device → host read of
    # (x, y), timed on the host clock.
    pin = lambda a: torch.tensor(a, dtype=torch.float64).pin_memory()
    Ph, Ah, qh, lh, uh = pin(qp.P.data), pin(qp.A.data), pin(qp.q), pin(qp.l), pin(qp.u)
    xh, yh = torch.empty(n, dtype=torch.float64).pin_memory(), torch.empty(m, dtype=torch.float64).pin_memory()
    L = B.lib()

    def e2e_step():
        B.osqp_load_data(h, Ph.data_ptr(), qh.data_ptr(), Ah.data_ptr(), lh.data_ptr(), uh.data_ptr())
        B.osqp_solve_async(h)
        rc = L.osqp_get_solution(h, xh.data_ptr(), yh.data_ptr(), None, None)
        if rc != 0:
            raise SystemExit(f"osqp_get_solution failed {rc}")

    for _ in range(args.warmup):
        e2e_step()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        e2e_step()
    torch.cuda.synchronize()
    e2e_dt = D.max_over_ranks(time.perf_counter() - t0, device=dev)

    nnz_kn = qp.P_full().nnz + qp.A.nnz
    sv = 8 if prec == B.FP64 else 4
    K_avg = iters / args.steps
    J_avg = pcg / args.steps
    C_avg = sum((r.iter + 24) // 25 for r in infos) / args.steps
    bytes_launch = admm_bytes(n, m, nnz_kn, qp.A.nnz, sv, K_avg, J_avg, C_avg)
    t_admm = statistics.mean(admm_s)
    peaks_path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(peaks_path):
        peak = json.load(open(peaks_path))["hbm_gbs"]
        peak_src = "measured"
    else:
        peak, peak_src = 6800.0, "fallback"
    achieved = bytes_launch / t_admm / 1e9
    lat = sorted(step_s)
    line = {
        "metric": METRIC,
        "value": ws * args.steps / total_max,
        "unit": UNIT,
        "n_gpus": ws,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": 1e3 * total_max / args.steps,
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f64" if prec == B.FP64 else "f32+f64",
        "data": "synthetic",
        "config": {"workload": desc, "precision": args.precision, "eps": 1e-3,
                   "l2": "flushed between steps (256 MB write outside the timed events)",
                   "parallelism": "replicas" if ws > 1 else "single",
                   "team": {1: "one CTA", 2: "whole-GPU grid", 3: "8-CTA cluster"}.get(
                       infos[-1].launch, str(infos[-1].launch))
                   + (" (library rule)" if args.launch == 0 else " (--launch)"),
                   "row_groups": {"Kn": groups[0], "A": groups[1],
                                  "chosen_by": {1: "timing", 0: "rule"}.get(groups[2], "rule (timing failed)"),
                                  **({"ms_Kn": [round(v, 4) for v in groups[3]],
                                      "ms_A": [round(v, 4) for v in groups[4]]} if groups[2] == 1 else {})}},
        "admm_iter_per_s": iters_all / total_max,
        "p50_ms": 1e3 * lat[len(lat) // 2],
        "p99_ms": 1e3 * lat[min(len(lat) - 1, int(round(0.99 * (len(lat) - 1))))],
        "admm_iters_per_solve": K_avg,
        "pcg_iters_per_solve": J_avg,
        "admm_kernel_ms": 1e3 * t_admm,
        "roofline": {"bound": "hbm",
                     "kernel": {1: "k_admm_block", 2: "k_admm_grid", 3: "k_admm_cluster"}.get(
                         infos[-1].launch, "k_admm_grid"),
                     "achieved": achieved, "peak": peak,
                     "unit": "GB/s", "frac": achieved / peak,
                     "traffic": (TRAFFIC.get((args.workload, args.precision))
                                 if TRAFFIC_GROUPS.get((args.workload, args.precision)) == tuple(groups[:2])
                                 else None),
                     "peak_source": peak_src,
                     "algorithmic_bytes_per_launch": bytes_launch},
        "e2e": {"value": ws * args.steps / e2e_dt, "unit": UNIT,
                "h2d_bytes_per_step": 8 * (qp.P.nnz + qp.A.nnz + n + 2 * m),
                "d2h_bytes_per_step": 8 * (n + m)},
        "gpu_launches": 4 * args.steps,
        "clocks": clocks,
    }
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"], o = cpu_baseline(args, qp)
        g = infos[-1]
        line["oracle_error"] = dict(result_error(qp, g.x, g.y, g.obj_val, o.x, o.obj_val),
                                    reference="oracle (FP64, direct method) at the same eps")
    s.close()
    return line


def main():
    args = parse()
    ws, rank, local = dist_env()
    if args.impl == "reference":
        return run_reference(args, ws, rank)
    if args.workload == "mpc_batch":
        return batch_main(args, ws, rank, local)
    if args.workload == "serve":
        return serve_main(args, ws, rank, local)
    if args.workload in PARAM_LEN:
        return param_main(args, ws, rank, local)
    line = single_main(args, ws, rank, local)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())

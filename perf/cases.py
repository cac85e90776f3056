"""Performance cases: the work that users of this solver have it do, through
the C ABI binding and the thin Python layers over it.

A case is a dict of plain values.  ``kind`` names the call pattern, ``fp32``
picks the FP32-mixed precision mode, the other entries are sizes.  The
problem classes and sizes are those of ``problems.py`` and of the benchmark's
workloads; every problem is generated from the seed.

Row partitions come from the row-length rule (``autotune = 0``, the setting
that gives the same arithmetic on every setup), and batches keep each problem
on one CTA (``launch = 1``), so that a pass does the same arithmetic whenever
and wherever it runs.
"""
import math

import numpy as np

from paper_1711_08013_gb300 import _binding as B
from paper_1711_08013_gb300 import parametric
from paper_1711_08013_gb300 import problems as pb
from paper_1711_08013_gb300.solver import BatchSolver, Solver


def listed():
    return [
        # The smallest serving request: a ten-variable QP solved cold from new
        # host data.  Latency of the one-CTA solver and of the calls around it.
        {"name": "qp_n10", "kind": "solve", "cls": "random", "size": 10, "fp32": False},
        # The single small QP of the benchmark (n = 50, m = 500), in both modes.
        {"name": "qp_n50", "kind": "solve", "cls": "random", "size": 50, "fp32": False},
        {"name": "qp_n50_fp32", "kind": "solve", "cls": "random", "size": 50, "fp32": True},
        # The largest random QP of the measured serving pool, on the whole GPU.
        {"name": "qp_n500", "kind": "solve", "cls": "random", "size": 500, "fp32": False},
        # The benchmark's Lasso QP (20000 × 200 data matrix), in both modes.
        {"name": "lasso_n200", "kind": "solve", "cls": "lasso", "size": 200, "fp32": False},
        {"name": "lasso_n200_fp32", "kind": "solve", "cls": "lasso", "size": 200, "fp32": True},
        # SVM training, 100 features × 10⁴ points.
        {"name": "svm_n100", "kind": "solve", "cls": "svm", "size": 100, "fp32": False},
        # Portfolio optimisation, 10⁴ assets and 100 factors: the longest solve.
        {"name": "portfolio_k100", "kind": "solve", "cls": "portfolio", "size": 100, "fp32": False},
        # Monthly risk-model update of the portfolio back test: new matrix
        # values on the same pattern, scaling and Jacobi diagonal rebuilt.
        {"name": "rescale_k100", "kind": "rescale", "size": 100, "fp32": False},
        # One step of a model predictive controller that has a fixed budget of
        # iterations per sampling period: new initial state, previous solution
        # as the starting point.
        {"name": "mpc_step_nx80", "kind": "mpc_step", "size": 80, "fp32": False},
        # Ragged batch of MPC problems with new data for each, in the mode of
        # the benchmark's batched workload.
        {"name": "mpc_batch_608_fp32", "kind": "mpc_batch", "size": 608, "fp32": True},
        # A burst of serving requests: the small ones in one launch, each large
        # one on a slot of its own, warm-started from the pool's last solutions.
        {"name": "serve_24", "kind": "serve", "size": 24, "fp32": False},
    ]


def draw(rng):
    kind = rng.choice(["random", "random", "lasso", "svm", "portfolio", "rescale", "mpc_step",
                       "mpc_batch", "serve"])
    logu = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    fp32 = rng.random() < 0.4
    if kind == "random":
        return {"kind": "solve", "cls": "random", "size": logu(10, 500), "fp32": fp32}
    if kind == "lasso":
        return {"kind": "solve", "cls": "lasso", "size": logu(20, 200), "fp32": fp32}
    if kind == "svm":
        return {"kind": "solve", "cls": "svm", "size": logu(15, 100), "fp32": fp32}
    if kind == "portfolio":
        return {"kind": "solve", "cls": "portfolio", "size": rng.randint(45, 85), "fp32": False}
    if kind == "rescale":
        return {"kind": "rescale", "size": logu(5, 100), "fp32": fp32}
    if kind == "mpc_step":
        return {"kind": "mpc_step", "size": rng.randint(12, 80), "fp32": False}
    if kind == "mpc_batch":
        return {"kind": "mpc_batch", "size": logu(20, 600), "fp32": fp32}
    return {"kind": "serve", "size": rng.randint(6, 24), "fp32": False}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
MPC_BUDGET = 25  # iterations per sampling period: one check interval


def _solve_problem(case, seed):
    n = int(case["size"])
    if case["cls"] == "random":
        return pb.random_qp(n, 10 * n, seed=seed)
    if case["cls"] == "lasso":
        return pb.lasso(n, seed=seed)
    if case["cls"] == "svm":
        return pb.svm(n, seed=seed)
    return pb.portfolio(n, seed=seed)


def _portfolio_update(qp, seed):
    """New risk model of the back test: (P values, A values), same pattern."""
    seq = parametric.portfolio_backtest(qp, days=2, days_per_month=1, seed=seed)
    next(seq)
    upd = next(seq)
    return upd["P_val"], upd["A_val"]


def _mpc_shift(qp, x):
    """Previous primal solution moved one period on: the start of the next step."""
    nx, nu, T = qp.meta["nx"], qp.meta["nu"], qp.meta["T"]
    xs, us = x[:nx * (T + 1)], x[nx * (T + 1):]
    return np.concatenate([xs[nx:], xs[-nx:], us[nu:], us[-nu:]])


def _serve_sizes(case):
    # n ~ logU[10, 500], stratified so that every burst spans the range; the
    # sizes belong to the case, the problems to the seed
    count = int(case["size"])
    rng = np.random.default_rng(count)
    lo, hi = math.log(10.0), math.log(500.0)
    return [int(round(math.exp(lo + (hi - lo) * (k + rng.random()) / count)))
            for k in range(count)]


def _serve_pool(case, seed):
    return [pb.random_qp(n, 10 * n, seed=seed + 1 + k)
            for k, n in enumerate(_serve_sizes(case))]


def _serve_requests(qps, seed):
    """Two rounds of requests, one per problem of the pool."""
    rng = np.random.default_rng(seed + 7)
    return [[pb.perturb_vectors(rng, qp) for qp in qps] for _ in range(2)]


def prepare(case, seed):
    prec = B.FP32_MIXED if case["fp32"] else B.FP64
    kind = case["kind"]
    if kind == "solve":
        qp = _solve_problem(case, seed)
        return {"kind": kind, "qp": qp, "solver": Solver(qp, precision=prec, autotune=0)}
    if kind == "rescale":
        qp = pb.portfolio(int(case["size"]), seed=seed)
        P_val, A_val = _portfolio_update(qp, seed)
        return {"kind": kind, "solver": Solver(qp, precision=prec, autotune=0),
                "P_val": P_val, "A_val": A_val}
    if kind == "mpc_step":
        qp = pb.mpc_paper(int(case["size"]), T=10, seed=seed)
        with Solver(qp, precision=prec, autotune=0, max_iter=4 * MPC_BUDGET) as first:
            r = first.solve()
        nx = qp.meta["nx"]
        x1 = r.x[nx:2 * nx] + 0.01 * np.random.default_rng(seed).standard_normal(nx)
        l, u = qp.l.copy(), qp.u.copy()
        l[:nx] = -x1
        u[:nx] = -x1
        return {"kind": kind, "l": l, "u": u, "x": _mpc_shift(qp, r.x), "y": r.y,
                "solver": Solver(qp, precision=prec, autotune=0, max_iter=MPC_BUDGET)}
    if kind == "mpc_batch":
        count = int(case["size"])
        qps = [pb.mpc(nx, T, seed=seed + 1 + i)  # the workload's sizes, this seed's problems
               for i, (nx, T, _) in enumerate(pb.mpc_batch_spec(count))]
        rng = np.random.default_rng(seed)
        vecs = [pb.perturb_vectors(rng, qp, 0.02) for qp in qps]
        batch = BatchSolver(qps, precision=prec, autotune=0, launch=1)
        return {"kind": kind, "batch": batch,
                "q": np.concatenate([v[0] for v in vecs]),
                "l": np.concatenate([v[1] for v in vecs]),
                "u": np.concatenate([v[2] for v in vecs])}
    qps = _serve_pool(case, seed)
    batch = BatchSolver(qps, precision=prec, autotune=0)
    large = [i for i in range(len(qps)) if B.osqp_batch_uses_cluster(batch.handle, i)]
    small = [i for i in range(len(qps)) if i not in set(large)]
    launches = [small] + [[i] for i in large]
    # every slot's stream and buffers come with its first launch, and the
    # pool's first solutions with it: a large problem opens each slot (the top
    # of the size range is always large), then the small ones share slot 0
    for slot, ids in enumerate([[large[0]]] + launches[1:] + [small]):
        slot %= len(launches)
        B.osqp_batch_launch(batch.handle, slot, ids)
        B.osqp_batch_slot_wait(batch.handle, slot)
    return {"kind": kind, "batch": batch, "rounds": _serve_requests(qps, seed), "next": 0,
            "launches": launches}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "solve":  # new host data, cold solve, solution back on the host
        s, qp = state["solver"], state["qp"]
        B.osqp_load_data(s.handle, qp.P.data, qp.q, qp.A.data, qp.l, qp.u)
        r = s.solve()
        return {"x": r.x, "y": r.y, "z": r.z, "status": r.status}
    if kind == "rescale":
        s = state["solver"]
        s.update_matrices(state["P_val"], state["A_val"])
        D, E, c, jac = s.scaling()
        return {"D": D, "E": E, "c": c, "jacobi": jac}
    if kind == "mpc_step":
        s = state["solver"]
        s.update_rho(s.settings.rho)
        s.update_vectors(l=state["l"], u=state["u"])
        s.warm_start(state["x"], state["y"])
        r = s.solve()
        return {"x": r.x, "y": r.y, "z": r.z, "status": r.status}
    if kind == "mpc_batch":
        b = state["batch"]
        b.reset()
        B.osqp_batch_update_all(b.handle, state["q"], state["l"], state["u"])
        b.solve()
        x = np.empty(sum(n for n, _ in b.sizes))
        y = np.empty(sum(m for _, m in b.sizes))
        B.osqp_batch_get_all(b.handle, x, y)
        return {"x": x, "y": y}
    b = state["batch"]
    req = state["rounds"][state["next"]]
    state["next"] ^= 1
    for slot, ids in enumerate(state["launches"]):
        B.osqp_batch_launch(b.handle, slot, ids, [req[i][0] for i in ids], [req[i][1] for i in ids],
                            [req[i][2] for i in ids])
    for slot in range(len(state["launches"])):
        B.osqp_batch_slot_wait(b.handle, slot)
    res = [b.result(i) for i in range(len(b.sizes))]
    return {"x": [r.x for r in res], "y": [r.y for r in res]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _solve_sizes(case):
    """(n, m, expected nonzeros of upper P, of A) of a single problem."""
    k = float(case["size"])
    cls = case.get("cls")
    if cls == "random":
        p = 1.0 - (1.0 - 0.15 ** 2) ** k  # density of M Mᵀ
        return k, 10 * k, k + p * k * (k - 1) / 2, 0.15 * 10 * k * k
    if cls == "lasso":
        return 102 * k, 102 * k, 100 * k, 0.15 * 100 * k * k + 104 * k
    if cls == "svm":
        return 101 * k, 200 * k, k, 0.15 * 100 * k * k + 200 * k
    if case["kind"] == "mpc_step":
        nx, nu, T = k, k // 2, 10
        n = nx * (T + 1) + nu * T
        return n, nx * (T + 1) + n, 0.7 * nx * T + nx * (nx + 1) / 2 + nu * T, \
            T * nx * (nx + nu + 1) + nx + n
    return 101 * k, 101 * k + 1, 101 * k, 0.5 * 100 * k * k + 201 * k  # portfolio


def _matrix_work(n, m, p, a):
    """(bytes of values, indices and vectors in and out; operations of the
    products of one check interval with one linear-solver step each)."""
    nbytes = 12 * (p + a) + 4 * (2 * n + 2) + 8 * (n + 2 * m) + 8 * (n + 2 * m)
    return nbytes, 25 * 2 * (2 * p + 2 * a)


def work(case):
    kind = case["kind"]
    if kind == "mpc_batch":
        probs = []
        for nx, T, _ in pb.mpc_batch_spec(int(case["size"])):
            nu = nx // 2
            n = nx * (T + 1) + nu * T
            probs.append((n, nx * (T + 1) + n, 0.1 * nx * (T + 1) + nu * T,
                          T * nx * (nx + nu + 1) + nx + n))
    elif kind == "serve":
        probs = [_solve_sizes({"kind": "solve", "cls": "random", "size": n})
                 for n in _serve_sizes(case)]
    else:
        probs = [_solve_sizes(case)]
    total = [_matrix_work(*p) for p in probs]
    if kind == "rescale":  # matrices in, scaling out; two products' worth of passes
        n, m, p, a = probs[0]
        return {"bytes": 8 * (p + a) + 4 * (p + a + 2 * n + 2) + 8 * (2 * n + m), "flops": 8 * (p + a)}
    return {"bytes": sum(t[0] for t in total), "flops": sum(t[1] for t in total)}


# ---------------------------------------------------------------------------
# the same in 64 bits without the library
# ---------------------------------------------------------------------------
def _optimum(qp, q=None, l=None, u=None):
    """(x, z) of a small QP's minimiser: Algorithm 1 with dense direct solves,
    run to 1e-11."""
    P, A = qp.P_full().toarray(), qp.A.toarray()
    q, l, u = (v if w is None else w for v, w in ((qp.q, q), (qp.l, l), (qp.u, u)))
    n, m = P.shape[0], A.shape[0]
    x, z, y = np.zeros(n), np.zeros(m), np.zeros(m)
    eq = np.where(l == u, 1e3, 1.0)
    rho, inv = 0.1, None
    for k in range(1, 20001):
        if inv is None:
            r = rho * eq
            inv = np.linalg.inv(P + 1e-6 * np.eye(n) + A.T @ (r[:, None] * A))
        xt = inv @ (1e-6 * x - q + A.T @ (r * z - y))
        v = 1.6 * (A @ xt) - 0.6 * z + y / r
        x = 1.6 * xt - 0.6 * x
        z = np.clip(v, l, u)
        y = r * (v - z)
        if k % 50 == 0:
            ax, px, aty = A @ x, P @ x, A.T @ y
            rp, rd = np.abs(ax - z).max(), np.abs(px + q + aty).max()
            if max(rp, rd) < 1e-11:
                break
            ratio = math.sqrt(rp * max(np.abs(px).max(), np.abs(aty).max(), np.abs(q).max())
                              / max(rd * max(np.abs(ax).max(), np.abs(z).max()), 1e-300))
            if k % 200 == 0 and not 0.2 < ratio < 5.0:
                rho, inv = rho * min(max(ratio, 1e-2), 1e2), None
    return x, z


def _lasso_optimum(qp):
    """(x, z) of the Lasso's minimiser by coordinate descent on the normal
    equations."""
    nf, md, lam = qp.meta["n_feat"], qp.meta["m_data"], qp.meta["lam"]
    Ad = qp.A[:md, :nf].toarray()
    b = qp.l[:md]
    G, g = Ad.T @ Ad, Ad.T @ b
    w = np.zeros(nf)
    grad = -g.copy()  # Gw − g
    for _ in range(2000):
        moved = 0.0
        for j in range(nf):
            t = w[j] - grad[j] / G[j, j]
            new = math.copysign(max(abs(t) - 0.5 * lam / G[j, j], 0.0), t)
            if new != w[j]:
                grad += G[:, j] * (new - w[j])
                moved = max(moved, abs(new - w[j]))
                w[j] = new
        if moved < 1e-15:
            break
    x = np.concatenate([w, Ad @ w - b, np.abs(w)])
    return x, np.asarray(qp.A @ x)


def _ruiz(qp, P_val, A_val, rho):
    """Modified Ruiz scaling and the Jacobi diagonal on the entry lists."""
    n, m = qp.n, qp.m
    pc, ac = (np.repeat(np.arange(n), np.diff(M.indptr)) for M in (qp.P, qp.A))
    pr, ar = qp.P.indices, qp.A.indices
    off = pr != pc  # the other triangle
    pr, pc = np.concatenate([pr, pc[off]]), np.concatenate([pc, pr[off]])
    pv, av = np.abs(np.concatenate([P_val, P_val[off]])), np.abs(A_val)
    D, E, c = np.ones(n), np.ones(m), 1.0

    def colmax(size, at, v):
        out = np.zeros(size)
        np.maximum.at(out, at, v)
        return out

    def delta(nrm):
        return np.where(nrm == 0.0, 1.0, 1.0 / np.sqrt(np.clip(nrm, 1e-4, 1e4)))

    for _ in range(10):
        sa = E[ar] * av * D[ac]
        dn = delta(np.maximum(colmax(n, pc, c * D[pr] * pv * D[pc]), colmax(n, ac, sa)))
        dm = delta(colmax(m, ar, sa))
        D, E = D * dn, E * dm
        mean = colmax(n, pc, c * D[pr] * pv * D[pc]).mean()
        qn = np.abs(c * D * qp.q).max()
        mean, qn = (1.0 if v < 1e-4 else v for v in (mean, qn))
        c /= min(max(mean, qn, 1e-4), 1e4)
        if max(np.abs(1.0 - dn).max(), np.abs(1.0 - dm).max() if m else 0.0) <= 1e-3:
            break
    r = np.where(qp.l == qp.u, 1e3 * rho, rho)
    jac = np.zeros(n)
    on = pr == pc
    signed = np.concatenate([P_val, P_val[off]])
    np.add.at(jac, pc[on], (c * D[pr] * signed * D[pc])[on])
    np.add.at(jac, ac, r[ar] * (E[ar] * A_val * D[ac]) ** 2)
    return {"D": D, "E": E, "c": float(c), "jacobi": jac + 1e-6}


def exact(case, seed):
    """The minimiser for small QPs and the Lasso, the scaling for matrix
    updates.  At the default tolerance multipliers are only determined to
    several per cent on some problems, so they have no value here; nor have
    large QPs without a closed form, degenerate ones, and solves stopped by a
    budget."""
    kind = case["kind"]
    if kind == "rescale":
        qp = pb.portfolio(int(case["size"]), seed=seed)
        return _ruiz(qp, *_portfolio_update(qp, seed), rho=0.1)
    if kind == "solve" and case["cls"] == "lasso":
        x, z = _lasso_optimum(_solve_problem(case, seed))
        return {"x": x, "y": None, "z": z, "status": None}
    if kind == "solve" and case["cls"] == "random" and case["size"] <= 150:
        x, z = _optimum(_solve_problem(case, seed))
        return {"x": x, "y": None, "z": z, "status": None}
    if kind == "serve":
        qps = _serve_pool(case, seed)
        return {"x": [_optimum(qp, *req)[0] if qp.n <= 60 else None
                      for qp, req in zip(qps, _serve_requests(qps, seed)[0])],
                "y": [None] * len(qps)}
    return None

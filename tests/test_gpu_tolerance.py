"""The PCG tolerance of an FP64 solve is the same number whether ‖b‖∞ was formed
or only bounded: the bound's column sum belongs to the matrices in force."""
import dataclasses

import numpy as np
import pytest

from paper_1711_08013_gb300 import _binding as B
from paper_1711_08013_gb300 import problems as pb

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_08013_gb300.solver import BatchSolver, Solver  # noqa: E402

RUN = dict(autotune=0, check_interval=5, max_iter=100, eps_abs=1e-12, eps_rel=0.0,
           eps_pinf=1e-300, eps_dinf=1e-300)


def assert_same_bits(a, b):
    assert (a.iter, a.pcg_iters, a.rho_updates) == (b.iter, b.pcg_iters, b.rho_updates)
    for v in ("x", "y", "z"):
        assert np.array_equal(getattr(a, v), getattr(b, v)), v


@pytest.mark.parametrize("launch", [1, 2, 3], ids=["block", "grid", "cluster"])
@pytest.mark.parametrize("floor", [1e-4, 1e-3, 1e-2, 1e-1])
def test_column_sum_follows_the_matrices(floor, launch):
    """New matrices with far larger scaled column sums in a solver that has
    solved the old ones: the solve of a solver set up on them."""
    new = pb.random_qp(20, 200, seed=8)
    small = new.A.copy()
    small.data = np.where(np.random.default_rng(9).random(small.nnz) < 0.9, 1e-4, 1.0) * small.data
    old = dataclasses.replace(new, A=small)
    with Solver(new, launch=launch, pcg_tol_floor=floor, **RUN) as s:
        want = s.solve()
    with Solver(old, launch=launch, pcg_tol_floor=floor, **RUN) as s:
        s.solve()
        B.osqp_load_data(s.handle, new.P.data, new.q, new.A.data, new.l, new.u)
        assert_same_bits(s.solve(), want)


def weak_cost(qp):
    """q scaled down, so that Āᵀ(Rz − y) dominates b."""
    return dataclasses.replace(qp, q=1e-3 * qp.q)


PROBLEMS = {
    "random": lambda: weak_cost(pb.random_qp(20, 200, seed=1)),
    "random_n50": lambda: pb.random_qp(50, 500, seed=2),
    "control": lambda: weak_cost(pb.mpc_paper(4, T=10, seed=3)),
    "svm": lambda: pb.svm(3, seed=4),
    "lasso": lambda: pb.lasso(2, seed=5),
}


@pytest.mark.parametrize("floor", [0.0, 1e-8, 1e-6, 1e-5, 1e-4, 1e-3, 1e-2, 1e-1])
@pytest.mark.parametrize("name", PROBLEMS)
def test_bounded_b_gives_the_tolerance_of_b(name, floor):
    """A single one-CTA solve may leave b out of the restart residual, the
    batch kernel always forms it.  The floors lie on both sides of κ times the
    residuals: with a bound that were too small the first would stop PCG at
    another tolerance than the second."""
    qp = PROBLEMS[name]()
    with Solver(qp, launch=1, pcg_tol_floor=floor, **RUN) as s:
        one = s.solve()
    with BatchSolver([qp], launch=1, pcg_tol_floor=floor, **RUN) as b:
        b.solve()
        assert_same_bits(one, b.result(0))

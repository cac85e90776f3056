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

from paper_1711_08013_gb300.solver import Solver  # noqa: E402

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

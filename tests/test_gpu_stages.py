"""Stages of the solve at the edges of their rules: the numbering of the
whole-GPU team's warps, the tolerance without ‖b‖∞, the scaling passes."""
import numpy as np
import pytest

from paper_1711_08013_gb300 import problems as pb

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_08013_gb300.solver import Solver  # noqa: E402

STEP = dict(adaptive_rho=0, eps_abs=0.0, eps_rel=0.0, eps_pinf=1e-300, eps_dinf=1e-300,
            check_interval=1, max_iter=7)


def rel_err(a, b):
    return np.max(np.abs(a - b), initial=0.0) / max(1.0, np.max(np.abs(b), initial=0.0))


def half_warps():
    return torch.cuda.get_device_properties(0).multi_processor_count * 16 // 2


# Kn of a box QP has two nonzeros a row and 16 rows a slice (group width 2):
# 16·half rows fill exactly half as many slices as there are warps.
CASES = {
    "box_at_half": lambda: pb.box_qp(16 * half_warps(), seed=1),
    "box_over_half": lambda: pb.box_qp(16 * half_warps() + 1, seed=2),
    "one_row": lambda: pb.box_qp(1, seed=3),
    "whole_warp_rows": lambda: pb.random_qp(150, 450, seed=4),
    "long_rows": lambda: pb.svm(4, seed=5),
}


@pytest.mark.parametrize("name", CASES)
def test_step_parity_on_the_grid(oracle_mod, name):
    """Exact linear solves, fixed ρ: the iterates are the oracle's to 1e-8
    (PCG residual 1e-14 relative, condition numbers below 1e6)."""
    qp = CASES[name]()
    o = oracle_mod.solve(qp, **STEP)
    with Solver(qp, launch=2, autotune=0, pcg_tol_fraction=0.0, pcg_tol_floor=1e-14,
                pcg_max_iter=2000, **STEP) as s:
        g = s.solve()
    assert g.iter == 7
    assert rel_err(g.x, o.x) <= 1e-8 and rel_err(g.z, o.z) <= 1e-8 and rel_err(g.y, o.y) <= 1e-8


@pytest.mark.parametrize("launch", [1, 2, 3], ids=["block", "grid", "cluster"])
@pytest.mark.parametrize("name", ["lasso", "random"])
def test_tolerance_floor_is_kept_when_b_is_left_out(name, launch):
    """A PCG floor of 10³‖b‖∞ is above the first residual (x̃ = 0, r⁰ = b) in
    every iteration, before and after checks: no PCG iteration may run,
    whether ‖b‖∞ was formed or only bounded."""
    qp = pb.lasso(5, seed=6) if name == "lasso" else pb.random_qp(20, 90, seed=7)
    with Solver(qp, launch=launch, pcg_tol_floor=1e3, check_interval=5, max_iter=60,
                eps_abs=1e-9, eps_rel=1e-9, eps_pinf=1e-300, eps_dinf=1e-300) as s:
        g = s.solve()
    assert g.iter == 60 and g.pcg_iters == 0


@pytest.mark.parametrize("launch", [1, 2], ids=["block", "grid"])
@pytest.mark.parametrize("passes", [0, 1, 2, 10])
def test_scaling_after_a_number_of_passes(oracle_mod, passes, launch):
    """D, E and c after the last pass, whose cost factor needs one more product
    than its norms: the oracle's to 1e-12."""
    qp = pb.portfolio(3, seed=5)
    want = oracle_mod.ruiz(qp.P_full(), qp.q, qp.A, qp.l, qp.u, scaling_iters=passes)
    with Solver(qp, launch=launch, scaling_iters=passes) as s:
        D, E, c, _ = s.scaling()
    assert rel_err(D, want["D"]) <= 1e-12 and rel_err(E, want["E"]) <= 1e-12
    assert abs(c - want["c"]) <= 1e-12 * want["c"]

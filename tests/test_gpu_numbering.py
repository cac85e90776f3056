"""The grouping of the PCG's inner products is part of a solve's result: a sum
of the same terms in another order moves it by a rounding, and a long run of
conjugate gradients amplifies that.  The numbering of a team's warps therefore
has to leave the terms of one CTA's partial sum together.  Where all rows of
both matrices fit the warps of one CTA, that makes the whole-GPU and the
cluster team's partial sums those of the one-CTA team, and every bit of the
FP64 iterates with them."""
import ctypes as C

import numpy as np
import pytest
import scipy.sparse as sp

from paper_1711_08013_gb300 import _binding as B
from paper_1711_08013_gb300 import problems as pb

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_08013_gb300.solver import Solver  # noqa: E402

CTA_WARPS = 16


def long_row_qp():
    """One variable in all 256 constraints and in a dense row of P: its row of
    [P Aᵀ] has 276 nonzeros, two chunks."""
    n, m = 20, 256
    rng = np.random.default_rng(11)
    M = np.diag(2.0 + rng.random(n))
    M[0, 1:] = 0.05 * rng.standard_normal(n - 1)
    rows = np.arange(m)
    A = sp.csc_matrix((rng.standard_normal(2 * m),
                       (np.concatenate([rows, rows]),
                        np.concatenate([np.zeros(m, int), 1 + rows % (n - 1)]))), shape=(m, n))
    mid = A @ rng.standard_normal(n)
    return pb._finish("long_row", M + M.T, rng.standard_normal(n), A, mid - 0.3 * rng.random(m),
                      mid + 0.3 * rng.random(m))


PROBLEMS = {
    "all_warps": lambda: pb.mpc_paper(4, T=10, seed=1),  # 16 slices of Kn
    "nine_warps": lambda: pb.mpc_paper(3, T=8, seed=2),
    "whole_warp_rows": lambda: pb.random_qp(10, 100, seed=3),
    "quarter_warp_rows": lambda: pb.svm(1, seed=4),
    "long_row": long_row_qp,
}


def partition(M, nwarps):
    """(group, long-row threshold, slices, positions, long rows, chunks)."""
    f = B.lib().osqp_diag_sliced_layout
    rp = np.ascontiguousarray(M.indptr, dtype=np.int32)
    stats = np.zeros(6, dtype=np.int32)
    assert f(C.c_int32(M.shape[0]), C.c_void_p(rp.ctypes.data), C.c_int64(nwarps), None, None,
             C.c_void_p(stats.ctypes.data)) == B.OSQP_OK
    return tuple(int(v) for v in stats)


@pytest.mark.parametrize("launch", [2, 3], ids=["grid", "cluster"])
@pytest.mark.parametrize("name", PROBLEMS)
def test_teams_give_the_bits_of_one_cta(name, launch):
    qp = PROBLEMS[name]()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    warps = CTA_WARPS * (sms if launch == 2 else 8)
    for M in (sp.hstack([qp.P_full(), qp.A.T]).tocsr(), qp.A.tocsr()):
        part = partition(M, CTA_WARPS)
        assert part == partition(M, warps) and part[2] <= CTA_WARPS and part[5] <= CTA_WARPS
        assert part[4] == (1 if name == "long_row" and M.shape[0] == qp.n else 0)
    res = []
    for team in (1, launch):
        with Solver(qp, launch=team, autotune=0, max_iter=100, eps_abs=1e-12, eps_rel=0.0) as s:
            res.append(s.solve())
    one, many = res
    assert (many.iter, many.pcg_iters, many.status) == (one.iter, one.pcg_iters, one.status)
    for v in ("x", "y", "z"):
        assert np.array_equal(getattr(many, v), getattr(one, v)), v

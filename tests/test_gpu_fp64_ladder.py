"""FP64 solves of LPs whose optimum is a face end as they do in FP64 arithmetic.

In their last iterations pivots are clamped, and a direction from a factor with digit
updates can stall at a residual that passes as an inexact Newton step.  Such steps sent
the iterates off where FP64 arithmetic converges, so a stalled direction first gets a
factor in FP64 arithmetic.  With FP64 arithmetic throughout, 200 such LPs took at most 11
iterations each; one more is allowed for."""
import numpy as np
import pytest

from instances import random_block_lp
from oracle import lp as olp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", range(24))
def test_degenerate_solve_converges(seed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2412_07731_gb300 as P
    r = np.random.default_rng(seed)
    N = int(r.integers(2, 5))
    m = [int(v) for v in r.integers(70, 260, N)]
    lp = random_block_lp(seed, N=N, m_sizes=m, n_sizes=[3 * v // 2 for v in m], nnz_per_col=8,
                         n0=int(r.integers(4, 200)), w_density=0.05, l=int(r.integers(1, 8)),
                         mg=int(r.integers(0, 9)), plant="half_zero")
    A, b, c = olp.assemble(lp)
    prob = P.arrowhead_lp_create(lp, P.default_options(max_correctors=0, max_iter=40))
    (x, y, z), res = P.ipm_solve(prob)
    prob.close()
    assert res["status"] == 0 and res["iterations"] <= 12, res
    meas = olp.measures(A, b, c, x, y, z)
    assert meas["pinf"] <= 1e-8 and meas["dinf"] <= 1e-8 and meas["gap"] <= 1e-8, meas

"""The Schur-complement solve without refinement (refine_max = 0, no
regularisation): block solves, link-chain levels with several lanes per row, and
the border through the explicit inverse of its factor, at border orders around
the 64-column tiles and link counts around the 32 rows a chain CTA takes at once.

The points are mild (x, z in e^+-1), so the Newton matrix has a condition number
well below 1e6, and a direction computed through backward-stable FP64 stages has
a relative residual of about u times that times the growth of an explicit inverse
of order 64 tiles: 1e-9 leaves a factor of ten.
"""
import numpy as np
import pytest

from instances import random_block_lp
from oracle import lp as olp
from oracle import newton as onewton

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2412_07731_gb300 as P
    return P


@pytest.mark.parametrize("n0,mg,l", [(1, 0, 1), (63, 1, 5), (64, 2, 33), (65, 3, 32), (130, 0, 40),
                                     (0, 70, 3), (300, 5, 2)])
def test_direction_from_the_factor_alone(P, n0, mg, l):
    lp = random_block_lp(31, N=6, m_sizes=[90, 140, 120, 100, 130, 110],
                         n_sizes=[200, 260, 240, 220, 280, 230], nnz_per_col=5, n0=n0,
                         w_density=0.1, l=l, mg=mg, global_nnz=6, plant=None)
    lp.b = [np.zeros(a.shape[0]) for a in lp.A]
    lp.c = [np.zeros(a.shape[1]) for a in lp.A]
    lp.blink = [np.zeros(int(v)) for v in lp.l]
    A, _, _ = olp.assemble(lp)
    rng = np.random.default_rng(7)
    n, m = A.shape[1], A.shape[0]
    x, z = np.exp(rng.uniform(-1, 1, n)), np.exp(rng.uniform(-1, 1, n))
    r = rng.standard_normal(n), rng.standard_normal(m), rng.standard_normal(n)
    prob = P.arrowhead_lp_create(lp, P.default_options(refine_max=0))
    P.kkt_factor(prob, x, z, 0.0, 0.0)
    for solve in (P.kkt_solve, P.kkt_adjoint_solve):
        (dx, dy, dz), info = solve(prob, *r)
        assert info["refine_steps"] == 0
        if solve is P.kkt_solve:
            res = onewton.relative_residual(A, x, z, dx, dy, dz, *r)
        else:   # J' lam = g
            e = (A.T @ dy + z * dz - r[0], A @ dx - r[1], dx + x * dz - r[2])
            res = np.linalg.norm(np.concatenate(e)) / np.linalg.norm(np.concatenate(r))
        assert res <= 1e-9, res
        # the library's own residual is the same quantity
        assert abs(info["rel_residual"] - res) <= 0.05 * res + 1e-14
    prob.close()


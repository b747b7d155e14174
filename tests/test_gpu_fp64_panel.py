"""The FP64 panel kernel's lane layouts and the FP64 update's tile splits, which
the number of tiles of a step chooses.  A panel entry is one chain of multiply-adds
in every layout, so the bound of Cholesky in FP64 arithmetic holds as for the
tensor-core updates' test; the border's factor (FP64 updates, one to three panel
tiles) is checked through a refined direction, whose residual it preconditions."""
import numpy as np
import pytest

from instances import random_block_lp
from test_gpu_fp64_digits import P, _check  # noqa: F401

pytestmark = pytest.mark.gpu

# panel tiles of the first step: up to 38 (8 lanes per row), 76 (4) and more (2)
SETS = {"8 lanes": [65, 100, 129, 191], "4 lanes": [321, 449, 500] * 3,
        "2 lanes": [577, 640, 705] * 4}


@pytest.mark.parametrize("sizes", SETS.values(), ids=SETS.keys())
def test_backward_error(P, sizes):  # noqa: F811
    lp = random_block_lp(3, N=len(sizes), m_sizes=sizes, n_sizes=[2 * v for v in sizes],
                         nnz_per_col=4, n0=7, w_density=0.3, l=2, mg=3, global_nnz=3)
    _check(P, lp, 2, 2.0, blocks=(0, 1, len(sizes) - 1))


@pytest.mark.parametrize("n0,mg", [(64, 1), (70, 63), (150, 65), (700, 3)])
def test_border_factor(P, n0, mg):  # noqa: F811
    lp = random_block_lp(4, N=4, m_sizes=[230] * 4, n_sizes=[900] * 4, nnz_per_col=4, n0=n0,
                         w_density=0.2, l=2, mg=mg, global_nnz=40)
    rng = np.random.default_rng(2)
    n = lp.n_total
    x, z = np.exp(rng.uniform(-1, 1, n)), np.exp(rng.uniform(-1, 1, n))
    prob = P.arrowhead_lp_create(lp, P.default_options(refine_max=3))
    P.kkt_factor(prob, x, z)
    rhs = rng.standard_normal(n), rng.standard_normal(prob.m), rng.standard_normal(n)
    _, info = P.kkt_solve(prob, *rhs)
    # an unrefined FP64 factor of a system with condition near 1e4 leaves 1e-11 at
    # worst; three steps reach the tolerance with room
    assert info["rel_residual"] <= 1e-11
    prob.close()

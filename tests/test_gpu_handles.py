"""Handles side by side: what one handle sets up must not change what another one
can do.  The link chain's kernels take shared memory by the link count, up to 96
rows; the limit is the kernel's, shared by every handle of the process."""
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


@pytest.mark.parametrize("l", [40, 96])
def test_wide_links_after_a_handle_with_narrow_ones(P, l):
    """Factor and solve on a handle of l link rows per pair (three levels of cyclic
    reduction), before and after a handle with one link row was created: the same
    direction, bit for bit, and a correct one."""
    wide = random_block_lp(3, N=8, m_sizes=[120] * 8, n_sizes=[300] * 8, nnz_per_col=5, n0=3,
                           w_density=0.2, l=l)
    narrow = random_block_lp(4, N=3, m_sizes=[20] * 3, n_sizes=[30] * 3, nnz_per_col=3, n0=1,
                             w_density=0.2, l=1)
    A, _, _ = olp.assemble(wide)
    rng = np.random.default_rng(5)
    n, m = A.shape[1], A.shape[0]
    x, z = np.exp(rng.uniform(-1, 1, n)), np.exp(rng.uniform(-1, 1, n))
    r = rng.standard_normal(n), rng.standard_normal(m), rng.standard_normal(n)
    first = P.arrowhead_lp_create(wide)
    P.kkt_factor(first, x, z)
    before, _ = P.kkt_solve(first, *r)
    second = P.arrowhead_lp_create(narrow)
    P.kkt_factor(first, x, z)
    after, _ = P.kkt_solve(first, *r)
    for u, v in zip(before, after):
        assert np.array_equal(u, v)
    assert onewton.relative_residual(A, x, z, *after, *r) <= 1e-9   # refine_tol is 1e-10
    P.kkt_factor(second, np.ones(narrow.n_total), np.ones(narrow.n_total))
    first.close()
    second.close()

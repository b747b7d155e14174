"""FP64 diagonal tiles over the whole range of FP64 pivots.

Pairs of rows 2i, 2i + 1 carry the columns e_2i, e_2i+1 and e_2i + e_2i+1 with
D = 2^k, so the block's normal matrix is block diagonal with 2^k [2 1; 1 2], whose
factor is known: L = 2^(k/2) [sqrt 2; 1 / sqrt 2, sqrt 1.5].  D, its sums and the
matrix are exact; the reciprocal square root is good to about one unit u = 2^-53,
the scaling adds half of one, the second pivot's update half of one of 2^k 1.5,
so 4 u bounds every entry.  A pivot that overflows to infinity leaves its row out
of the factor, and the other rows' solution as it is."""
import numpy as np
import pytest
import scipy.sparse as sp

from instances import BlockLP

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2412_07731_gb300 as P
    return P


def _lp(A):
    A = sp.csc_matrix(A)
    m, n = A.shape
    none = sp.csc_matrix((0, 0))
    return BlockLP(N=1, n0=0, mg=0, A=[A], W=[sp.csc_matrix((m, 0))], b=[np.ones(m)],
                   c=[np.ones(n)], c0=np.zeros(0), l=np.zeros(0, dtype=np.int64), FL=[], FR=[],
                   F0=[], blink=[], Fg=[sp.csc_matrix((0, n))], Fg0=none, bg=np.zeros(0))


def _power(k):
    """x, z with x / z = 2^k exactly, both normal."""
    a = np.ceil(k / 2).astype(int)
    return np.ldexp(1.0, a), np.ldexp(1.0, a - k)


def test_factor_over_all_exponents(P):
    from paper_2412_07731_gb300._lib import kkt_block_factor_dense
    rng = np.random.default_rng(1)
    # every eighth exponent and its successor, both parities, in random order
    k = rng.permutation(np.concatenate([np.arange(-1000, 1021, 8), np.arange(-999, 1021, 8)]))
    p = len(k)
    cols = []
    for i in range(p):
        cols += [{2 * i: 1.0}, {2 * i + 1: 1.0}, {2 * i: 1.0, 2 * i + 1: 1.0}]
    A = sp.lil_matrix((2 * p, 3 * p))
    for j, c in enumerate(cols):
        for r, v in c.items():
            A[r, j] = v
    x, z = _power(np.repeat(k, 3))
    prob = P.arrowhead_lp_create(_lp(A))
    P.kkt_factor(prob, x, z, 0.0, 0.0)
    F = kkt_block_factor_dense(prob, 0)
    prob.close()
    s = np.sqrt(np.ldexp(1.0, k & 1)) * np.ldexp(1.0, (k - (k & 1)) // 2)   # 2^(k/2)
    i = np.arange(p)
    for got, want in ((F[2 * i, 2 * i], s * np.sqrt(2.0)), (F[2 * i + 1, 2 * i], s * np.sqrt(0.5)),
                      (F[2 * i + 1, 2 * i + 1], s * np.sqrt(1.5))):
        assert (np.abs(got - want) <= 4 * U * want).all(), k[np.abs(got - want) > 4 * U * want]


@pytest.mark.parametrize("row", [0, 5, 70, 149])
def test_infinite_pivot_leaves_its_row_out(P, row):
    """Row `row` holds one column with D = 1e308 and coefficient 10: D is finite, the
    pivot is not.  With a zero right-hand side there, the direction of the other
    rows is that of the LP without it."""
    rng = np.random.default_rng(2)
    m, n = 150, 240
    A = sp.random(m, n, density=0.05, random_state=rng, format="lil")
    for r in range(m):
        A[r, r] = 2.0
    keep = np.arange(m) != row
    B = sp.lil_matrix((m, n + 1))
    B[:, :n] = A
    B[row, :] = 0.0
    B[row, n] = 10.0
    x, z = np.exp(rng.uniform(-1, 1, n)), np.exp(rng.uniform(-1, 1, n))
    rd, rp, rc = rng.standard_normal(n), rng.standard_normal(m), rng.standard_normal(n)
    rp[row] = 0.0
    small = P.arrowhead_lp_create(_lp(sp.csc_matrix(A)[keep]))
    P.kkt_factor(small, x, z, 0.0, 0.0)
    want, _ = P.kkt_solve(small, rd, rp[keep], rc)
    prob = P.arrowhead_lp_create(_lp(B))
    P.kkt_factor(prob, np.append(x, 1e154), np.append(z, 1e-154), 0.0, 0.0)
    (dx, dy, dz), info = P.kkt_solve(prob, np.append(rd, 0.0), rp, np.append(rc, 0.0))
    assert info["rel_residual"] <= 1e-10
    assert dx[n] == 0.0 and dy[row] == 0.0
    for got, ref in ((dx[:n], want[0]), (dy[keep], want[1]), (dz[:n], want[2])):
        assert np.linalg.norm(got - ref) <= 1e-8 * np.linalg.norm(ref)   # both at rounding level
    small.close()
    prob.close()

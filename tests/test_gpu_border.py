"""The border solve is as accurate as substitution with the border's factor.

One block with a single row that no global row shares, so the border of the B global
rows is S = F D F' (D = 1) and the y_g part of a direction is the border solve's result.
F holds m columns of norms up to sqrt(cond) and a diagonal: a matrix of low rank on
top of a graded diagonal.  A direction without refinement and regularisation, for a
right-hand side in the global rows alone, must solve S y = b as well as numpy's
substitution with the Cholesky factor of the same matrix: residuals in extended
precision, a factor of four in the geometric mean over eight seeds.  In numpy,
substitution by tiles of 64 rows with inverted diagonal tiles stays within a factor of
two of it on average, and the explicit inverse of the whole factor is 4 to 12 times as
far off at these orders."""
import numpy as np
import pytest
import scipy.linalg as sl
import scipy.sparse as sp

from instances import BlockLP

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2412_07731_gb300 as P
    return P


def case(B, m, cond, decades, seed):
    """F [B, m + B] and b of S y = F F' y = b with a random y."""
    rng = np.random.default_rng(seed)
    M = rng.standard_normal((B, m)) * 10.0 ** rng.uniform(0, np.log10(cond) / 2, m)
    F = np.hstack([M, np.diag(10.0 ** rng.uniform(0, decades, B))])
    return F, -residual_vector(F, np.zeros(B), rng.standard_normal(B))


def residual_vector(F, b, y):
    E = F.astype(np.longdouble)
    return (b - E @ (E.T @ y.astype(np.longdouble))).astype(np.float64)


def substitution(F, b):
    C = np.linalg.cholesky(F @ F.T)
    return sl.solve_triangular(C.T, sl.solve_triangular(C, b, lower=True), lower=False)


# 7, 11 and 20 tiles; the last order's factor has more than 152 trailing tiles, so its updates
# on the FP64 pipe run one CTA per tile.  Pivots stay above 1e-12 of their diagonals (no clamping)
CASES = [(420, 40, 1e10, 0.0), (420, 120, 1e10, 1.0), (700, 40, 1e8, 1.0), (1280, 20, 1e6, 1.0)]


@pytest.mark.parametrize("B,m,cond,decades", CASES)
def test_border_equation_is_solved_like_substitution(P, B, m, cond, decades):
    ratio = []
    for seed in range(8):
        F, b = case(B, m, cond, decades, seed)
        n = 1 + F.shape[1]
        A = sp.csc_matrix(([1.0], ([0], [0])), shape=(1, n))
        Fg = sp.csc_matrix(np.hstack([np.zeros((B, 1)), F]))
        lp = BlockLP(N=1, n0=0, mg=B, A=[A], W=[sp.csc_matrix((1, 0))], b=[np.ones(1)],
                     c=[np.ones(n)], c0=np.zeros(0), l=np.zeros(0, dtype=np.int64), FL=[], FR=[],
                     F0=[], blink=[], Fg=[Fg], Fg0=sp.csc_matrix((B, 0)), bg=np.ones(B))
        prob = P.arrowhead_lp_create(lp, P.default_options(refine_max=0))
        P.kkt_factor(prob, np.ones(n), np.ones(n), 0.0, 0.0)
        (_, dy, _), _ = P.kkt_solve(prob, np.zeros(n), np.append(0.0, b), np.zeros(n))
        prob.close()
        ratio.append(np.linalg.norm(residual_vector(F, b, dy[1:])) /
                     np.linalg.norm(residual_vector(F, b, substitution(F, b))))
    assert np.exp(np.mean(np.log(ratio))) <= 4.0, ratio

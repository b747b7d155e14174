"""FP64 block factors whose trailing updates run on the tensor cores (eight
exact FP16 digits per entry): the backward error of every block's partial
Cholesky stays within the bound of Cholesky in FP64 arithmetic.

With F = [L; Y'] the factor of [M G; G' .] and u = 2^-53, FP64 Cholesky of
order m gives |M - L L'|_ij <= (m + 2) u sqrt(M_ii M_jj) (1 + O(u)) and, row
by row, |G - L Y|_ij <= (m + 2) u sqrt(M_ii) |Y_j|_2.  The digit products add
at most 2^-55 of the row scales' product per 64 columns, below one rounding of
the chain they replace; forming M and G costs a few roundings per entry.  The
bound checked is (m + 16) u of the same scales.  Block orders sit at the edges
of the 64-row tiles and of the 128-row jobs, with partial last pivot tiles
that also hold Schur columns; D spans up to 1e12.
"""
import numpy as np
import pytest

from instances import random_block_lp

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2412_07731_gb300 as P
    return P


def _check(P, lp, seed, decades, blocks=None):
    from paper_2412_07731_gb300._lib import kkt_block_factor_dense
    rng = np.random.default_rng(seed)
    h = decades * np.log(10.0) / 4
    n = lp.n_total
    x, z = np.exp(rng.uniform(-h, h, n)), np.exp(rng.uniform(-h, h, n))
    prob = P.arrowhead_lp_create(lp)
    P.kkt_factor(prob, x, z, 0.0, 0.0)
    xo = lp.x_offsets()
    for i in (range(lp.N) if blocks is None else blocks):
        F = kkt_block_factor_dense(prob, i)
        m = lp.A[i].shape[0]
        # extended precision is slow: the first and last rows and a few between
        rows = np.unique(np.concatenate([[0, m - 1], rng.integers(0, m, 14)]))
        L, Yt = F[:m, :m].astype(np.longdouble), F[m:, :m].astype(np.longdouble)
        A = lp.A[i].toarray().astype(np.longdouble)
        d = (x[xo[i]:xo[i + 1]] / z[xo[i]:xo[i + 1]]).astype(np.longdouble)
        s = np.sqrt(((A * A) * d).sum(1))
        err = np.abs((A[rows] * d) @ A.T - L[rows] @ L.T) / np.outer(s[rows], s)
        err[np.arange(m)[None, :] > rows[:, None]] = 0   # the lower triangle
        assert err.max() <= (m + 16) * U, (i, m, float(err.max() / U))
        # the linking-variable columns come first among the Schur columns
        W = lp.W[i].toarray().astype(np.longdouble)
        Yw = Yt[:lp.n0].T
        err = np.abs(W[rows] - L[rows] @ Yw) / np.maximum(
            np.outer(s[rows], np.sqrt((Yw ** 2).sum(0))), 1e-300)
        assert err.max() <= (m + 16) * U, (i, m, float(err.max() / U))
    prob.close()


@pytest.mark.parametrize("decades", [2.0, 12.0])
def test_backward_error_at_tile_edges(P, decades):
    m = [17, 63, 64, 65, 127, 128, 129, 191, 192, 193, 320, 389]
    lp = random_block_lp(21, N=len(m), m_sizes=m, n_sizes=[3 * v // 2 for v in m], nnz_per_col=6,
                         n0=5, w_density=0.3, l=3, mg=2, global_nnz=4)
    _check(P, lp, 3, decades)


def test_backward_error_with_several_jobs_per_cta(P):
    """60 blocks of about ten tiles: thousands of jobs, so that every CTA reuses its
    operand stages and accumulators across barrier phases."""
    rng = np.random.default_rng(4)
    m = [int(v) for v in rng.integers(560, 660, 60)]
    lp = random_block_lp(22, N=60, m_sizes=m, n_sizes=[3 * v // 2 for v in m], nnz_per_col=6,
                         n0=40, w_density=0.1, l=3)
    _check(P, lp, 5, 6.0, blocks=(0, 17, 31, 46, 58, 59))


def test_backward_error_with_mixed_last_tiles(P):
    """500 small blocks: a CTA's jobs of one step mix blocks whose pivot tile is full with
    blocks whose last one has one, two or three slices of 16 columns, so the operand
    buffers are reused with different numbers of slices."""
    rng = np.random.default_rng(6)
    m = [int(v) for v in rng.integers(66, 200, 500)]
    lp = random_block_lp(24, N=500, m_sizes=m, n_sizes=[3 * v // 2 for v in m], nnz_per_col=6,
                         n0=70, w_density=0.1, l=1)
    _check(P, lp, 7, 4.0, blocks=[int(b) for b in rng.integers(0, 500, 40)])


def test_nan_pivot_is_reported(P):
    """A block whose diagonal overflows to infinity: rows with a NaN or an infinity pass
    through the digit staging, and the factor is refused as before."""
    lp = random_block_lp(23, N=2, m_sizes=[200, 150], n_sizes=[300, 230], nnz_per_col=6, n0=2,
                         w_density=0.3, l=2)
    x, z = np.ones(lp.n_total), np.ones(lp.n_total)
    x[:300] = 1e200
    z[:300] = 1e-200
    prob = P.arrowhead_lp_create(lp)
    with pytest.raises(P.AHLPError) as e:
        P.kkt_factor(prob, x, z, 0.0, 0.0)
    assert e.value.status == -4
    prob.close()

"""The jobs of the FP64 digit update: job order, early-stopping CTAs, tile-sparse tables
and blocks whose next diagonal tile no job touches.

  * With events between the launches (profile_kernels) the next step's diagonal tiles
    wait for the whole update instead of running beside it; the factor must be the same,
    bit for bit.  A left-out or repeated job shows in the backward error of [M; G']: (m +
    16) u for the factor, as in FP64 arithmetic, and m u for the products that check it in
    FP64.
  * Tile jobs that are left out would add exact zeros, so factors, Schur complement and
    directions with and without tile_sparse are the same, bit for bit."""
import numpy as np
import pytest
import scipy.sparse as sp

from instances import config3, random_block_lp

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2412_07731_gb300 as P
    return P


SETS = {
    "spare SMs": [640, 577, 130],
    "one round": [700] * 6 + [65, 66],
    "several rounds": [1300, 1100, 1280, 640] * 4 + [100] * 3,
    "many tiles": [129, 190, 64] * 70,
}


@pytest.mark.parametrize("sizes", SETS.values(), ids=SETS.keys())
def test_overlapped_factor_is_the_serial_one(P, sizes):
    from paper_2412_07731_gb300._lib import kkt_block_factor_dense
    lp = random_block_lp(5, N=len(sizes), m_sizes=sizes, n_sizes=[3 * v // 2 for v in sizes],
                         nnz_per_col=4, n0=5, w_density=0.3, l=2, mg=2, global_nnz=3)
    rng = np.random.default_rng(9)
    x, z = np.exp(rng.uniform(-1, 1, lp.n_total)), np.exp(rng.uniform(-1, 1, lp.n_total))
    probs = [P.arrowhead_lp_create(lp, P.default_options(profile_kernels=k)) for k in (0, 1)]
    for prob in probs:
        P.kkt_factor(prob, x, z, 0.0, 0.0)
    xo = lp.x_offsets()
    for i in range(lp.N):
        F = kkt_block_factor_dense(probs[0], i)
        assert np.array_equal(F, kkt_block_factor_dense(probs[1], i)), i
        m = lp.A[i].shape[0]
        A = lp.A[i].toarray()
        d = x[xo[i]:xo[i + 1]] / z[xo[i]:xo[i + 1]]
        s = np.sqrt(((A * A) * d).sum(1))
        L = np.tril(F[:m, :m])
        assert (np.abs((A * d) @ A.T - L @ L.T) <= (3 * m + 32) * U * np.outer(s, s)).all(), i
        Y = F[m:m + lp.n0, :m]
        e = np.abs(lp.W[i].toarray() - L @ Y.T)
        assert (e <= (3 * m + 32) * U * np.outer(s, np.sqrt((Y ** 2).sum(1)))).all(), i
    for prob in probs:
        prob.close()


def _block_diagonal():
    """Blocks of row groups that no column couples, as many as whole tiles: the tile left of the
    second diagonal tile is zero, so the first step has no job there.  One dense block beside."""
    lp = random_block_lp(8, N=4, m_sizes=[218, 192, 150, 218], n_sizes=[340, 300, 230, 340],
                         nnz_per_col=5, n0=4, w_density=0.3, l=3, mg=2, global_nnz=3, plant=None)
    rng = np.random.default_rng(2)
    for i, groups in ((0, ((64, 100), (64, 100), (90, 140))), (1, ((128, 200), (64, 100))),
                      (3, ((64, 100), (154, 240)))):
        part = []
        for m, n in groups:
            a = sp.random(m, n, density=0.08, random_state=rng, format="lil")
            a.setdiag(2.0)
            part.append(a)
        lp.A[i] = sp.csc_matrix(sp.block_diag(part))
    lp.b = [np.zeros(a.shape[0]) for a in lp.A]
    lp.c = [np.zeros(a.shape[1]) for a in lp.A]
    lp.blink = [np.zeros(int(v)) for v in lp.l]
    return lp


@pytest.mark.parametrize("make", [lambda: config3(days=3), _block_diagonal],
                         ids=["banded", "block diagonal"])
def test_tile_sparse_factor_is_the_dense_one(P, make):
    from paper_2412_07731_gb300._lib import kkt_block_factor_dense
    lp = make()
    rng = np.random.default_rng(3)
    n, m = lp.n_total, lp.m_total
    x, z = np.exp(rng.standard_normal(n)), np.exp(rng.standard_normal(n))
    r = rng.standard_normal(n), rng.standard_normal(m), rng.standard_normal(n)
    probs = [P.arrowhead_lp_create(lp, P.default_options(tile_sparse=s)) for s in (0, 1)]
    dirs = []
    for prob in probs:
        P.kkt_factor(prob, x, z)
        P.kkt_factor(prob, x, z)   # the counts start anew
        dirs.append(P.kkt_solve(prob, *r)[0])
    for i in range(lp.N):
        F = [kkt_block_factor_dense(prob, i) for prob in probs]
        assert np.isfinite(F[0]).all() and np.array_equal(*F), i
    assert np.array_equal(P.kkt_schur_dense(probs[0]), P.kkt_schur_dense(probs[1]))
    for u, v in zip(*dirs):
        assert np.array_equal(u, v)
    (k0, d0), (k1, d1) = (P.kkt_update_jobs(prob) for prob in probs)
    assert k0 == d0 == d1 > 0 and 0 < k1 < d1
    for prob in probs:
        prob.close()

"""kkt_solve and kkt_adjoint_solve on an FP64 factor whose digit updates precondition too
badly: the factor is redone in FP64 arithmetic and the solve repeated.

The points are iterates of the CPU oracle on an LP whose optimum is a face (half of
the variables zero on both sides), close to it: block pivots are clamped there.  At
the last but one iterate 40 Krylov steps leave residuals of 3e-3 to 4e-3 with the
digits' factor and about 1e-4 with FP64 arithmetic's; the line between is drawn at their
geometric mean, 6e-4."""
import numpy as np
import pytest

from instances import random_block_lp
from oracle import ipm as oipm
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


@pytest.fixture(scope="module")
def face():
    m = [90, 140, 70, 110]
    lp = random_block_lp(6, N=4, m_sizes=m, n_sizes=[3 * v // 2 for v in m], nnz_per_col=8,
                         n0=200, w_density=0.05, l=5, mg=10, plant="half_zero")
    A, b, c = olp.assemble(lp)
    rec = []
    oipm.solve(A, b, c, record=rec, max_iter=30)
    return lp, A, rec


def _rhs(A, x, z, mu):
    rng = np.random.default_rng(1)
    s = np.sqrt(mu)
    return s * rng.standard_normal(A.shape[1]), s * rng.standard_normal(A.shape[0]), -x * z


def _factors(prob, lp):
    from paper_2412_07731_gb300._lib import kkt_block_factor_dense
    return [kkt_block_factor_dense(prob, i) for i in range(lp.N)]


@pytest.mark.parametrize("adjoint", [False, True])
def test_failed_solve_moves_to_fp64_arithmetic(P, face, adjoint):
    lp, A, rec = face
    it = rec[-2]
    x, z = it["x"], it["z"]
    r = _rhs(A, x, z, it["mu"])
    prob = P.arrowhead_lp_create(lp)
    solve = P.kkt_adjoint_solve if adjoint else P.kkt_solve
    P.kkt_factor(prob, x, z)
    digits = _factors(prob, lp)
    d, info = solve(prob, *r)
    assert info["rel_residual"] <= 6e-4
    if not adjoint:   # the residual reported is that of the direction returned
        res = onewton.relative_residual(A, x, z, *d, *r)
        assert abs(res - info["rel_residual"]) <= 1e-3 * res
    pipe = _factors(prob, lp)
    assert any(not np.array_equal(a, b) for a, b in zip(digits, pipe))
    # the factor stays, and so does what it gives
    e, again = solve(prob, *r)
    assert again["rel_residual"] == info["rel_residual"]
    assert all(np.array_equal(a, b) for a, b in zip(d, e))
    assert all(np.array_equal(a, b) for a, b in zip(pipe, _factors(prob, lp)))
    # a new factor starts on the tensor cores again
    P.kkt_factor(prob, x, z)
    assert all(np.array_equal(a, b) for a, b in zip(digits, _factors(prob, lp)))
    prob.close()


def test_converged_solve_keeps_its_factor(P, face):
    lp, A, rec = face
    it = rec[-3]
    x, z = it["x"], it["z"]
    prob = P.arrowhead_lp_create(lp)
    P.kkt_factor(prob, x, z)
    before = _factors(prob, lp)
    _, info = P.kkt_solve(prob, *_rhs(A, x, z, it["mu"]))
    assert info["rel_residual"] <= 1e-10   # refine_tol
    assert all(np.array_equal(a, b) for a, b in zip(before, _factors(prob, lp)))
    prob.close()


@pytest.mark.parametrize("back", [1, 2])
def test_every_point_gives_a_usable_handle(P, face, back):
    """The last iterates, where FP64 arithmetic itself may break down: a factor that was
    accepted still gives finite directions, with the residual that is reported."""
    lp, A, rec = face
    it = rec[-back]
    x, z = it["x"], it["z"]
    r = _rhs(A, x, z, it["mu"])
    prob = P.arrowhead_lp_create(lp)
    P.kkt_factor(prob, x, z)
    for _ in range(2):
        d, info = P.kkt_solve(prob, *r)
        res = onewton.relative_residual(A, x, z, *d, *r)
        assert np.isfinite(res) and abs(res - info["rel_residual"]) <= 1e-3 * res
    prob.close()


def test_nan_right_hand_side_does_not_refactor(P, face):
    lp, A, rec = face
    it = rec[-3]
    prob = P.arrowhead_lp_create(lp)
    P.kkt_factor(prob, it["x"], it["z"])
    before = _factors(prob, lp)
    rd, rp, rc = _rhs(A, it["x"], it["z"], it["mu"])
    rd[0] = np.nan
    with pytest.raises(P.AHLPError) as e:
        P.kkt_solve(prob, rd, rp, rc)
    assert e.value.status == -4
    assert all(np.array_equal(a, b) for a, b in zip(before, _factors(prob, lp)))
    prob.close()

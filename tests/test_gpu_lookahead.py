"""Diagonal tiles factored beside the trailing update of the step before.

The persistent updates count off the tiles that the next step's diagonal
factorisation waits for, and leave it some SMs; neither changes an operation.
So a block's factor must equal, bit for bit, the one-CTA-per-job kernel's
(FP32, float-float: its diagonal tiles wait for the whole update), and repeat
bit for bit (FP64).  The block sets lie at the edges of the rule: fewer jobs
than SMs, jobs for less than a round of the SMs left, several rounds with some
CTAs stopping early, more diagonal tiles than SMs, and blocks that end at
different steps."""
import numpy as np
import pytest

from instances import random_block_lp

pytestmark = pytest.mark.gpu


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
@pytest.mark.parametrize("prec", ["fp32", "ff", "fp64"])
def test_factor_is_the_one_without_overlap(P, sizes, prec):
    from paper_2412_07731_gb300._lib import kkt_block_factor_dense
    lp = random_block_lp(5, N=len(sizes), m_sizes=sizes, n_sizes=[3 * v // 2 for v in sizes],
                         nnz_per_col=4, n0=5, w_density=0.3, l=2, mg=2, global_nnz=3)
    rng = np.random.default_rng(9)
    x, z = np.exp(rng.uniform(-1, 1, lp.n_total)), np.exp(rng.uniform(-1, 1, lp.n_total))
    if prec == "fp64":
        kws = [dict()] * 2
    else:
        key, cond = ("fp32_update", 1e300) if prec == "fp32" else ("ff_update", 1.0)
        kws = [{"precision": P.PREC_MIXED, "fp32_cond_max": cond, key: u} for u in (2, 3)]
    out = []
    for kw in kws:
        prob = P.arrowhead_lp_create(lp, P.default_options(**kw))
        P.kkt_factor(prob, x, z)
        P.kkt_factor(prob, x, z)   # the counts start anew
        out.append([kkt_block_factor_dense(prob, i) for i in range(lp.N)])
        prob.close()
    for i in range(lp.N):
        assert np.isfinite(out[0][i]).all()
        assert np.array_equal(out[0][i], out[1][i]), i

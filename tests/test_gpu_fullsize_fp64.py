"""A complete FP64 solve of the 512-block workload with the trailing updates on the
tensor cores.  Its last iteration clamps pivots and overflows inside blocks
(NaN pivots); there the digit factors, which keep an entry relative to its row's
largest, precondition worse than FP64 arithmetic (a step taken on such a direction
sent the iterates off: 34 iterations in place of 17), so the solve moves to the FP64
pipe.  With FP64 arithmetic throughout it takes 17 iterations; two more are
allowed for."""
import pytest

from instances import config2
from oracle import lp as olp

pytestmark = pytest.mark.gpu


def test_fp64_solve_keeps_its_iterations():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2412_07731_gb300 as P
    lp = config2()
    A, b, c = olp.assemble(lp)
    prob = P.arrowhead_lp_create(lp, P.default_options(precision=P.PREC_FP64, max_correctors=0))
    (x, y, z), r = P.ipm_solve(prob)
    assert r["status"] == 0 and r["iterations"] <= 19, r
    meas = olp.measures(A, b, c, x, y, z)
    assert meas["pinf"] <= 1e-8 and meas["dinf"] <= 1e-8 and meas["gap"] <= 1e-8, meas
    prob.close()

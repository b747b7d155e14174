"""The gradient's last resort (host logic, no GPU): FP64 factors with more and more
regularisation until the transposed solve converges, whether a factor breaks down or
is accepted and then stalls.  The library's calls are replaced by recorded answers."""
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")

import paper_2412_07731_gb300 as P
from paper_2412_07731_gb300 import autograd as ag


class Calls:
    """kkt_factor and kkt_adjoint_solve answering from lists: 'nan' or a residual."""

    def __init__(self, monkeypatch, answers):
        self.answers, self.factors, self.precisions = list(answers), [], []
        self.prob = SimpleNamespace(options=P.default_options(precision=P.PREC_MIXED), n=3, m=2,
                                    factor_gen=0)
        monkeypatch.setattr(ag.L, "set_options", self.set_options)
        monkeypatch.setattr(ag.L, "kkt_factor", self.kkt_factor)
        monkeypatch.setattr(ag.L, "kkt_adjoint_solve", self.kkt_adjoint_solve)

    def set_options(self, prob, options):
        prob.options = ag.L.Options.from_buffer_copy(options)

    def kkt_factor(self, prob, x, z, delta=-1.0, rho=-1.0):
        prob.factor_gen += 1
        self.factors.append((delta, rho))
        self.precisions.append(prob.options.precision)
        if self.answers[0] == "nan":
            self.answers.pop(0)
            raise P.AHLPError(-4, "NaN pivot")

    def kkt_adjoint_solve(self, prob, gx, gy, gz):
        return (gx + 1, gy + 1, gz), {"rel_residual": self.answers.pop(0), "refine_steps": 40}

    def backward(self):
        v, w = torch.ones(3, dtype=torch.float64), torch.ones(2, dtype=torch.float64)
        ctx = SimpleNamespace(prob=self.prob, factor_gen=self.prob.factor_gen,
                              saved_tensors=(v, v))
        return ag.LPSolve.backward(ctx, v, w, None)


@pytest.mark.parametrize("answers,tried", [
    ([1e-9], []),                                    # the factor at hand does
    ([1e-3, 1e-9], [(-1.0, -1.0)]),                  # an FP64 one does
    ([1e-3, "nan", 1e-9], [(-1.0, -1.0), (1e-6, 1e-8)]),
    ([1e-3, 0.5, 1e-7], [(-1.0, -1.0), (1e-6, 1e-8)]),
    ([1e-3, "nan", float("nan"), 1e-9], [(-1.0, -1.0), (1e-6, 1e-8), (1e-4, 1e-6)])])
def test_regularisation_until_the_solve_converges(monkeypatch, answers, tried):
    c = Calls(monkeypatch, answers)
    lx, ly, none = c.backward()
    assert none is None and float(lx[0]) == 2.0 and float(ly[0]) == 2.0
    assert c.factors == tried and all(p == P.PREC_FP64 for p in c.precisions)
    assert c.prob.options.precision == P.PREC_MIXED and not c.answers


def test_nothing_converges(monkeypatch):
    c = Calls(monkeypatch, [1e-3, 0.5, "nan", 0.4])
    with pytest.raises(RuntimeError, match="did not converge"):
        c.backward()
    assert len(c.factors) == 3 and c.prob.options.precision == P.PREC_MIXED


def test_other_errors_pass_through(monkeypatch):
    c = Calls(monkeypatch, [1e-3, 1e-9])
    monkeypatch.setattr(ag.L, "kkt_factor",
                        lambda *a: (_ for _ in ()).throw(P.AHLPError(-9, "no memory")))
    with pytest.raises(P.AHLPError) as e:
        c.backward()
    assert e.value.status == -9 and c.prob.options.precision == P.PREC_MIXED

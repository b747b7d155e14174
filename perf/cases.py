"""Performance cases: what a user of this library has it do, through its public entry points.

Two kinds of program use the library.  One hands it an LP and takes the optimum
(``ipm_solve``, or ``lp_solve`` with its gradient).  The other keeps its own
outer method and asks for Newton directions at an interior point
(``kkt_factor``, ``kkt_solve`` for a predictor and a corrector right-hand side,
``kkt_adjoint_solve`` for the transposed system).

A case is one LP shape with one such pass:

    what     "direction": kkt_factor and two kkt_solve;  "adjoint": kkt_factor, kkt_solve and
             kkt_adjoint_solve;  "solve": ipm_solve;  "gradient": lp_solve and its backward pass
    shape    "blocks": N random sparse blocks of m_lo .. m_hi rows and 1.5 times as many columns;
             "energy": daily blocks of an hourly network with storage (banded blocks);
             "full": small blocks with bounds of every kind and inequality rows
    prec     "fp64": FP64 block factors;  "mixed": FP32 ones, or float-float ones where the
             scaling D = X Z^-1 spans more than the library's FP32 limit
    decades  the span of D at the point of a direction, in powers of ten: a few in the first
             iterations, 15 and more near the optimum
    batch    LPs in one handle (their direct sum)
"""
from __future__ import annotations

import numpy as np
import torch

import instances
import paper_2412_07731_gb300 as P
from paper_2412_07731_gb300.autograd import lp_solve

DEV = torch.device("cuda", 0)


def _case(name, what, shape, prec, N, m_lo, m_hi, n0, links, mg=0, batch=1, decades=4.0):
    case = dict(what=what, shape=shape, prec=prec, N=N, m_lo=m_lo, m_hi=m_hi, n0=n0, links=links,
                mg=mg, batch=batch, decades=decades)
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest LP of the test-suite: a user's unit test, or a small LP in a service that
        # answers many; one direction takes about a dozen launches of tiny kernels
        _case("tiny direction", "direction", "blocks", "fp64", 4, 40, 40, 3, 2),
        # a small LP solved from start to end
        _case("tiny solve", "solve", "blocks", "fp64", 4, 40, 40, 3, 2),
        # a model as written, with free, boxed and fixed variables and inequality rows
        _case("full statement", "direction", "full", "mixed", 24, 120, 120, 8, 4, mg=2),
        # the default precision on uneven blocks: what a caller gets who sets no option
        _case("uneven fp64", "direction", "blocks", "fp64", 32, 500, 4000, 100, 16),
        # the first iterations of a mixed-precision solve (FP32 block factors): 64 equal blocks
        _case("uniform mixed early", "direction", "blocks", "mixed", 64, 2000, 2000, 50, 20),
        # the same on uneven blocks, the largest case
        _case("uneven mixed early", "direction", "blocks", "mixed", 96, 500, 4000, 100, 16),
        # the last iterations of a mixed-precision solve (float-float block factors)
        _case("uneven mixed late", "direction", "blocks", "mixed", 64, 500, 4000, 100, 16,
              decades=15.0),
        # an energy model of one month: banded daily blocks, many linking variables
        _case("energy mixed", "direction", "energy", "mixed", 30, 0, 0, 600, 30, mg=1),
        # four independent LPs in one handle
        _case("batch mixed", "direction", "blocks", "mixed", 8, 500, 4000, 100, 16, batch=4),
        # sensitivities of a mid-sized LP: a direction and a transposed solve, ragged sizes
        _case("ragged adjoint", "adjoint", "blocks", "fp64", 13, 130, 517, 6, 7, mg=2),
        # a whole mixed-precision solve of mid-sized blocks
        _case("mid solve", "solve", "blocks", "mixed", 16, 300, 700, 20, 8),
        # an optimum inside a differentiable program: solve, then the gradient of a loss
        _case("gradient", "gradient", "blocks", "fp64", 6, 60, 200, 4, 3),
    ]


def draw(rng):
    def log(lo, hi):
        return lo * (hi / lo) ** rng.random()

    what = rng.choice(["direction", "direction", "direction", "adjoint", "solve", "gradient"])
    if what == "gradient":
        m = int(log(30, 250))
        return _case("", what, "blocks", "fp64", rng.randint(2, 8), max(20, m // 2), m,
                     rng.randint(1, 8), rng.randint(1, 5))
    if what == "solve":
        m = int(log(30, 900))
        return _case("", what, "blocks", rng.choice(["fp64", "mixed"]), rng.randint(2, 20),
                     max(24, m // 2), m, rng.randint(1, 30), rng.randint(1, 12))
    prec = rng.choice(["fp64", "mixed", "mixed"])
    decades = rng.choice([2.0, 4.0, 6.0] if prec == "fp64" else [3.0, 5.0, 15.0])
    shape = rng.choice(["blocks", "blocks", "blocks", "energy", "full"])
    if shape == "energy":
        return _case("", what, shape, prec, rng.randint(3, 20), 0, 0, rng.randint(100, 600), 30,
                     mg=1, decades=min(decades, 6.0))
    if shape == "full":
        return _case("", what, shape, prec, rng.randint(4, 30), *[rng.randint(20, 150)] * 2,
                     rng.randint(1, 12), rng.randint(1, 8), mg=rng.randint(0, 3),
                     decades=min(decades, 6.0))
    m = int(log(60, 4000))
    N = max(2, min(int(log(2, 64)), int(60e9 / (m / 1.5) ** 3) + 2 if prec == "fp64" else 64))
    return _case("", what, shape, prec, N, max(24, m // rng.randint(1, 8)), m,
                 rng.randint(1, 100), rng.randint(1, 20), mg=rng.randint(0, 3),
                 batch=rng.choice([1, 1, 1, 2, 3]) if N <= 16 else 1, decades=decades)


def _rows(case, k):
    """Rows of the k-th LP's blocks: a property of the case, not of the seed."""
    r = np.random.default_rng([case["N"], case["m_lo"], case["m_hi"], k])
    return r.integers(case["m_lo"], case["m_hi"] + 1, size=case["N"])


def _lps(case, seed):
    out = []
    for k in range(case["batch"]):
        s = 1000 * seed + k
        if case["shape"] == "energy":
            out.append(instances.config3(s, days=case["N"], nodes=case["links"],
                                         n_invest=case["n0"]))
        elif case["shape"] == "full":
            # its kinds of bounds decide the sizes of the equality form: one model, other points
            out.append(instances.general_block_lp(
                case["N"], N=case["N"], m=case["m_lo"], n=3 * case["m_lo"] // 2, n0=case["n0"],
                l=case["links"], mg=case["mg"], mD=case["m_lo"] // 4))
        else:
            m = _rows(case, k)
            out.append(instances.random_block_lp(
                s, N=case["N"], m_sizes=m, n_sizes=(3 * m) // 2, nnz_per_col=8, n0=case["n0"],
                w_density=0.05, l=case["links"], mg=case["mg"],
                plant="basis_blocks" if case["what"] in ("solve", "gradient") else "half_zero"))
    return out


def _options(case):
    # directions for a caller's own outer method are asked for well below its tolerances; whole
    # solves stop at a tight gap, so that a vertex is told apart from its neighbours
    tight = dict(tol=1e-10, ipm_refine_tol=1e-10) if case["what"] in ("solve", "gradient") else {}
    return P.default_options(
        precision=P.PREC_FP64 if case["prec"] == "fp64" else P.PREC_MIXED, refine_tol=1e-13,
        **tight)


def _point(case, n, m, seed):
    """An interior point and two right-hand sides: D = x / z log-uniform over the case's decades
    around an iterate of complementarity mu, residuals of an infeasible iterate."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    f = dict(dtype=torch.float64, device=DEV, generator=g)
    h = case["decades"] * np.log(10.0) / 4
    t = (2 * torch.rand(n, **f) - 1) * h
    mu = 10.0 ** (-case["decades"] / 2)
    w = torch.exp(0.2 * torch.randn(n, **f)) * np.sqrt(mu)
    x, z = w * torch.exp(t), w * torch.exp(-t)
    s = np.sqrt(mu)
    r = [s * torch.randn(n, **f), s * torch.randn(m, **f), -x * z]
    r2 = [torch.zeros_like(r[0]), torch.zeros_like(r[1]),
          mu * (0.1 - 0.05 * torch.randn(n, **f))]
    return x, z, r, r2


def prepare(case, seed):
    lps = _lps(case, seed)
    prob = P.arrowhead_lp_create(lps if len(lps) > 1 else lps[0], _options(case))
    st = {"what": case["what"], "prob": prob}
    f = dict(dtype=torch.float64, device=DEV)
    if case["what"] in ("direction", "adjoint"):
        st["x"], st["z"], st["r"], st["r2"] = _point(case, prob.n, prob.m, seed)
    elif case["what"] == "solve":
        st["out"] = tuple(torch.empty(k, **f) for k in (prob.n, prob.m, prob.n))
    else:
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        st["c"] = torch.tensor(lps[0].c_global(), device=DEV)
        st["b"] = torch.tensor(lps[0].b_global(), device=DEV)
        st["w"] = torch.randn(prob.m, generator=g, **f)
    return st


def run(state):
    prob, what = state["prob"], state["what"]
    if what == "solve":
        out, _ = P.ipm_solve(prob, out=state["out"])
        return out
    if what == "gradient":
        # the loss c'x + w'y: its gradient in c and b goes through the transposed Newton system
        c = state["c"].clone().requires_grad_(True)
        b = state["b"].clone().requires_grad_(True)
        x, y, z = lp_solve(c, b, prob)
        (torch.dot(c, x) + torch.dot(state["w"], y)).backward()
        return x.detach(), y.detach(), z.detach(), c.grad, b.grad
    P.kkt_factor(prob, state["x"], state["z"])
    d, _ = P.kkt_solve(prob, *state["r"])
    e, _ = (P.kkt_adjoint_solve if what == "adjoint" else P.kkt_solve)(prob, *state["r2"])
    return d, e


# ---------------------------------------------------------------------------
# work and exact values
# ---------------------------------------------------------------------------
# iterations an interior-point method takes on these LPs, for the work of a whole solve
_ITERATIONS = 10


def _sizes(case):
    """Per block: rows m, columns n, Schur columns k (links on both sides, x_0, global rows)."""
    out = []
    for q in range(case["batch"]):
        if case["shape"] == "energy":
            mn = [(2400 - (30 if d else 0), 24 * 205 + (d == case["N"] - 1))
                  for d in range(case["N"])]
        elif case["shape"] == "full":
            # the equality form: about a quarter more rows for the inequality rows, one more per
            # boxed variable (a fifth of them), a slack per new row, free variables split in two
            m, n = case["m_lo"], 3 * case["m_lo"] // 2
            mn = [(m + m // 4 + n // 5, n + m // 4 + 2 * n // 5)] * case["N"]
        else:
            mn = [(int(m), 3 * int(m) // 2) for m in _rows(case, q)]
        for i, (m, n) in enumerate(mn):
            links = case["links"] * ((i > 0) + (i < case["N"] - 1))
            out.append((m, n, links + case["n0"] + case["mg"]))
    return out


def work(case):
    """Flops: the partial Cholesky of each block with its Schur columns, two triangular sweeps per
    right-hand side.  Bytes: the LP's nonzeros (value and index) and the vectors, once."""
    sizes = _sizes(case)
    n, m = sum(s[1] for s in sizes) + case["n0"], sum(s[0] for s in sizes)
    factor = sum(p ** 3 / 3 + p * p * k + p * k * k for p, _, k in sizes)
    solve = sum(2 * (p + k) ** 2 for p, _, k in sizes)
    nnz = 8 * n + 0.05 * m * case["n0"] if case["shape"] == "blocks" else 3 * n
    times = {"direction": (1, 2), "adjoint": (1, 2), "solve": (_ITERATIONS, 2 * _ITERATIONS),
             "gradient": (_ITERATIONS + 1, 2 * _ITERATIONS + 1)}[case["what"]]
    vectors = 8 * (2 * n + 2 * (2 * n + m) * 2) if case["what"] in ("direction", "adjoint") \
        else 8 * (3 * n + 2 * m + 2 * (n + m))
    return {"bytes": 12 * nnz + vectors, "flops": times[0] * factor + times[1] * solve}


def _dense(M):
    return torch.tensor(M.toarray(), dtype=torch.float64, device=DEV)


def _global_matrix(lps):
    """A of the direct sum in the library's orderings (x: blocks then x_0; y: blocks, links,
    global rows; each LP after LP), as a sparse FP64 tensor on the device."""
    nb = [sum(a.shape[1] for a in q.A) for q in lps]
    mb = [sum(a.shape[0] for a in q.A) for q in lps]
    ml = [int(np.sum(q.l)) for q in lps]
    R, C, V = [], [], []

    def put(M, r, c):
        M = M.tocoo()
        R.append(M.row.astype(np.int64) + r)
        C.append(M.col.astype(np.int64) + c)
        V.append(M.data)

    c, r = 0, 0
    c0, lk, gl = sum(nb), sum(mb), sum(mb) + sum(ml)
    for q in lps:
        co, ro = [], []
        for i in range(q.N):
            co.append(c)
            ro.append(r)
            put(q.A[i], r, c)
            put(q.W[i], r, c0)
            put(q.Fg[i], gl, c)
            r += q.A[i].shape[0]
            c += q.A[i].shape[1]
        for j in range(q.N - 1):
            put(q.FL[j], lk, co[j])
            put(q.FR[j], lk, co[j + 1])
            put(q.F0[j], lk, c0)
            lk += int(q.l[j])
        put(q.Fg0, gl, c0)
        c0 += q.n0
        gl += q.mg
    m = sum(mb) + sum(ml) + sum(q.mg for q in lps)
    n = sum(nb) + sum(q.n0 for q in lps)
    ix = torch.tensor(np.stack([np.concatenate(R), np.concatenate(C)]), device=DEV)
    A = torch.sparse_coo_tensor(ix, torch.tensor(np.concatenate(V), device=DEV), (m, n))
    return A.coalesce(), sum(nb), sum(mb)


class _Newton:
    """[0 A' I; A 0 0; Z 0 X] d = r by dense block elimination in FP64 and iterative refinement.

    The block variables go first (A_i D_i A_i' by Cholesky), then the dense system in the rows
    that couple blocks and x_0."""

    def __init__(self, lps, x, z):
        self.A, self.nb, self.mb = _global_matrix(lps)
        self.At = self.A.t().coalesce()
        self.x, self.z, self.d = x, z, x / z
        A = self.A.to_sparse_csr()
        m, n = self.A.shape
        ix, v = self.A.indices(), self.A.values()
        # rows and columns outside the blocks: couplings (dense in the coupling rows)
        low = ix[0] >= self.mb
        nc, n0 = m - self.mb, n - self.nb
        self.nc, self.n0 = nc, n0
        F = torch.sparse_coo_tensor(torch.stack([ix[0][low] - self.mb, ix[1][low]]), v[low],
                                    (nc, n)).coalesce()
        fi, fv = F.indices(), F.values()
        S = torch.zeros(nc + n0, nc + n0, dtype=torch.float64, device=DEV)
        self.blocks = []
        r = c = 0
        for q in lps:
            for i in range(q.N):
                mi, ni = q.A[i].shape
                Ai = _dense(q.A[i])
                di = self.d[c:c + ni]
                L = torch.linalg.cholesky((Ai * di) @ Ai.t())
                on = (fi[1] >= c) & (fi[1] < c + ni)
                rows = torch.unique(fi[0][on])
                pos = torch.full((max(nc, 1),), -1, dtype=torch.int64, device=DEV)
                pos[rows] = torch.arange(len(rows), device=DEV)
                Fi = torch.zeros(len(rows), ni, dtype=torch.float64, device=DEV)
                Fi[pos[fi[0][on]], fi[1][on] - c] = fv[on]
                Wi = torch.zeros(mi, n0, dtype=torch.float64, device=DEV)
                w = (ix[0] >= r) & (ix[0] < r + mi) & (ix[1] >= self.nb)
                Wi[ix[0][w] - r, ix[1][w] - self.nb] = v[w]
                # columns of [y couplings, x_0] in the block's rows
                G = torch.cat([(Ai * di) @ Fi.t(), Wi], 1)
                at = torch.cat([rows, nc + torch.arange(n0, device=DEV)])
                Y = torch.linalg.solve_triangular(L, G, upper=False)
                k = len(rows)
                Cb = torch.zeros(k + n0, k + n0, dtype=torch.float64, device=DEV)
                Cb[:k, :k] = (Fi * di) @ Fi.t()
                S[at[:, None], at[None, :]] += Cb - Y.t() @ Y
                self.blocks.append((r, mi, L, G, at))
                r, c = r + mi, c + ni
        F0 = torch.zeros(nc, n0, dtype=torch.float64, device=DEV)
        on = fi[1] >= self.nb
        F0[fi[0][on], fi[1][on] - self.nb] = fv[on]
        S[:nc, nc:] += F0
        S[nc:, :nc] += F0.t()
        S[nc:, nc:] -= torch.diag(1.0 / self.d[self.nb:])
        self.S = torch.linalg.lu_factor(S) if nc + n0 else None
        self.csr, self.csrt = A, self.At.to_sparse_csr()

    def _solve(self, rd, rp, rc):
        f = rd - rc / self.x                  # -D^-1 dx + A'dy = f
        fb = f.clone()
        fb[self.nb:] = 0
        g = rp + self.csr @ (self.d * fb)     # with dx_b = D (A'dy - f) put in
        u = torch.cat([g[self.mb:], f[self.nb:]])
        t = g[:self.mb].clone()
        for r, mi, L, G, at in self.blocks:
            u[at] -= G.t() @ torch.cholesky_solve(t[r:r + mi, None], L)[:, 0]
        s = torch.linalg.lu_solve(*self.S, u[:, None])[:, 0] if self.S is not None else u
        dy = torch.cat([t, s[:self.nc]])
        for r, mi, L, G, at in self.blocks:
            dy[r:r + mi] = torch.cholesky_solve((t[r:r + mi] - G @ s[at])[:, None], L)[:, 0]
        dx = self.d * (self.csrt @ dy - f)
        dx[self.nb:] = s[self.nc:]
        return dx, dy, (rc - self.z * dx) / self.x

    def solve(self, rd, rp, rc):
        d = [torch.zeros_like(v) for v in (rd, rp, rc)]
        best, out = float("inf"), None
        for _ in range(12):
            e = (rd - self.csrt @ d[1] - d[2], rp - self.csr @ d[0],
                 rc - self.z * d[0] - self.x * d[2])
            size = float(sum((v ** 2).sum() for v in e)) ** 0.5
            if not size < 0.5 * best:
                break
            best, out = size, [v.clone() for v in d]
            d = [a + b for a, b in zip(d, self._solve(*e))]
        return tuple(out)


def exact(case, seed):
    if case["shape"] == "full":
        return None   # the system solved is the library's own equality form of the LP
    lps = _lps(case, seed)
    what = case["what"]
    if what in ("solve", "gradient"):
        q = lps[0]   # the planted optimum, unique by its basis
        t = [torch.tensor(v, device=DEV) for v in (q.xstar, q.ystar, q.zstar)]
        if what == "solve":
            return tuple(t)
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        A, _, _ = _global_matrix(lps)
        w = torch.randn(A.shape[0], generator=g, dtype=torch.float64, device=DEV)
        B = torch.tensor(q.basis, device=DEV)
        # x_B = A_B^-1 b, y = A_B^-T c_B: d(c'x + w'y) / dc_B = x_B + A_B^-1 w, / db = y
        gc = t[0].clone()
        gc[B] += torch.linalg.solve(A.to_dense()[:, B], w)
        return (*t, gc, t[1])
    nt = sum(q.n_total for q in lps)
    mt = sum(q.m_total for q in lps)
    x, z, r, r2 = _point(case, nt, mt, seed)
    N = _Newton(lps, x, z)
    d = N.solve(*r)
    if what == "direction":
        return d, N.solve(*r2)
    # J' lam = g is the same symmetric system with right-hand side [g_x - Z X^-1 g_z; g_y]:
    # lam_x = dx, lam_y = dy of J (dx, dy, .) = (g_x, g_y, X (Z X^-1 g_z) = Z g_z)
    gx, gy, gz = r2
    lx, ly, _ = N.solve(gx, gy, z * gz)
    return d, (lx, ly, (gz - lx) / x)

"""Device allocations that fail: the call reports AHLP_ERR_OOM or does without the
memory, and the handle stays usable: the next call, with memory again, gives what an
undisturbed handle gives, bit for bit.

A child process runs with a shim in front of cudaMalloc that fails one chosen
allocation, so no device memory has to be used up.  Every allocation of a
handle's first factor is failed in turn (job tables, counters, staging, tensor
maps; the matrices of a precision that the factor moves to)."""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static long left = -1;          /* allocations until the one that fails; -1: none */
static long failed = 0;
void shim_fail_after(long n) { left = n; failed = 0; }
long shim_failed(void) { return failed; }
int cudaMalloc(void **p, size_t n) {
  static int (*real)(void **, size_t);
  if (!real) {
    void *h = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
    if (h) real = (int (*)(void **, size_t))dlsym(h, "cudaMalloc");
    if (!real) return 999;      /* cudaErrorUnknown */
  }
  if (left == 0) { left = -1; ++failed; return 2; }   /* cudaErrorMemoryAllocation */
  if (left > 0) --left;
  return real(p, n);
}
"""

CHILD = r"""
import ctypes, sys
import numpy as np
from instances import config3, random_block_lp
import paper_2412_07731_gb300 as P
from paper_2412_07731_gb300._lib import kkt_block_factor_dense

shim = ctypes.CDLL(sys.argv[1])
shim.shim_failed.restype = ctypes.c_long
prec, shape = sys.argv[2], sys.argv[3]
if shape == "large":        # more than 152 trailing tiles: the FP64 pipe's undivided updates
    lp = random_block_lp(6, N=2, m_sizes=[1300, 500], n_sizes=[1950, 750], nnz_per_col=4, n0=5,
                         w_density=0.3, l=2)
elif shape == "banded":     # a tile-sparse job table, blocks without a job at the next diagonal tile
    lp = config3(days=2)
else:
    lp = random_block_lp(5, N=3, m_sizes=[200, 150, 90], n_sizes=[300, 230, 140], nnz_per_col=4,
                         n0=5, w_density=0.3, l=2, mg=2, global_nnz=3)
kw = {"fp64": dict(), "fp32": dict(precision=P.PREC_MIXED, fp32_cond_max=1e300),
      "ff": dict(precision=P.PREC_MIXED, fp32_cond_max=1.0)}[prec]
rng = np.random.default_rng(9)
x, z = np.exp(rng.uniform(-1, 1, lp.n_total)), np.exp(rng.uniform(-1, 1, lp.n_total))

def factors(prob):
    return [kkt_block_factor_dense(prob, i) for i in range(lp.N)]

def make():
    return P.arrowhead_lp_create(lp, P.default_options(**kw))

prob = make()
P.kkt_factor(prob, x, z)
want = factors(prob)
prob.close()
tried = 0
for k in range(64):
    prob = make()
    shim.shim_fail_after(k)
    status = 0
    try:
        P.kkt_factor(prob, x, z)
    except P.AHLPError as e:
        status = e.status
    hit = shim.shim_failed()
    shim.shim_fail_after(-1)
    if not hit:
        prob.close()
        break
    tried += 1
    # FP64 factors need no memory beyond the handle's own: they fall back
    assert status == (0 if prec == "fp64" else -9), (k, status)
    if status == 0:
        for i, L in enumerate(factors(prob)):   # another rounding of the same factor
            m = lp.A[i].shape[0]
            V, W = L[:, :m], want[i][:, :m]
            s = np.sqrt((W ** 2).sum(1))
            d = np.abs(V @ V[:m].T - W @ W[:m].T)   # each within (m + 16) u of [M; G']
            assert (d <= 4 * (m + 16) * 2.0 ** -53 * np.outer(s, s[:m])).all(), (k, i)
    P.kkt_factor(prob, x, z)
    got = factors(prob)
    assert all(np.array_equal(a, b) for a, b in zip(got, want)), k
    prob.close()
print("allocations failed in turn:", tried)
assert tried >= int(sys.argv[4])
"""


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    cc = shutil.which("gcc") or shutil.which("cc")
    if not cc:
        pytest.skip("no C compiler")
    d = tmp_path_factory.mktemp("shim")
    src, lib = d / "shim.c", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run([cc, "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    return str(lib)


# at least: offsets and counters; digit planes and exponents | tensor maps and staging;
# on banded blocks also the job table and the blocks without a diagonal job
@pytest.mark.parametrize("prec,shape,least", [("fp64", "random", 4), ("fp64", "banded", 5),
                                              ("fp64", "large", 4),
                                              ("fp32", "random", 4), ("ff", "random", 5)])
def test_every_failed_allocation_leaves_the_handle_usable(shim, prec, shape, least):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, LD_PRELOAD=shim,
               PYTHONPATH=root + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CHILD, shim, prec, shape, str(least)], env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr

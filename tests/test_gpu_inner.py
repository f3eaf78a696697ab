"""The inner iteration's kernels (the product forms of the triangular solves,
the split updates) at the sizes where their tiling changes: one column, the
edges of the 32-row blocks, of the register tiles (64, 128, 256, 512 rows)
and of the four entries per CTA, and the largest n; for all three methods.

Bars as everywhere (C ABI, constructed problems): Karlson-Walden backward
error <= 1e-13, forward error within 10x of the oracle's Householder QR
solve; the step-2 count is Theorem 7.1's and step 1 stops by its rule."""
import numpy as np
import pytest

import oracle
import paper_2406_03468_gb300 as lsq
from gpu_util import H, T, empty
from lsq_problems import problem_svd

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 5, 31, 32, 33, 63, 64, 65, 127, 129, 255, 257, 511, 513, 700, 770, 1021, 1024]


@pytest.mark.parametrize("method", ["fossils", "spir", "spir_lsqr"])
@pytest.mark.parametrize("n", SIZES)
def test_inner_sizes(method, n):
    m = 12 * n + 61
    P = problem_svd(m, n, 1e6 if n > 1 else 1.0, 1e-4, seed=n, keep_factors=False)
    plan = lsq.Plan(m, n, seed=3)
    x = empty(n)
    st, info = plan.solve(T(P["A"]), T(P["b"]), x, method)
    xh = H(x)
    plan.close()
    assert st == 0
    x_qr, R_A = oracle.qr_solve_lapack(P["A"], P["b"], return_R=True)
    be = oracle.kw_relative(P["A"], P["b"], xh, R_A=R_A)
    assert be <= 1e-13, (be, info)
    # a forward error below 2^-50 is a correctly rounded answer's own level
    fe, fq = oracle.forward_error(xh, P["x_true"]), oracle.forward_error(x_qr, P["x_true"])
    assert fe <= 10 * max(fq, 2.0 ** -50), (fe, fq)
    assert 1 <= info["iters"][0] < 100
    if method == "fossils":
        assert info["iters"][1] == oracle.step2_updates(info["condest"], np.sqrt(1.0 / 12.0))

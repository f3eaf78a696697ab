"""Which form a many-right-hand-side solve takes, and that the library says so:
both passes in fixed point on the tensor cores, only the inner one (columns
whose typical entry lies between the two gates), neither (dominated columns;
multi_df; inner_fp64_fma).  Sizes with n % 4 != 0 and k = 64 also keep the
k-tiled double-float kernel covered at its edges, and its inner pass at n > 128.

Bars: the inner pass per element within 4 (n + m) u |A|^T |A| |z| of the
oracle's compensated A^T (A z) (the FP64 bound), every column of X backward
stable (Karlson-Walden <= 1e-13)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2406_03468_gb300 as lsq
from gpu_util import H, T, empty

pytestmark = pytest.mark.gpu
u = 2.0 ** -53


def _matrix(rng, m, n, kind):
    A = rng.standard_normal((m, n)) * 10.0 ** rng.uniform(-1, 1, n)
    if kind == "between":      # one entry of every row 2^6 above the others
        A[np.arange(m), rng.integers(0, n, m)] *= 2.0 ** 6
    elif kind == "dominated":  # one entry of every column 1e8 above the others
        A[rng.permutation(m)[:n], np.arange(n)] *= 10.0 ** rng.uniform(6, 10, n)
    return A


@pytest.mark.parametrize("m,n,k,kind,opts,form,kernel", [
    (2500, 24, 16, "plain", {}, 3, 5),
    (2500, 113, 64, "between", {}, 1, 5),
    (3001, 24, 8, "between", {}, 1, 5),
    (2500, 24, 16, "dominated", {}, 0, 5),
    (2500, 24, 16, "plain", {"multi_df": 1}, 0, 5),
    (2500, 24, 16, "plain", {"inner_fp64_fma": 1}, 0, 4),
    (1999, 130, 64, "plain", {"multi_df": 1}, 0, 5),
    (2500, 177, 32, "plain", {"multi_df": 1}, 0, 5),
    (2500, 241, 64, "plain", {"multi_df": 1}, 0, 5),
    (3001, 255, 64, "plain", {"multi_df": 1}, 0, 5)])
def test_form_is_reported(m, n, k, kind, opts, form, kernel):
    rng = np.random.default_rng(m + n + k)
    A, B = _matrix(rng, m, n, kind), rng.standard_normal((m, k))
    plan = lsq.Plan(m, n, seed=5, nrhs=k, **opts)
    dA, X, Hd = T(A), torch.empty((n, k), dtype=torch.float64, device="cuda"), empty(n * k)
    assert lsq.lsq_multi_form(plan.handle) == 0
    st, info = lsq.lsq_solve_fossils_multi(plan.handle, dA, T(B), k, X)
    assert st == 0 and lsq.lsq_multi_form(plan.handle) == form
    assert info.inner_kernel == kernel or (kernel == 5 and not form and info.inner_kernel == 3)
    Z = rng.standard_normal((k, n))
    lsq.lsq_apply_normal_multi(plan.handle, dA, T(Z), Hd)
    Xh, Hh = H(X), H(Hd).reshape(k, n)
    plan.close()
    absA = np.abs(A)
    for c in range(0, k, 5):
        h = oracle.residual_dot2(A, np.zeros(m), -Z[c])[2]
        bound = 4 * (n + m) * u * (absA.T @ (absA @ np.abs(Z[c])))
        assert (np.abs(Hh[c] - h) <= bound).all(), c
        assert oracle.kw_relative(A, B[:, c], Xh[:, c]) <= 1e-13, c


def test_leading_weights_are_exact():
    """Every digit large and of one sign, other third digits in every row, several
    accumulations per CTA: the sums of the three leading weights need all of
    FP32's 24 bits at 256 rows and would round beyond them (at 2^-38 of the result
    at 1024 rows).  A has 40 bits, so its digits are exact; what remains (z and y
    to 2^-55 of the largest, the dropped digit pairs, the FP64 sums) is below
    16 u of the result, which has no cancellation."""
    m, n, k = 160000, 24, 8
    rng = np.random.default_rng(9)
    q = np.full((m, n), 127 * 256 + 127, dtype=np.int64)
    q = q * 256 + rng.integers(64, 128, (m, n))
    q = q * 65536 + rng.integers(0, 65536, (m, n))          # 40 bits
    A = np.ldexp(q.astype(np.float64), -40)
    s = q.sum(axis=1)                                         # exact, < 2^45
    # y = z0 sum_j a_ij just below a power of two: its leading digits are 127 too
    z0 = (127 / 128 + 127 / 32768 + 60 / 2.0 ** 23) / (np.ldexp(float(s.mean()), -40))
    plan = lsq.Plan(m, n, seed=5, nrhs=k)
    dA, X, Hd = T(A), torch.empty((n, k), dtype=torch.float64, device="cuda"), empty(n * k)
    B = rng.standard_normal((m, k))
    # the columns are nearly equal: only the pass is of interest here
    lsq.lsq_solve_fossils_multi(plan.handle, dA, T(B), k, X)
    assert lsq.lsq_multi_form(plan.handle) & lsq.LSQ_MULTI_TC_INNER
    lsq.lsq_apply_normal_multi(plan.handle, dA, T(np.full((k, n), z0)), Hd)
    Hh = H(Hd).reshape(k, n)
    plan.close()
    for j in range(0, n, 6):
        exact = int((q[:, j].astype(object) * s.astype(object)).sum())   # units of 2^-80
        h = exact / 2 ** 80 * z0
        assert np.abs(Hh[:, j] - h).max() <= 16 * u * h, j


@pytest.mark.parametrize("n", [1, 2, 3, 7, 8, 13, 15, 33, 65])
def test_few_columns_strides_and_zeros(n):
    """Few columns (A x then has bits to spare in 64), lda > n and ldb > k with
    NaN between the rows, rows of zeros, a right-hand side of zeros."""
    m, k = 70 * n + 643, 24
    rng = np.random.default_rng(n)
    A = np.full((m, n + 3), np.nan)
    A[:, :n] = rng.standard_normal((m, n)) * 2.0 ** rng.integers(-3, 4, (m, 1))
    A[5:300:7, :n] = 0.0
    B = np.full((m, k + 5), np.nan)
    B[:, :k] = A[:, :n] @ rng.standard_normal((n, k)) + 0.1 * rng.standard_normal((m, k))
    B[:, 3] = 0.0
    plan = lsq.Plan(m, n, seed=5, nrhs=k, lda=n + 3)
    X = torch.empty((n, k), dtype=torch.float64, device="cuda")
    st, _ = lsq.lsq_solve_fossils_multi(plan.handle, T(A), T(B), k + 5, X)
    assert st == 0 and lsq.lsq_multi_form(plan.handle) == 3
    Xh = H(X)
    plan.close()
    A = np.ascontiguousarray(A[:, :n])
    assert not Xh[:, 3].any()
    for c in (0, 9, k - 1):
        assert oracle.kw_relative(A, np.ascontiguousarray(B[:, c]), Xh[:, c]) <= 1e-13, c


def test_plan_pointed_at_other_sizes():
    """One plan, its digits and sums reused for fewer rows and columns and back."""
    rng = np.random.default_rng(2)
    k = 40
    plan = lsq.Plan(3001, 200, seed=5, nrhs=k)
    for m, n in [(3001, 200), (1203, 90), (2999, 129), (700, 16), (3001, 200)]:
        lsq.lsq_plan_configure(plan.handle, lsq.lsq_options_default(m=m, n=n, seed=5, nrhs=k))
        A, B = rng.standard_normal((m, n)), rng.standard_normal((m, k))
        X = torch.empty((n, k), dtype=torch.float64, device="cuda")
        st, _ = lsq.lsq_solve_fossils_multi(plan.handle, T(A), T(B), k, X)
        assert st == 0 and lsq.lsq_multi_form(plan.handle) == 3
        Xh = H(X)
        for c in (0, k - 1):
            assert oracle.kw_relative(A, B[:, c], Xh[:, c]) <= 1e-13, (m, n, c)
    plan.close()

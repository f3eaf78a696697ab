"""Many right-hand sides on matrices whose rows differ in size by powers of two:
one direction of x is determined by a few percent of rows that are far smaller
than the others.  What the small rows hold must not be measured against the
large ones.

Reference: iterative refinement with the oracle's compensated residuals from
LAPACK's QR, to convergence (kappa < 1e10).  Bars: the forward error within
10x of the same solve on the plan's FP64 kernels (inner_fp64_fma = 1; 2^-50
is a correctly rounded answer's own level), and within 10x of the QR solve's
own."""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_2406_03468_gb300 as lsq
from gpu_util import H, T

pytestmark = pytest.mark.gpu


def _solve(A, B, **opts):
    n, k = A.shape[1], B.shape[1]
    plan = lsq.Plan(*A.shape, seed=1, nrhs=k, **opts)
    X = torch.empty((n, k), dtype=torch.float64, device="cuda")
    st, _ = lsq.lsq_solve_fossils_multi(plan.handle, T(A), T(B), k, X)
    plan.close()
    assert st == 0
    return H(X)


@pytest.mark.parametrize("e", [0, -6, -14, -30])
@pytest.mark.parametrize("noise", [0.0, 1.0])
def test_small_rows_keep_their_bits(e, noise):
    m, n, k, small = 20000, 32, 8, 1000
    rng = np.random.default_rng(11)
    A = rng.standard_normal((m, n))
    A[:, n - 1] = A[:, :n - 1] @ rng.standard_normal(n - 1) / math.sqrt(n)
    A[:small] = rng.standard_normal((small, n)) * 2.0 ** e
    A = A[rng.permutation(m)]
    rows = np.abs(A).max(axis=1) < 2.0 ** (e / 2) if e < -6 else np.zeros(m, bool)
    B = A @ (np.round(rng.standard_normal((n, k)) * 256) / 256)
    B += noise * 2.0 ** e * rng.standard_normal((m, k)) * rows[:, None]  # in the small rows only
    X, X64 = _solve(A, B), _solve(A, B, inner_fp64_fma=1)
    Q, R = np.linalg.qr(A)
    for c in (0, k - 1):
        x = np.linalg.solve(R, Q.T @ B[:, c])
        fq = x.copy()
        for _ in range(8):
            g = oracle.residual_dot2(A, B[:, c], x)[2]
            x = x + np.linalg.solve(R, np.linalg.solve(R.T, g))
        err = [np.linalg.norm(v - x) / np.linalg.norm(x) for v in (X[:, c], X64[:, c], fq)]
        assert err[0] <= 10 * max(err[1], 2.0 ** -50), (c, err)
        assert err[0] <= 10 * max(err[2], 2.0 ** -50), (c, err)


def test_apply_after_a_refused_solve():
    """A refused solve leaves no digits or planes behind: the pass that follows
    works on the matrix it is given (bound: 4 (n + m) u |A|^T |A| |z|)."""
    m, n, k = 3000, 24, 8
    rng = np.random.default_rng(3)
    A, B = rng.standard_normal((m, n)), rng.standard_normal((m, k))
    plan = lsq.Plan(m, n, seed=1, nrhs=k)
    X = torch.empty((n, k), dtype=torch.float64, device="cuda")
    assert lsq.lsq_solve_fossils_multi(plan.handle, T(A), T(B), k, X)[0] == 0
    bad = A.copy()
    bad[7, 3] = np.nan
    with pytest.raises(lsq.LsqError):
        lsq.lsq_solve_fossils_multi(plan.handle, T(bad), T(B), k, X)
    C, Z = rng.standard_normal((m, n)), rng.standard_normal((k, n))
    Hd = torch.empty(n * k, dtype=torch.float64, device="cuda")
    lsq.lsq_apply_normal_multi(plan.handle, T(C), T(Z), Hd)
    Hh = H(Hd).reshape(k, n)
    plan.close()
    absC = np.abs(C)
    for c in range(k):
        h = oracle.residual_dot2(C, np.zeros(m), -Z[c])[2]
        bound = 4 * (n + m) * 2.0 ** -53 * (absC.T @ (absC @ np.abs(Z[c])))
        assert (np.abs(Hh[c] - h) <= bound).all(), c

"""The fixed-point residual pass against the FP64 one: the answers of the
tensor-core form are no further from the exact solution than those of the
same solve on the plan's FP64 kernels (inner_fp64_fma = 1).

Exact solution: refinement with the oracle's compensated residuals from
LAPACK's QR.  Compared is the root mean square over 64 right-hand sides; both
forms' errors are sums of many roundings, so that figure spreads by 1 / sqrt(128)
of itself: bar 1.5 times the larger of the FP64 form's and 2^-52 (the rounding
of the answer itself)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2406_03468_gb300 as lsq
from gpu_util import H, T

pytestmark = pytest.mark.gpu


def _problem(m, n, k, kind, graded_x, rho, seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((m, n))
    if kind == "spiky rows":  # one entry of every row 11 times the others
        A[np.arange(m), rng.integers(0, n, m)] *= 2.0 ** 3.5
    else:                     # condition 1e3 or 1e6
        V = np.linalg.qr(rng.standard_normal((n, n)))[0]
        A = np.ascontiguousarray((A * np.logspace(0, -kind, n)) @ V.T)
    X = rng.standard_normal((n, k)) * 10.0 ** rng.uniform(-graded_x, 0, (n, 1))
    B = A @ X
    B += rho * np.linalg.norm(B, axis=0) / np.sqrt(m) * rng.standard_normal((m, k))
    Q, R = np.linalg.qr(A)
    ref = np.linalg.solve(R, Q.T @ B)
    for c in range(k):
        for _ in range(5):
            g = oracle.residual_dot2(A, B[:, c], ref[:, c])[2]
            ref[:, c] += np.linalg.solve(R, np.linalg.solve(R.T, g))
    return A, np.ascontiguousarray(B), ref


@pytest.mark.parametrize("m,n,kind,graded_x,rho", [
    (20000, 16, 3, 3, 0.0), (20000, 16, 6, 0, 0.0), (400, 16, 6, 3, 0.3), (5000, 48, 6, 0, 0.3),
    (1000, 64, "spiky rows", 3, 0.0), (1000, 64, "spiky rows", 0, 0.3),
    (2500, 129, "spiky rows", 3, 0.0), (3000, 200, 3, 3, 0.0)])
def test_no_further_off_than_fp64(m, n, kind, graded_x, rho):
    err = {}
    k = 32
    for seed in (1, 2):
        A, B, ref = _problem(m, n, k, kind, graded_x, rho, seed)
        for opts in ({}, {"inner_fp64_fma": 1}):
            plan = lsq.Plan(m, n, seed=1, nrhs=k, **opts)
            X = torch.empty((n, k), dtype=torch.float64, device="cuda")
            st, _ = lsq.lsq_solve_fossils_multi(plan.handle, T(A), T(B), k, X)
            form = lsq.lsq_multi_form(plan.handle)
            plan.close()
            assert st == 0 and form == (0 if opts else 3)
            e = np.linalg.norm(H(X) - ref, axis=0) / np.linalg.norm(ref, axis=0)
            err.setdefault(form, []).extend(e)
    tc, fp64 = (float(np.sqrt(np.mean(np.square(err[f])))) for f in (3, 0))
    assert tc <= 1.5 * max(fp64, 2.0 ** -52), (tc, fp64)

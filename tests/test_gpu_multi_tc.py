"""The tensor-core passes of the many-right-hand-side solve at the edges of
their tiles: rows around 64 and 128, column counts around 16, 64 and 128 (the
packed last column chunk), vector counts that pad to 16, 32, 48 and 64, fewer
rows than one tile; and a matrix whose columns are dominated by single
entries, where the library takes the double-float form.

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


@pytest.mark.parametrize("m,n,k,outlier", [
    (100, 16, 8, False), (127, 17, 16, False), (129, 31, 24, False), (640, 64, 40, False),
    (1025, 65, 48, False), (2000, 112, 56, False), (1999, 113, 64, False), (3001, 129, 8, False),
    (2500, 177, 32, False), (2500, 241, 64, False), (5000, 24, 16, True)])
def test_multi_tc_edges(m, n, k, outlier):
    rng = np.random.default_rng(m + 3 * n + k)
    A = rng.standard_normal((m, n)) * 10.0 ** rng.uniform(-1, 1, n)
    if outlier:
        A[rng.permutation(m)[:n], np.arange(n)] *= 1e6
    B = rng.standard_normal((m, k))
    plan = lsq.Plan(m, n, seed=5, nrhs=k)
    dA = T(A)
    X = torch.empty((n, k), dtype=torch.float64, device="cuda")
    st, info = lsq.lsq_solve_fossils_multi(plan.handle, dA, T(B), k, X)
    assert st == 0 and info.inner_kernel == 5
    Xh = H(X)
    Z = rng.standard_normal((k, n))
    Hd = empty(n * k)
    lsq.lsq_apply_normal_multi(plan.handle, dA, T(Z), Hd)
    Hh = H(Hd).reshape(k, n)
    plan.close()
    absA = np.abs(A)
    for c in range(0, k, 5):
        _, _, h = oracle.residual_dot2(A, np.zeros(m), -Z[c])
        bound = 4 * (n + m) * u * (absA.T @ (absA @ np.abs(Z[c])))
        assert (np.abs(Hh[c] - h) <= bound).all(), c
        assert oracle.kw_relative(A, B[:, c], Xh[:, c]) <= 1e-13, c


def test_multi_tc_equal_rows():
    """Runs of equal rows whose entries have the digit 127 in every place: the
    digit products of a run all add up with one sign.  |A| and |z| lie within a
    factor 2, so every rounding of the fixed-point pass (A, z, y to 2^-56 of the
    largest, the dropped digit pairs) is below 2 u of |A|^T |A| |z| and all of
    them together below 16 u."""
    runs, run, n, k = 30, 1100, 24, 8
    m = runs * run
    rng = np.random.default_rng(7)
    v = sum(127.0 * 256.0 ** -(t + 1) for t in range(6))
    A = np.repeat(v * rng.choice([-1.0, 1.0], (runs, n)), run, axis=0)
    plan = lsq.Plan(m, n, seed=5, nrhs=k)
    dA = T(A)
    X = torch.empty((n, k), dtype=torch.float64, device="cuda")
    st, info = lsq.lsq_solve_fossils_multi(plan.handle, dA, T(rng.standard_normal((m, k))), k, X)
    assert st == 0 and info.inner_kernel == 5
    Z = rng.choice([-1.0, 1.0], (k, n)) * rng.uniform(0.5, 1.0, (k, n))
    Hd = empty(n * k)
    lsq.lsq_apply_normal_multi(plan.handle, dA, T(Z), Hd)
    Hh = H(Hd).reshape(k, n)
    plan.close()
    absA = np.abs(A)
    for c in range(k):
        _, _, h = oracle.residual_dot2(A, np.zeros(m), -Z[c])
        assert (np.abs(Hh[c] - h) <= 16 * u * (absA.T @ (absA @ np.abs(Z[c])))).all(), c

"""Both sides of the size rules that choose a kernel: the QR's column-by-column
and blocked forms (n = 7 / 8) with partial first panels (n = 9 .. 17) and, at d =
3n, panel CTAs that hold no rows; its one-stream and two-stream forms (768 / 769);
the Karlson-Walden test's QR of a 16 x 8 matrix; the CSR pass whose rows are
staged in shared memory at the largest n.

Bars: R and t within 1e3 n u of the oracle's Householder QR of the same sketch
(kappa <= 30); answers backward stable (Karlson-Walden <= 1e-13)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2406_03468_gb300 as lsq
from gpu_util import H, T, empty

pytestmark = pytest.mark.gpu
u = 2.0 ** -53


def _problem(m, n, seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((m, n)) * 10.0 ** rng.uniform(-0.5, 0.5, n)
    return A, A @ rng.standard_normal(n) + 0.1 * rng.standard_normal(m)


@pytest.mark.parametrize("n,times", [(n, t) for n in (7, 8, 9, 15, 16, 17) for t in (3, 12)]
                         + [(768, 3), (769, 3)])
def test_qr_of_sketch(n, times):
    m, d = 4 * times * n, times * n
    A, b = _problem(m, n, seed=n)
    plan = lsq.Plan(m, n, seed=4, d=d)
    lsq.lsq_sketch(plan.handle, T(A), T(b))
    S, R, t = empty(d * (n + 1)), empty(n * n), empty(n)
    lsq.lsq_get_sketch(plan.handle, S, None)
    lsq.lsq_get_R(plan.handle, R, t)
    S, R, t = H(S).reshape(n + 1, d).T, H(R).reshape(n, n), H(t)
    plan.close()
    R_or, V = oracle.householder_qr(S[:, :n])
    t_or = oracle.apply_qt(V, S[:, n])[:n]
    assert np.linalg.cond(R_or) <= 30 and not np.tril(R, -1).any()
    assert np.linalg.norm(R - R_or, 2) <= 1e3 * n * u * np.linalg.norm(R_or, 2)
    assert np.linalg.norm(t - t_or) <= 1e3 * n * u * np.linalg.norm(S[:, n])


@pytest.mark.parametrize("method", ["fossils", "spir", "spir_lsqr"])
@pytest.mark.parametrize("n,opts", [(7, {}), (8, {}), (9, {}), (15, {}), (16, {}), (17, {}),
                                    (8, {"d": 24}), (15, {"d": 45}), (8, {"kw_stop": 1})])
def test_solve(n, opts, method):
    A, b = _problem(40 * n + 3, n, seed=100 + n)
    plan = lsq.Plan(*A.shape, seed=3, **opts)
    x = empty(n)
    st, info = plan.solve(T(A), T(b), x, method)
    x = H(x)
    plan.close()
    assert st == 0 and oracle.kw_relative(A, b, x) <= 1e-13, info


@pytest.mark.parametrize("method", [0, 1, 2])
@pytest.mark.parametrize("n", [1000, 1024])
def test_csr_staged_largest(n, method):
    m, per = 5003, 24
    rng = np.random.default_rng(n)
    col = np.sort(np.argsort(rng.random((m, n)), axis=1)[:, :per], axis=1).astype(np.int32)
    val = rng.standard_normal((m, per))
    A = np.zeros((m, n))
    np.put_along_axis(A, col.astype(np.int64), val, axis=1)
    b = rng.standard_normal(m)
    rp = np.arange(m + 1, dtype=np.int64) * per
    plan = lsq.Plan(m, n, seed=3, sparse=1, d=4 * n)
    x = empty(n)
    dev = [torch.from_numpy(a).cuda() for a in (rp, col.ravel(), val.ravel(), b)]
    st, _ = lsq.lsq_solve_csr(plan.handle, method, *dev, x)
    x = H(x)
    plan.close()
    assert st == 0 and oracle.kw_relative(A, b, x) <= 1e-13

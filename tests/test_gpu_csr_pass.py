"""The CSR passes on ragged rows: empty rows, rows of 1 to 33 entries and
longer, 8 consecutive rows that do not fit the staged pass's 256 entries, row
counts around its blocks of 8 and 64 rows, fewer rows than CTAs; and mean row
lengths beyond 32, where the unstaged pass runs.

Bars: the answer backward stable (Karlson-Walden <= 1e-13) and, per element,
within 100 (n + m) u kappa ||x|| of the oracle's Householder QR solve (both
solve the same well-conditioned problem, kappa < 30, residual included)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2406_03468_gb300 as lsq
from gpu_util import H, empty

pytestmark = pytest.mark.gpu
u = 2.0 ** -53


def _ragged(m, n, lengths, weights, seed):
    rng = np.random.default_rng(seed)
    lens = np.minimum(rng.choice(lengths, m, p=weights), n)
    lens[:2 * n:2] = np.maximum(lens[:2 * n:2], min(n, 8))  # every column is met
    rp = np.concatenate(([0], np.cumsum(lens))).astype(np.int64)
    col = np.concatenate([np.sort(rng.permutation(n)[:k]) for k in lens]).astype(np.int32)
    val = rng.standard_normal(rp[-1])
    A = np.zeros((m, n))
    for i in range(m):
        A[i, col[rp[i]:rp[i + 1]]] = val[rp[i]:rp[i + 1]]
    return rp, col, val, A, rng.standard_normal(m)


@pytest.mark.parametrize("method", [0, 1, 2])
@pytest.mark.parametrize("m,n,lengths,weights", [
    (1999, 40, [0, 1, 3, 8], [0.1, 0.3, 0.3, 0.3]),
    (4003, 130, [0, 5, 31, 32, 33, 100, 130], [0.1, 0.5, 0.1, 0.1, 0.1, 0.08, 0.02]),
    (30001, 64, [2, 32, 33], [0.3, 0.4, 0.3]),
    (2065, 100, [32], [1.0]),
    (2500, 130, [20, 64, 129], [0.4, 0.3, 0.3])])
def test_csr_ragged(m, n, lengths, weights, method):
    rp, col, val, A, b = _ragged(m, n, lengths, weights, seed=m + n)
    plan = lsq.Plan(m, n, seed=3, sparse=1)
    dx = empty(n)
    dev = [torch.from_numpy(a).cuda() for a in (rp, col, val, b)]
    st, _ = lsq.lsq_solve_csr(plan.handle, method, *dev, dx)
    plan.close()
    assert st == 0
    x = H(dx)
    x_qr, R_A = oracle.qr_solve(A, b, return_R=True)
    sv = np.linalg.svd(A, compute_uv=False)
    assert sv[0] < 30 * sv[-1]
    assert oracle.kw_relative(A, b, x, R_A=R_A) <= 1e-13
    scale = np.linalg.norm(x_qr) + np.linalg.norm(b) / sv[-1]
    assert np.abs(x - x_qr).max() <= 100 * (n + m) * u * (sv[0] / sv[-1]) * scale

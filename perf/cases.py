"""Performance cases of the least-squares library: what a user's program has it
do, through the public entry points, from the smallest solves (launch and
latency bound) to the largest (bound by the passes over A).

Every problem is built on the GPU from its seed: A = (G / sqrt(m)) diag(sigma)
V^T with Gaussian G, log-spaced sigma (1 .. 1 / kappa) and Haar V, and
b = A x + r with ||r|| = rho ||A x||.  rho = min(0.5, 10 / kappa): the relative
residuals of regression problems (0.5) where A is well conditioned, falling to
those of fits to nearly exact data (Prony's method) where it is not.
"""
import math
import random

import numpy as np
import torch

import paper_2406_03468_gb300 as lsq

F64 = torch.float64


def listed():
    return [
        # one small problem at a time (the paper's Fig. 1 shape): launches and latency
        dict(name="fossils_4000x50", kind="solve", method="fossils", precision=1, m=4000, n=50,
             kappa=1e4),
        # small and odd in both sizes, conjugate gradient inner solver
        dict(name="spir_20011x97", kind="solve", method="spir", precision=1, m=20011, n=97,
             kappa=1e3),
        # one request of a served stream (m 2e4..4e5, n 32..256)
        dict(name="fossils_120000x128", kind="solve", method="fossils", precision=1, m=120000,
             n=128, kappa=1e5),
        # the headline size: kernel-regression-like, 4 GB of A
        dict(name="fossils_1000000x500", kind="solve", method="fossils", precision=1, m=1000000,
             n=500, kappa=1e4),
        # LSQR-based SPIR on an odd, ragged size
        dict(name="lsqr_300007x333", kind="solve", method="spir_lsqr", precision=1, m=300007,
             n=333, kappa=1e3),
        # the mixed-precision tier (chosen by the library from its condition estimate), wide A
        dict(name="auto_400000x1000", kind="solve", method="fossils", precision=0, m=400000,
             n=1000, kappa=1e4),
        # many right-hand sides on one matrix
        dict(name="multi_500000x200_k64", kind="multi", m=500000, n=200, k=64, kappa=1e4),
        # a batch of independent uneven problems, as a server collects them
        dict(name="batch_32", kind="batch", count=32, m_lo=20000, m_hi=400000, sizes=11,
             kappa=1e4),
        # a sparse matrix in CSR form, SPIR with the small sketch (d = 3n)
        dict(name="csr_500000x500_d3n", kind="csr", method=1, m=500000, n=500, per_row=32,
             d_over_n=3, delta=1e-4),
        # complex: the first solve of Prony's method
        dict(name="complex_200000x128", kind="complex", method=0, m=200000, n=128),
        # data in page-locked host memory, solved end to end
        dict(name="host_200000x300", kind="host", method=0, m=200000, n=300, kappa=1e4),
        # sketch, QR and condition estimate alone: a preconditioner for the caller's own solver
        dict(name="sketch_400000x256", kind="sketch", m=400000, n=256, kappa=1e4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "multi", "batch", "csr", "complex",
                       "host", "sketch"])
    kappa = 10.0 ** rng.randint(1, 5)
    if kind == "multi":
        n = _log(rng, 16, 256)
        return dict(kind=kind, m=_log(rng, max(5000, 40 * n), 300000), n=n,
                    k=8 * rng.randint(1, 8), kappa=kappa)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 32), m_lo=_log(rng, 5000, 20000),
                    m_hi=_log(rng, 40000, 400000), sizes=rng.randint(0, 10 ** 6), kappa=kappa)
    if kind == "csr":
        n = 2 * _log(rng, 32, 250)
        return dict(kind=kind, method=rng.choice([0, 1, 2]), m=_log(rng, 20000, 500000), n=n,
                    per_row=2 * rng.randint(4, 16), d_over_n=12, delta=10.0 ** -rng.randint(2, 4))
    if kind == "complex":
        n = _log(rng, 16, 200)
        return dict(kind=kind, method=rng.choice([0, 1, 2]), m=_log(rng, 50 * n, 200000), n=n)
    if kind == "host":
        n = _log(rng, 16, 400)
        return dict(kind=kind, method=rng.choice([0, 1]), m=_log(rng, 40 * n, 200000), n=n,
                    kappa=kappa)
    n = _log(rng, 16, 1000)
    m = _log(rng, max(2000, 20 * n), min(1000000, 300000000 // n))
    if kind == "sketch":
        return dict(kind=kind, m=m, n=n, kappa=kappa)
    return dict(kind=kind, method=rng.choice(["fossils", "spir", "spir_lsqr"]),
                precision=rng.choice([0, 1, 1]), m=m, n=n, kappa=kappa)


# ---- inputs ----------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, dtype=F64, device="cuda")


def _matrix(g, m, n, kappa):
    V, R = torch.linalg.qr(_randn(g, n, n))
    V = V * torch.sign(torch.diagonal(R))
    sigma = torch.logspace(0.0, -math.log10(kappa), n, dtype=F64, device="cuda")
    W = (sigma[:, None] * V.T) / math.sqrt(m)
    A = torch.empty(m, n, dtype=F64, device="cuda")
    for i in range(0, m, 131072):
        j = min(m, i + 131072)
        torch.matmul(_randn(g, j - i, n), W, out=A[i:j])
    return A


def _rhs(g, A, kappa, k=None):
    m, n = A.shape
    X = _randn(g, n, k or 1)
    B = A @ X
    E = _randn(g, m, k or 1)
    E *= min(0.5, 10.0 / kappa) * torch.linalg.norm(B, dim=0) / torch.linalg.norm(E, dim=0)
    B += E
    return B if k else B[:, 0].contiguous()


def _dense(g, m, n, kappa):
    A = _matrix(g, m, n, kappa)
    return A, _rhs(g, A, kappa)


def _batch_sizes(case):
    rng = random.Random(case["sizes"])
    out = []
    for _ in range(case["count"]):
        n = rng.choice([32, 64, 128, 256, rng.randint(20, 256)])
        out.append((_log(rng, max(case["m_lo"], 20 * n), case["m_hi"]), n))
    return out


def _csr(g, m, n, per_row, delta):
    """CSR rows of per_row entries in column pairs (2q, 2q + 1) with nearly
    dependent values (condition about 1 / delta), columns scaled by 10^U(-2, 2)."""
    h, w = n // 2, per_row // 2
    units = torch.tensor([u for u in range(1, h + 1) if math.gcd(u, h) == 1], device="cuda")
    start = torch.randint(0, h, (m, 1), generator=g, device="cuda")
    step = units[torch.randint(0, len(units), (m, 1), generator=g, device="cuda")]
    q = ((start + torch.arange(w, device="cuda") * step) % h).sort(dim=1).values
    col = torch.stack((2 * q, 2 * q + 1), dim=2).reshape(m, per_row)
    a = _randn(g, m, w)
    val = torch.stack((a, a * (1.0 + delta * _randn(g, m, w))), dim=2).reshape(m, per_row)
    scale = 10.0 ** (4.0 * torch.rand(n, generator=g, dtype=F64, device="cuda") - 2.0)
    val *= scale[col]
    b = (val * (_randn(g, n) / math.sqrt(n))[col]).sum(dim=1)
    b += 1e-3 * _randn(g, m)
    rp = torch.arange(m + 1, dtype=torch.int64, device="cuda") * per_row
    return rp, col.to(torch.int32).reshape(-1).contiguous(), val.reshape(-1).contiguous(), b


def _prony(g, m, n):
    """A[i, j] = f[n - 1 + i - j], b[i] = f[n + i] for noisy samples f of a sum
    of n undamped exponentials."""
    lam = (6.0 * torch.rand(n, generator=g, dtype=F64, device="cuda") - 3.0).sort().values
    mu = -torch.log(torch.rand(n, generator=g, dtype=F64, device="cuda"))
    mu = (mu / mu.sum()).to(torch.complex128)
    f = torch.empty(m + n, dtype=torch.complex128, device="cuda")
    for i in range(0, m + n, 65536):
        j = torch.arange(i, min(m + n, i + 65536), dtype=F64, device="cuda")
        f[i:i + len(j)] = torch.exp(-0.25j * (j[:, None] * lam[None, :])) @ mu
    f += 1e-6 / math.sqrt(2.0) * torch.complex(_randn(g, m + n), _randn(g, m + n))
    A = f.unfold(0, n, 1)[:m].flip(1).contiguous()
    return A, f[n:n + m].contiguous()


def _inputs(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind == "batch":
        return [_dense(g, m, n, case["kappa"]) for m, n in _batch_sizes(case)]
    if kind == "csr":
        return _csr(g, case["m"], case["n"], case["per_row"], case["delta"])
    if kind == "complex":
        return _prony(g, case["m"], case["n"])
    if kind == "multi":
        A = _matrix(g, case["m"], case["n"], case["kappa"])
        return A, _rhs(g, A, case["kappa"], case["k"])
    return _dense(g, case["m"], case["n"], case["kappa"])


# ---- what a user's program has before the call, and the call ----------------

class _Batch:
    """Owns a batch handle."""

    def __init__(self, count, n_max, elems):
        self.handle = lsq.lsq_batch_create(count, n_max, elems)

    def __del__(self):
        lsq.lsq_batch_destroy(self.handle)


def _empty(*shape):
    return torch.empty(*shape, dtype=F64, device="cuda")


def prepare(case, seed):
    kind, data = case["kind"], _inputs(case, seed)
    st = {"kind": kind, "case": case}
    if kind == "batch":
        sizes = _batch_sizes(case)
        st["items"] = [(A, b, _empty(A.shape[1])) for A, b in data]
        st["seeds"] = list(range(1, len(sizes) + 1))
        st["batch"] = _Batch(len(sizes), 256, sum(m * ((n + 3) // 4 * 4) for m, n in sizes))
        torch.cuda.synchronize()
        return st
    m, n = case["m"], case["n"]
    if kind == "solve":
        st["plan"] = lsq.Plan(m, n, seed=1, precision=case["precision"])
        st["A"], st["b"] = data
        st["x"] = _empty(n)
    elif kind == "multi":
        st["plan"] = lsq.Plan(m, n, seed=1, nrhs=case["k"])
        st["A"], st["B"] = data
        st["X"] = _empty(n, case["k"])
    elif kind == "csr":
        st["plan"] = lsq.Plan(m, n, seed=1, sparse=1, d=case["d_over_n"] * n)
        st["csr"], st["b"] = data[:3], data[3]
        st["x"] = _empty(n)
    elif kind == "complex":
        st["plan"] = lsq.Plan(2 * m, 2 * n, seed=1)
        st["A"], st["b"] = data
        st["x"] = torch.empty(n, dtype=torch.complex128, device="cuda")
        st["work"] = _empty(4 * m * n)
    elif kind == "host":
        st["plan"] = lsq.Plan(m, n, seed=1)
        st["A"], st["b"] = data[0].cpu().pin_memory(), data[1].cpu().pin_memory()
        st["x"] = torch.empty(n, dtype=F64).pin_memory()
    else:
        st["plan"] = lsq.Plan(m, n, seed=1)
        st["A"], st["b"] = data
        st["R"], st["t"], st["x0"] = _empty(n, n), _empty(n), _empty(n)
        st["SAb"], st["colnorm"] = _empty(n + 1, 12 * n), _empty(n)
    torch.cuda.synchronize()
    return st


def run(st):
    kind = st["kind"]
    if kind == "batch":
        lsq.lsq_batch_solve(st["batch"].handle, st["items"], seeds=st["seeds"])
        return [x for _, _, x in st["items"]]
    h = st["plan"].handle
    if kind == "solve":
        st["plan"].solve(st["A"], st["b"], st["x"], st["case"]["method"])
        return st["x"]
    if kind == "multi":
        lsq.lsq_solve_fossils_multi(h, st["A"], st["B"], 0, st["X"])
        return st["X"]
    if kind == "csr":
        lsq.lsq_solve_csr(h, st["case"]["method"], *st["csr"], st["b"], st["x"])
        return st["x"]
    if kind == "complex":
        lsq.lsq_solve_complex(h, st["case"]["method"], st["A"], st["b"], st["x"], st["work"])
        return st["x"]
    if kind == "host":
        lsq.lsq_solve_host(h, st["case"]["method"], st["A"], st["b"], st["x"])
        return st["x"]
    lsq.lsq_sketch(h, st["A"], st["b"])
    lsq.lsq_get_R(h, R=st["R"], t=st["t"], x0=st["x0"])
    lsq.lsq_get_sketch(h, st["SAb"], st["colnorm"])
    return {"R": st["R"], "t": st["t"], "x0": st["x0"], "SAb": st["SAb"],
            "colnorm": st["colnorm"]}


# ---- what a pass cannot do without ------------------------------------------

def _solve_flops(m, n, kappa, d_over_n=12, nnz=None, k=1):
    """Sketch (8 nonzeros per column), QR of the sketch, and the 4 flops per
    entry of A of each residual and inner pass.  The inner updates of the two
    steps contract by sqrt(n / d) each, together from 1 to u / kappa."""
    nnz = m * n if nnz is None else nnz
    updates = 2.0 * math.log(1.0 / (kappa * 1.1e-16)) / math.log(math.sqrt(d_over_n))
    return 16.0 * nnz + 2.0 * d_over_n * n * n * n + 4.0 * nnz * k * (2.0 + max(updates, 11.0))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        sizes = _batch_sizes(case)
        return {"bytes": sum(8.0 * (m * n + m + n) for m, n in sizes),
                "flops": sum(_solve_flops(m, n, case["kappa"]) for m, n in sizes)}
    m, n = case["m"], case["n"]
    if kind == "multi":
        k = case["k"]
        return {"bytes": 8.0 * (m * n + m * k + n * k),
                "flops": _solve_flops(m, n, case["kappa"], k=k)}
    if kind == "csr":
        nnz = m * case["per_row"]
        return {"bytes": 12.0 * nnz + 8.0 * (2 * m + 1 + n),
                "flops": _solve_flops(m, n, 1.0 / case["delta"], case["d_over_n"], nnz)}
    if kind == "complex":
        return {"bytes": 16.0 * (m * n + m + n),
                "flops": _solve_flops(m, 2 * n, 1e6) + 2.0 * 4.0 * m * n}
    if kind == "sketch":
        return {"bytes": 8.0 * (m * n + m + n * n + 2 * n + 12 * n * (n + 1)),
                "flops": 16.0 * m * n + 24.0 * n * n * n}
    return {"bytes": 8.0 * (m * n + m + n), "flops": _solve_flops(m, n, case["kappa"])}


# ---- the same results in plain 64-bit torch ----------------------------------

def _lstsq(A, B):
    """min ||B - A X||: Cholesky factor of the scaled Gram matrix, then
    refinement with 64-bit residuals until the correction stalls."""
    s = torch.linalg.norm(A, dim=0)
    Gm = (A.mH @ A) / s[:, None] / s[None, :]
    L = torch.linalg.cholesky(Gm)
    X = torch.zeros(A.shape[1], B.shape[1], dtype=A.dtype, device=A.device)
    for _ in range(12):
        g = (A.mH @ (B - A @ X)) / s[:, None]
        X = X + torch.cholesky_solve(g, L) / s[:, None]
    return X


def exact(case, seed):
    kind, data = case["kind"], _inputs(case, seed)
    if kind == "batch":
        return [_lstsq(A, b[:, None])[:, 0] for A, b in data]
    if kind == "multi":
        return _lstsq(*data)
    if kind == "csr":
        m, n = case["m"], case["n"]
        A = torch.zeros(m, n, dtype=F64, device="cuda")
        A.scatter_(1, data[1].reshape(m, -1).long(), data[2].reshape(m, -1))
        return _lstsq(A, data[3][:, None])[:, 0]
    if kind == "sketch":
        # S depends on the library's own random pattern; the column norms do not
        norms = np.sqrt((data[0] * data[0]).sum(dim=0).cpu().numpy())
        return {"R": None, "t": None, "x0": None, "SAb": None, "colnorm": norms}
    x = _lstsq(data[0], data[1][:, None])[:, 0]
    return x.cpu() if kind == "host" else x

"""The batched engine's lo planes start on a 16-byte boundary whatever plane
capacity the caller asks for (their rows are fetched with bulk copies).

The capacity is a promise of its own: a batch that needs more elements than
elems_max is refused, also where rounding it up would hold the batch."""
import ctypes

import pytest

import oracle
import paper_2406_03468_gb300 as lsq
from lsq_problems import problem_svd


def test_plane_offset_is_16_byte_aligned():
    lib = ctypes.CDLL(lsq.library_path())
    f = lib["_ZN3lsq18batch_plane_floatsEl"]
    f.restype, f.argtypes = ctypes.c_int64, [ctypes.c_int64]
    for e in (1, 2, 3, 4, 5, 1023, 1024, 2 ** 33 + 1, 2 ** 33 + 2, 2 ** 33 + 3):
        assert f(e) % 4 == 0 and e <= f(e) < e + 4, e


@pytest.mark.gpu
@pytest.mark.parametrize("extra", [0, 1, 2, 3])
def test_batch_with_any_plane_capacity(extra):
    from gpu_util import H, T, empty
    shapes = [(1501, 30, 1e3), (2003, 17, 1e6)]
    elems = sum(m * ((n + 3) // 4 * 4) for m, n, _ in shapes)
    Ps = [problem_svd(m, n, k, 1e-6, seed=i, keep_factors=False)
          for i, (m, n, k) in enumerate(shapes)]
    dev = [(T(P["A"]), T(P["b"]), empty(P["A"].shape[1])) for P in Ps]
    h = lsq.lsq_batch_create(2, 32, elems + extra)
    st, stats, _ = lsq.lsq_batch_solve(h, dev, seeds=[1, 2])
    lsq.lsq_batch_destroy(h)
    assert st >= 0 and all(s >= 0 for s in stats)
    for P, (_, _, x) in zip(Ps, dev):
        assert oracle.kw_relative(P["A"], P["b"], H(x)) <= 1e-13
    if extra == 0:
        h = lsq.lsq_batch_create(2, 32, elems - 1)
        with pytest.raises(lsq.LsqError):
            lsq.lsq_batch_solve(h, dev, seeds=[1, 2])
        lsq.lsq_batch_destroy(h)

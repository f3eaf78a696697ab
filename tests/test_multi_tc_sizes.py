"""The buffers of the tensor-core passes hold every problem within the plan's
capacity: a plan of n columns may be pointed at fewer, and the passes then
split the work otherwise (host arithmetic only, no GPU)."""
import ctypes

import pytest

import paper_2406_03468_gb300 as lsq


class TcSizes(ctypes.Structure):
    _fields_ = [(f, ctypes.c_size_t) for f in ("p1", "p2", "q", "y", "y64", "h", "r2")]


def _sizes(m, n, k, nsm):
    f = ctypes.CDLL(lsq.library_path())["_ZN3lsq14multi_tc_sizesEliii"]
    f.restype, f.argtypes = TcSizes, [ctypes.c_int64] + 3 * [ctypes.c_int]
    return f(m, n, k, nsm)


@pytest.mark.parametrize("nsm", [2, 3, 148, 151, 152])
@pytest.mark.parametrize("k", [8, 24, 64])
def test_sizes_cover_smaller_problems(nsm, k):
    m, nv = 5000, (k + 15) // 16 * 16
    for cap in (16, 64, 128, 129, 200, 256):
        z = _sizes(m, cap, k, nsm)
        for n in range(8, cap + 1, 3):
            tiles = (n + 127) // 128                       # row tiles of A^T
            ranges = nsm // tiles                          # CTAs per tile
            assert z.h >= ranges * tiles * nv * 128 * 16, (cap, n)
            small = _sizes(m - 700, n, k, nsm)
            for f in ("p1", "p2", "q", "y", "y64", "r2"):
                assert getattr(z, f) >= getattr(small, f), (f, cap, n)

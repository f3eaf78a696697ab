"""The QR's panel is launched with a cluster and a shared-memory size that the
device was asked for: on a part of a GPU a cluster of 16 CTAs may fit with the
panel's own bytes and not with whole SMs (host arithmetic with a stand-in for
the device's answer, no GPU)."""
import ctypes

import pytest

import paper_2406_03468_gb300 as lsq

FITS = ctypes.CFUNCTYPE(ctypes.c_bool, ctypes.c_int, ctypes.c_size_t)
WHOLE_SM = 227 * 1024


class QrPanel(ctypes.Structure):
    _fields_ = [("ctas", ctypes.c_int), ("alone", ctypes.c_int), ("bytes", ctypes.c_size_t)]


def _choice(d, n, fits):
    f = ctypes.CDLL(lsq.library_path())["_ZN3lsq15qr_panel_choiceEiiPFbimE"]
    f.restype, f.argtypes = QrPanel, [ctypes.c_int, ctypes.c_int, FITS]
    granted = set()

    def ask(ctas, nbytes):
        if fits(ctas, nbytes):
            granted.add((ctas, nbytes))
            return True
        return False

    return f(d, n, FITS(ask)), granted


@pytest.mark.parametrize("d,n", [(96, 8), (600, 50), (6000, 500), (9216, 768), (9228, 769)])
def test_launch_is_what_was_granted(d, n):
    whole, granted = _choice(d, n, lambda c, b: True)
    assert whole.ctas == 16 and (whole.ctas, whole.bytes) in granted
    assert whole.alone == (n <= 768) and (whole.bytes == WHOLE_SM) == bool(whole.alone)
    # a part with 16 CTAs of one cluster, but not 16 whole SMs
    part, granted = _choice(d, n, lambda c, b: b < WHOLE_SM)
    assert part.ctas == 16 and not part.alone and part.bytes < WHOLE_SM
    assert (part.ctas, part.bytes) in granted
    # a part with whole SMs for clusters of 8 only
    part, granted = _choice(d, n, lambda c, b: c == 8)
    assert part.ctas == 8 and part.alone == (n <= 768)
    if part.alone:
        assert (8, part.bytes) in granted
    # no cluster granted: the portable size, the panel's own bytes
    part, granted = _choice(d, n, lambda c, b: False)
    assert part.ctas == 8 and not part.alone


def test_answers_are_per_size():
    """A small panel's answer does not stand for a larger one's."""
    limit = 100 * 1024
    small, _ = _choice(600, 50, lambda c, b: c == 8 or b <= limit)
    large, _ = _choice(6000, 500, lambda c, b: c == 8 or b <= limit)
    assert small.ctas == 16 and large.ctas == 8

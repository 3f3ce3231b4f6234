"""The root tables e^{-2 pi i k / n} of the passes (host_roots in greens.cu), for
every line length a plan may choose and the half lengths of its rows: bitwise
symmetric about the axes and (but for the diagonals themselves, where cos and
sin of pi/4 differ by an ulp) the diagonals of the circle, and within an ulp
of the roots in long double.  Runs on the CPU."""
import ctypes

import numpy as np
import pytest

from paper_1106_0557_gb300 import native

LENGTHS = [16, 24, 32, 48, 64, 72, 96, 128, 144, 162, 192, 256, 288, 324, 384, 432, 512, 576, 648, 768, 1024, 1152,
           1296, 1536, 2048, 2304]


def _roots(n):
    f = native.lib()._ZN6isofft10host_rootsEllPdS0_
    f.argtypes, f.restype = [ctypes.c_long, ctypes.c_long, ctypes.c_void_p, ctypes.c_void_p], None
    re, im = np.empty(n), np.empty(n)
    f(n, n, re.ctypes.data, im.ctypes.data)
    return re, im


@pytest.mark.parametrize("n", LENGTHS)
def test_roots_are_symmetric_and_accurate(n):
    re, im = _roots(n)
    k = np.arange(n)
    assert np.array_equal(re[-k % n], re) and np.array_equal(im[-k % n], -im)  # about the real axis
    h = (n // 2 - k) % n
    assert np.array_equal(re[h], -re) and np.array_equal(im[h], im)            # about the imaginary one
    if n % 4 == 0:
        q = (n // 4 - k) % n
        off = 8 * k % n != 0                                                       # about the diagonals
        assert np.array_equal(re[q][off], -im[off]) and np.array_equal(im[q][off], -re[off])
    a = 2 * np.longdouble("3.14159265358979323846264338327950288") * k.astype(np.longdouble) / n
    # the angle's roundings (two products' worth) and the function's own
    assert np.abs(re - np.cos(a)).max() <= 2.3e-16 and np.abs(im + np.sin(a)).max() <= 2.3e-16

"""The trace passes' coefficients against a 60-digit conversion (host only)."""
from __future__ import annotations

import ctypes
from decimal import Decimal, getcontext

import numpy as np
import pytest

from oracle.leja import fast_leja_points


@pytest.mark.parametrize("lmin,lmax,m", [(1.0, 1.5, 7), (1.0, 1200.0, 60), (1.0, 8080.0, 80), (1.0, 1e6, 250), (1.0, 1e9, 250), (0.37, 2.9, 1),
                                          (1.0, 2.0, 0)])
def test_moment_coefficients_are_the_rounded_exact_ones(lmin, lmax, m):
    """Within 2^-52 of each coefficient and of 2^-80 of the largest (106-bit arithmetic over at most 250 stages
    whose errors Leja-ordered points keep at that scale)."""
    from paper_2603_02207_gb300 import _ffi
    import paper_2603_02207_gb300 as L
    try:
        lib = _ffi.load()
    except ImportError:
        pytest.skip("libleja.so is not built")
    d = np.ascontiguousarray(L.ll_divided_differences_q(lmin, lmax, m))
    c = np.zeros(m + 1)
    ptr = ctypes.POINTER(ctypes.c_double)
    assert lib.ll_moment_coefficients(m, d.ctypes.data_as(ptr), c.ctypes.data_as(ptr)) == 0
    getcontext().prec = 60
    xi = [Decimal(float(x)) for x in fast_leja_points(m + 1)]
    q = [Decimal(float(d[m]))]
    for j in range(m - 1, -1, -1):   # q <- (x - xi_j) q + d_j, by x D_0 = D_1, x D_1 = D_2 + 2 D_0, x D_k = D_{k+1} + D_{k-1}
        t = [Decimal(0)] * (len(q) + 1)
        for k, v in enumerate(q):
            t[k] -= xi[j] * v
            t[k + 1] += v
            if k:
                t[k - 1] += 2 * v if k == 1 else v
        t[0] += Decimal(float(d[j]))
        q = t
    top = max(abs(v) for v in q)
    for k in range(m + 1):
        assert abs(Decimal(float(c[k])) - q[k]) <= abs(q[k]) * Decimal(2) ** -52 + top * Decimal(2) ** -80, k


def test_moment_coefficients_reject_bad_arguments():
    from paper_2603_02207_gb300 import _ffi
    try:
        lib = _ffi.load()
    except ImportError:
        pytest.skip("libleja.so is not built")
    d = np.zeros(4)
    p = d.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
    assert lib.ll_moment_coefficients(-1, p, p) == 1
    assert lib.ll_moment_coefficients(3, None, p) == 1
    assert lib.ll_moment_coefficients(3, p, None) == 1

"""Gaussian probes against 50 digits (needs a GB300 and the library)."""
from __future__ import annotations

from decimal import Decimal, getcontext

import numpy as np
import pytest

from oracle import rng as R
from tests.gpu_util import lib, need_gpu

pytestmark = pytest.mark.gpu

PI = Decimal("3.14159265358979323846264338327950288419716939937510582097494459230781640628620899")


def _cos_turns(t: Decimal) -> Decimal:
    """cos(2 pi t) by folding to an eighth of a turn and the Taylor series."""
    t = t % 1
    t = min(t, 1 - t)
    sign = 1
    if t > Decimal("0.25"):
        t, sign = Decimal("0.5") - t, -1
    x = 2 * PI * (t if t <= Decimal("0.125") else Decimal("0.25") - t)
    odd = t > Decimal("0.125")   # sin of the complement
    term = x if odd else Decimal(1)
    total, k = term, 1 if odd else 0
    while abs(term) > Decimal(10) ** -48:
        term = -term * x * x / ((k + 1) * (k + 2))
        total += term
        k += 2
    return sign * total


def test_values_are_within_4e_16_of_50_digits():
    need_gpu()
    L = lib()
    getcontext().prec = 50
    n, cols, seed = 600, 5, 11
    got = L.ll_probes(L.Handle(), "gaussian", seed, 0, n, cols).cpu().numpy()
    x = R.raw_bits(seed, 0, n, cols)
    m1, m2 = (x >> np.uint64(11)) + np.uint64(1), R.mix(x) >> np.uint64(11)
    two53 = Decimal(2) ** 53
    worst = Decimal(0)
    for i in range(n):
        for j in range(cols):
            u1, u2 = Decimal(int(m1[i, j])) / two53, Decimal(int(m2[i, j])) / two53
            if u1 > 1 - Decimal(2) ** -10:   # (the plain FP64 formula)
                continue
            want = (-2 * u1.ln()).sqrt() * _cos_turns(u2)
            worst = max(worst, abs((Decimal(float(got[i, j])) - want) / want))
    assert worst <= Decimal("4e-16")

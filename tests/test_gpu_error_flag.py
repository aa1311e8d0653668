"""The pipeline error flag lives through a whole call (needs a GB300 and the library)."""
from __future__ import annotations

import pytest

from oracle import logdet as O
from synth import laplacian_2d, pentadiagonal
from tests.gpu_util import TOL, lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return lib()


@pytest.mark.parametrize("kernel", ["auto", "gather", "tma"])
@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("name", ["banded", "grid"])
def test_error_of_a_gram_reaches_the_caller_of_the_forward(L, name, prec, kernel):
    """The trace pass that follows the Grams does not clear what they reported, and the next call is clean."""
    A = pentadiagonal(3000, seed=3) if name == "banded" else laplacian_2d(55, 0.1)
    lo, hi = O.gershgorin(A)
    lo = max(lo, 0.1)
    dA = L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64")
    h = L.Handle()
    for what in ("none", "gram", "gram", "none"):
        h.debug_inject(what)
        o = L.options(degree=8, probes=15, seed=1, precision=prec, step_kernel=kernel, qr_gram="dfloat")
        if what == "gram":
            with pytest.raises(L.LejaError) as e:
                L.ll_logdet_forward(h, dA, lo, hi, o)
            assert e.value.name == "LL_ERR_TIMEOUT"
        else:
            want = O.logdet_leja(A, lo, hi, 8, 15, 1, f32=(prec == "f32"))["estimate"]
            assert abs(L.ll_logdet_forward(h, dA, lo, hi, o) - want) <= TOL[prec] * abs(want)


def test_error_of_a_gram_reaches_the_caller_of_the_sweep_and_the_gradient(L):
    A = laplacian_2d(40, 0.2)
    import numpy as np
    import torch
    dA = L.DeviceCSR.from_host(A)
    h = L.Handle()
    D = torch.full((A.n,), 1.0, dtype=torch.float64, device="cuda")
    h.debug_inject("gram")
    with pytest.raises(L.LejaError) as e:
        L.ll_logdet_sweep(h, dA, D, [0.5, 1.0], [(1.1, 5.1), (1.2, 9.2)], L.options(probes=15, seed=1, qr_gram="dfloat"), degrees=[8, 9])
    assert e.value.name == "LL_ERR_TIMEOUT"
    h.debug_inject("none")
    L.ll_logdet_forward(h, dA, 0.2, 8.2, L.options(degree=8, probes=15, seed=1, keep_for_backward=True))
    h.debug_inject("gram")
    with pytest.raises(L.LejaError) as e:
        L.ll_logdet_backward(h, dA, 1.0, through_qr=True)
    assert e.value.name == "LL_ERR_TIMEOUT"
    h.debug_inject("none")
    g = L.ll_logdet_backward(h, dA, 1.0, through_qr=True).cpu().numpy()
    assert np.all(np.isfinite(g))

"""The row products of the double-float CholeskyQR2 (needs a GB300 and the library): odd and even widths, one
column, a group of four and its remainders, the widest block (one tile in shared memory), ragged rows."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import logdet as O
from synth import diagonal, random_spd
from tests.gpu_util import lib, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return lib()


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 30, 33, 96])
@pytest.mark.parametrize("prec", ["df64", "f32"])
def test_estimate_and_gradient_match_the_oracle(L, prec, k):
    """Estimates to the rounding of the precision, and (DF64) the gradient, which sees every element of Q and G'."""
    A = random_spd(1000 + k, nnz_per_row=5, seed=k, empty_rows=2)
    lo, hi = O.gershgorin(A)
    lmin = max(lo, 0.05)
    dA = L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64")
    h = L.Handle()
    ref = O.logdet_leja(A, lmin, hi, 12, 3 * k, 3)
    est = L.ll_logdet_forward(h, dA, lmin, hi, L.options(degree=12, probes=3 * k, seed=3, precision=prec,
                                                          keep_for_backward=True))
    assert est == pytest.approx(ref["estimate"], rel=2e-5 if prec == "f32" else 1e-9)
    want = O.hutchpp_grad_values(A, lmin, hi, 12, ref["Q"], ref["Gp"])
    assert rel_err(L.ll_logdet_backward(h, dA, 1.0).cpu().numpy(), want) < (1e-4 if prec == "f32" else 1e-9)


@pytest.mark.parametrize("prec", ["f64", "df64"])
def test_ill_conditioned_sketch_keeps_the_deflation(L, prec):
    """A sketch of condition number 10^6 (the breakdown limit is 10^7): Q^T Q = I and Q^T G' = 0 to 2^-40, a few
    hundred roundings of 2^-48, and the estimate, whose trace over Q is all of it, to as much of every row."""
    n, k = 3000, 12
    logs = np.zeros(n)
    logs[::n // k] = 10.0 ** np.linspace(0, -4.5, k)
    h = L.Handle()
    est = L.ll_logdet_forward(h, L.DeviceCSR.from_host(diagonal(np.exp(logs))), 1.0, float(np.e),
                              L.options(degree=40, probes=3 * k, seed=4, precision=prec, probe_kind="gaussian", keep_for_backward=True))
    Q, G = (x.cpu().numpy() for x in L.ll_kept_basis(h))
    assert np.max(np.abs(Q.T @ Q - np.eye(k))) <= 2.0 ** -40
    assert np.max(np.abs(Q.T @ G)) <= 2.0 ** -40 * np.sqrt(n)
    assert abs(est - logs.sum()) <= 2.0 ** -40 * n

"""The trace pass in the moment form (needs a GB300 and the library): half the products with the matrix,
the same estimate. The stopping-rule passes run the Newton form, so a tolerance that no column
meets gives the Newton form's value of the same estimate."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import logdet as O
from synth import laplacian_2d, laplacian_3d, random_spd
from tests.gpu_util import TOL, lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return lib()


def _mat(name):
    A = {"lap2d_37": lambda: laplacian_2d(37, 0.1), "lap3d_17": lambda: laplacian_3d(17, 0.05),
         "random_900": lambda: random_spd(900, nnz_per_row=6, seed=4, empty_rows=3, dense_row=True)}[name]()
    lo, hi = O.gershgorin(A)
    return A, max(lo, 0.05), hi


@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("kernel", ["auto", "gather", "tma"])
@pytest.mark.parametrize("name", ["lap2d_37", "lap3d_17", "random_900"])
def test_moments_equal_newton_form(L, name, kernel, prec):
    """Degrees of both parities from the smallest, odd and even block widths. 1e-12: the rounding of
    the two forms, a few 2^-46 of sum |c_k| (below 10) times the columns' norms."""
    A, lo, hi = _mat(name)
    dA = L.DeviceCSR.from_host(A)
    h = L.Handle()
    for m in (1, 2, 3, 20, 41):
        for probes, est in ((15, "hutchpp"), (7, "hutchinson")):
            o = dict(degree=m, probes=probes, seed=2, precision=prec, step_kernel=kernel, estimator=est)
            got = L.ll_logdet_forward(h, dA, lo, hi, L.options(**o))
            i = h.info()
            want = L.ll_logdet_forward(h, dA, lo, hi, L.options(tol=1e-300, **o))
            j = h.info()
            scale = abs(want) + A.n
            assert abs(got - want) <= 1e-12 * scale, (m, est)
            assert abs(i["trace_q"] - j["trace_q"]) + abs(i["trace_res"] - j["trace_res"]) <= 2e-12 * scale


def test_moments_fp32_error_is_the_newton_forms(L):
    """FP32-mixed above the row threshold: against the FP64 estimate, the moment form is off by no
    more than twice the Newton form plus a part in 10^8, and within the FP32 bar."""
    A = laplacian_2d(257, 0.05)
    for seed in (1, 2):
        o = dict(degree=45, probes=30, seed=seed)
        ref = L.ll_logdet_forward(L.Handle(), L.DeviceCSR.from_host(A), 0.05, 8.05, L.options(precision="df64", **o))
        dA = L.DeviceCSR.from_host(A, "f32")
        mom = L.ll_logdet_forward(L.Handle(), dA, 0.05, 8.05, L.options(precision="f32", **o))
        newton = L.ll_logdet_forward(L.Handle(), dA, 0.05, 8.05, L.options(precision="f32", tol=1e-300, **o))
        assert abs(mom - ref) <= TOL["f32"] * abs(ref)
        assert abs(mom - ref) <= 2.0 * abs(newton - ref) + 1e-8 * abs(ref)


@pytest.mark.parametrize("kernel", ["auto", "gather", "tma"])
@pytest.mark.parametrize("n", [2000, 66000])
def test_clustered_spectra_keep_the_newton_forms_accuracy(L, n, kernel):
    """DF64 traces where most eigenvalues lie at the spectrum's low end: the moment form is at most twice as far
    from FP64 as the Newton form, which a kept forward runs (emulated: 0.6 times; the three-term recurrence ten
    times). Auto at n = 2000 is the cluster-resident pass."""
    from tests.test_gpu_moments_f32 import _outliers
    dA = L.DeviceCSR.from_host(_outliers(n))
    for m in (60, 61):
        def est(prec, keep):
            return L.ll_logdet_forward(L.Handle(), dA, 0.95, 1000.1, L.options(degree=m, probes=12, seed=3, precision=prec, step_kernel=kernel,
                                                                               estimator="hutchinson", keep_for_backward=keep))
        ref = est("f64", False)
        assert abs(est("df64", False) - ref) <= 2.0 * abs(est("df64", True) - ref), m

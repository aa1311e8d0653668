"""The cluster-resident pass (needs a GB300 and the library): small matrices run all steps of a pass
in one launch under the automatic choice, with the step kernels' per-row arithmetic."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import logdet as O
from synth import laplacian_2d, laplacian_3d, random_spd
from tests.gpu_util import TOL, lib, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return lib()


def _mat(name):
    if name == "random_517":   # uneven rows, operands from every CTA of a cluster, empty rows
        A = random_spd(517, nnz_per_row=4, seed=3, empty_rows=5)
    elif name == "lap2d_3":
        A = laplacian_2d(3, 0.5)
    elif name == "lap2d_100":
        A = laplacian_2d(100, 0.1)
    elif name == "lap3d_31":   # 29,791 rows: several rows per thread
        A = laplacian_3d(31, 0.05)
    else:
        A = laplacian_2d(int(name.split("_")[1]), 0.2)
    lo, hi = O.gershgorin(A)
    return A, max(lo, 0.05), hi


@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("name", ["lap2d_3", "random_517", "lap2d_23", "lap2d_100", "lap3d_31"])
@pytest.mark.parametrize("b", [1, 2, 5, 20])
def test_auto_pass_equals_gather_bitwise(L, name, prec, b):
    """p(A) V under the automatic choice (the cluster-resident pass on small matrices, where it is the
    faster one) and on the register-gather kernel: the same bits."""
    torch = need_gpu()
    A, lo, hi = _mat(name)
    dA = L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64")
    V = torch.as_tensor(np.random.default_rng(b).standard_normal((A.n, b))).cuda()
    h = L.Handle()
    got = [L.ll_apply_poly(h, dA, lo, hi, m, V, prec) for m in (1, 2, 17)]
    h.set_step_config("gather", 0, 0)
    for m, g in zip((1, 2, 17), got):
        assert torch.equal(g, L.ll_apply_poly(h, dA, lo, hi, m, V, prec)), m


@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("name,probes", [("lap2d_5", 9), ("random_517", 30), ("lap2d_100", 33), ("lap3d_31", 12)])
def test_auto_forward_matches_oracle_and_step_kernels(L, name, probes, prec):
    A, lo, hi = _mat(name)
    dA = L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64")
    h = L.Handle()
    o = dict(degree=21, probes=probes, seed=3, precision=prec)
    e = [L.ll_logdet_forward(h, dA, lo, hi, L.options(**o)) for _ in range(3)]   # eager, captured, replayed
    assert e[0] == e[1] == e[2]
    ref = L.ll_logdet_forward(h, dA, lo, hi, L.options(step_kernel="gather", **o))
    assert abs(e[0] - ref) <= (1e-12 if prec != "f32" else 1e-9) * abs(ref)
    want = O.logdet_leja(A, lo, hi, 21, probes, 3, f32=(prec == "f32"))["estimate"]
    assert abs(e[0] - want) <= TOL[prec] * abs(want)


@pytest.mark.parametrize("prec", ["f32", "df64"])
def test_cluster_trace_sums_keep_fp64_accuracy(L, prec):
    """One warp, one row a lane in both kernels, so that the same 25 terms are added: 8 2^-53 of the sum of their
    sizes, four times the usual error of two FP64 trees (a sum in double-float is off by up to 2^-48 of it)."""
    A = laplacian_2d(5, 0.3)
    dA = L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64")
    lo, hi = 0.3, 8.3
    c, g = (lo / 0.3 + hi / 0.3) / 2, (hi / 0.3 - lo / 0.3) / 4
    d, _ = L.ll_divided_differences(lo / 0.3, hi / 0.3, 1)
    M = O._scipy(A)
    worst = 0.0
    for seed in range(60):
        o = dict(degree=1, probes=1, seed=seed, precision=prec, estimator="hutchinson", keep_for_backward=True, probe_kind="gaussian")
        h, r = L.Handle(), L.Handle()
        h.debug_family("cluster")
        L.ll_logdet_forward(h, dA, lo, hi, L.options(**o))
        assert h.debug_families_run()[1] == "cluster"
        L.ll_logdet_forward(r, dA, lo, hi, L.options(step_kernel="gather", rows_per_thread=1, **o))
        v = L.ll_probes(h, "gaussian", seed, 1, A.n, 1).cpu().numpy()
        w = M @ v / (0.3 * g) - (c / g + 2.0) * v
        size = (abs(d[0]) * np.abs(v * v) + abs(d[1]) * np.abs(v * w)).sum()
        worst = max(worst, abs(h.info()["trace_res"] - r.info()["trace_res"]) / size)
    assert worst <= 8 * 2.0 ** -53

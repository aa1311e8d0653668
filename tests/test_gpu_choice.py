"""What the cached choice of a step kernel rests on (needs a GB300 and the library)."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import logdet as O
from synth import CSR, powerlaw_laplacian
from tests.gpu_util import lib, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return lib()


def _regular(n, nnz):
    """Rows of nearly equal length with columns next to the diagonal, with n rows and nnz entries."""
    length = np.full(n, nnz // n)
    length[: nnz - n * (nnz // n)] += 1
    rowptr = np.concatenate([[0], np.cumsum(length)]).astype(np.int32)
    row = np.repeat(np.arange(n), length)
    start = np.clip(np.arange(n) - length // 2, 0, n - length)
    col = start[row] + np.arange(nnz) - rowptr[row]
    return CSR(n, rowptr, col.astype(np.int32), np.where(col == row, 2.0, 0.01))


@pytest.mark.parametrize("first", ["irregular", "regular"])
def test_choice_is_not_taken_over_by_another_kind_of_matrix(L, first):
    """Two matrices of equal n and nnz on one handle, one of which the row kernel does not suit."""
    torch = need_gpu()
    P = powerlaw_laplacian(1 << 17, seed=1)
    R = _regular(P.n, P.nnz)
    assert R.nnz == P.nnz
    V = torch.as_tensor(np.random.default_rng(0).standard_normal((P.n, 40))).cuda()
    mats = {"irregular": (L.DeviceCSR.from_host(P, "f32"), 0.01, O.gershgorin(P)[1]), "regular": (L.DeviceCSR.from_host(R, "f32"), 1.0, 3.0)}
    g = L.Handle()
    g.set_step_config("gather", 0, 0)
    h = L.Handle()
    for name in (first, "regular" if first == "irregular" else "irregular"):
        dA, lo, hi = mats[name]
        got = L.ll_apply_poly(h, dA, lo, hi, 4, V, "f32")
        assert h.debug_families_run()[0] == ("rows" if name == "irregular" else "step")
        assert torch.equal(got, L.ll_apply_poly(g, dA, lo, hi, 4, V, "f32")), name


def test_stopping_rule_takes_a_timed_kernel_that_has_it(L):
    """On an irregular matrix the row kernel is the fixed-degree choice but has no stopping rule; the rule's passes take
    the TMA kernel (eight times as fast there as the register kernel's default shape)."""
    P = powerlaw_laplacian(1 << 17, seed=1)
    dA, hi = L.DeviceCSR.from_host(P, "f32"), O.gershgorin(P)[1]
    h, g = L.Handle(), L.Handle()
    o = dict(degree=10, probes=60, seed=1, precision="f32", reorder="none")
    L.ll_logdet_forward(h, dA, 0.01, hi, L.options(**o))
    assert h.debug_families_run()[0] == "rows"
    got = L.ll_logdet_forward(h, dA, 0.01, hi, L.options(tol=1e-30, **o))
    i = h.info()
    assert (i["kernel_pass1"], i["kernel_pass2"]) == (L.STEP_KERNELS["tma"],) * 2
    want = L.ll_logdet_forward(g, dA, 0.01, hi, L.options(tol=1e-30, step_kernel="gather", **o))
    assert abs(got - want) <= 1e-9 * abs(want)


def test_wide_stencil_gets_its_far_windows(L):
    """An 81-point stencil: rows of more than 64 entries, whose far entries lie on diagonal runs. With windows for
    the runs a stage holds tens of rows; with a gather for each of 72 far entries a row, four."""
    N = 200
    g = np.arange(N * N).reshape(N, N)
    row, col = [], []
    for dy in range(-4, 5):
        for dx in range(-4, 5):
            a = g[max(0, -dy): N - max(0, dy), max(0, -dx): N - max(0, dx)].ravel()
            row.append(a)
            col.append(a + dy * N + dx)
    row, col = np.concatenate(row), np.concatenate(col)
    o = np.lexsort((col, row))
    row, col = row[o], col[o]
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=N * N))]).astype(np.int32)
    dA = L.DeviceCSR.from_host(CSR(N * N, rowptr, col.astype(np.int32), np.where(row == col, 100.0, -1.0)), "f32")
    h, r = L.Handle(), L.Handle()
    o = dict(degree=10, probes=30, seed=1, precision="f32")
    got = L.ll_logdet_forward(h, dA, 15.0, 185.0, L.options(step_kernel="tma", **o))
    i = h.info()
    assert (i["kernel_pass1"], i["kernel_pass2"]) == (L.STEP_KERNELS["tma"],) * 2
    assert min(i["rows_pass1"], i["rows_pass2"]) >= 16
    want = L.ll_logdet_forward(r, dA, 15.0, 185.0, L.options(step_kernel="gather", **o))
    assert abs(got - want) <= 1e-9 * abs(want)

"""Kernels that the automatic choice takes by timing, each forced and seen to have run (needs a GB300 and the
library): the row-per-lane-group kernel in every mode it has, and the cluster-resident pass over its shapes."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import logdet as O
from synth import laplacian_2d, powerlaw_laplacian, random_spd
from tests.gpu_util import lib, need_gpu, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return lib()


def _mat(name):
    kind, n = name.split("_")
    A = {"lap2d": lambda: laplacian_2d(int(n), 0.1), "powerlaw": lambda: powerlaw_laplacian(int(n), seed=2),
         "spd": lambda: random_spd(int(n), nnz_per_row=5, seed=3, empty_rows=3),
         "dense": lambda: random_spd(int(n), nnz_per_row=7, seed=5, empty_rows=6, dense_row=True)}[kind]()
    lo, hi = O.gershgorin(A)
    return A, max(lo, 0.05), hi + (hi <= lo)   # (one row: an interval of some length)


def _poly(L, h, dA, lo, hi, m, V, prec, family, ran):
    h.debug_family(family)
    out = L.ll_apply_poly(h, dA, lo, hi, m, V, prec)
    assert h.debug_families_run()[0] == ran
    return out


@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("name", ["lap2d_1", "lap2d_6", "spd_517", "dense_2500", "powerlaw_3000"])
def test_rows_kernel_pass_equals_gather_bitwise(L, name, prec):
    torch = need_gpu()
    A, lo, hi = _mat(name)
    dA = L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64")
    h, g = L.Handle(), L.Handle()
    g.set_step_config("gather", 0, 0)
    for b in (1, 3, 8, 33, 36, 40, 66, 80):
        V = torch.as_tensor(np.random.default_rng(b).standard_normal((A.n, b))).cuda()
        got = _poly(L, h, dA, lo, hi, 4, V, prec, "rows", "rows")
        assert torch.equal(got, L.ll_apply_poly(g, dA, lo, hi, 4, V, prec)), b


@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("name,probes", [("spd_517", 30), ("powerlaw_3000", 99), ("powerlaw_70000", 12)])
def test_rows_kernel_traces_match_the_step_kernels(L, name, probes, prec):
    """The trace pass by moments and, kept for a backward, in the Newton form. 1e-12 as the step kernels' own
    agreement in the 64-bit modes, 1e-9 where the same FP32 W_j are reduced in another order."""
    A, lo, hi = _mat(name)
    dA = L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64")
    for keep in (False, True):
        est, run = {}, {}
        for fam in ("rows", "step"):
            h = L.Handle()
            h.debug_family(fam)
            o = L.options(degree=13, probes=probes, seed=3, precision=prec, keep_for_backward=keep, reorder="none")
            e = [L.ll_logdet_forward(h, dA, lo, hi, o) for _ in range(3)]   # eager, captured, replayed
            assert e[0] == e[1] == e[2]
            est[fam], run[fam] = e[0], h.debug_families_run()
        assert run["rows"][:2] == ("rows", "rows") and run["step"][:2] == ("step", "step")
        assert abs(est["rows"] - est["step"]) <= (1e-9 if prec == "f32" else 1e-12) * abs(est["step"]), keep


@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("ckpt", [0, 3])
def test_rows_kernel_gradient_matches_the_oracle(L, ckpt, prec):
    """Reverse steps (with the second block of the half-length recurrence in the 64-bit modes) and, with
    checkpoints, plain steps; widths of one and two 16-byte units a lane."""
    A, lo, hi = _mat("dense_700")
    dA = L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64")
    for probes in (12, 54):
        ref = O.logdet_leja(A, lo, hi, 9, probes, 4)
        want = O.hutchpp_grad_values(A, lo, hi, 9, ref["Q"], ref["Gp"])
        h = L.Handle()
        h.set_adjoint_fusion("off")
        h.debug_family("rows")
        L.ll_logdet_forward(h, dA, lo, hi, L.options(degree=9, probes=probes, seed=4, precision=prec, keep_for_backward=True,
                                                     ckpt_stride=ckpt))
        got = L.ll_logdet_backward(h, dA, 1.0).cpu().numpy()
        assert h.debug_families_run()[2] == "rows"
        assert rel_err(got, want) < (2e-4 if prec == "f32" else 1e-9)


@pytest.mark.parametrize("prec,name,b", [("f64", "lap2d_1", 1), ("df64", "lap2d_31", 5), ("f64", "spd_517", 20), ("f32", "spd_517", 8),
                                         ("df64", "lap2d_150", 2), ("f64", "lap2d_190", 3), ("f32", "lap2d_190", 6),
                                         ("f32", "lap2d_240", 4)])
def test_cluster_pass_equals_gather_bitwise(L, prec, name, b):
    """One to eight rows a thread, one to sixteen CTAs a cluster, one and two column pairs a thread."""
    torch = need_gpu()
    A, lo, hi = _mat(name)
    dA = L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64")
    V = torch.as_tensor(np.random.default_rng(b).standard_normal((A.n, b))).cuda()
    h, g = L.Handle(), L.Handle()
    g.set_step_config("gather", 0, 0)
    for m in (1, 2, 7):
        assert torch.equal(_poly(L, h, dA, lo, hi, m, V, prec, "cluster", "cluster"), L.ll_apply_poly(g, dA, lo, hi, m, V, prec)), m


@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
@pytest.mark.parametrize("name", ["spd_517", "lap2d_150"])
def test_cluster_traces_and_kept_blocks(L, name, prec):
    """Traces of the short and of the kept trace pass against the step kernels' (tolerances as above), and the
    gradient from the blocks that the cluster pass kept."""
    A, lo, hi = _mat(name)
    dA = L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64")
    for keep in (False, True):
        est, grad = {}, {}
        for fam in ("cluster", "step"):
            h = L.Handle()
            h.debug_family(fam)
            est[fam] = L.ll_logdet_forward(h, dA, lo, hi, L.options(degree=12, probes=12, seed=5, precision=prec, keep_for_backward=keep))
            assert h.debug_families_run()[:2] == (fam, fam)
            if keep:
                grad[fam] = L.ll_logdet_backward(h, dA, 1.0).cpu().numpy()
        assert abs(est["cluster"] - est["step"]) <= (1e-9 if prec == "f32" else 1e-12) * abs(est["step"]), keep
        if keep:
            assert rel_err(grad["cluster"], grad["step"]) < (1e-6 if prec == "f32" else 1e-11)


def test_family_values_are_checked(L):
    from paper_2603_02207_gb300 import _ffi
    h = L.Handle()
    for bad in (-1, 4):
        with pytest.raises(L.LejaError):
            h.check(_ffi.load().ll_debug_family(h.ptr, bad))
    assert h.debug_families_run() == ("auto", "auto", "auto")

"""The half-length reverse recurrence (needs a GB300 and the library): FP64 and DF64 gradients with U = W_0
at the shortest degrees, odd and even, with every W_j kept, strides of one and more, and a stride past the
half, against the oracle's full recurrence."""
from __future__ import annotations

import pytest

from oracle import logdet as O
from synth import laplacian_2d, random_spd
from tests.gpu_util import lib, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return lib()


@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("m", [1, 2, 3, 4, 7, 12])
def test_short_degrees_match_the_full_recurrence(L, m, prec):
    A = random_spd(260, nnz_per_row=5, seed=8, empty_rows=2)
    lo, hi = O.gershgorin(A)
    lmin = max(lo, 0.05)
    dA = L.DeviceCSR.from_host(A)
    ref = O.logdet_leja(A, lmin, hi, m, 12, 4)
    want = O.hutchpp_grad_values(A, lmin, hi, m, ref["Q"], ref["Gp"])
    h = L.Handle()
    for ckpt in (0, 1, 2, 5):
        L.ll_logdet_forward(h, dA, lmin, hi, L.options(degree=m, probes=12, seed=4, precision=prec,
                                                        keep_for_backward=True, ckpt_stride=ckpt))
        assert rel_err(L.ll_logdet_backward(h, dA, 1.0).cpu().numpy(), want) < 1e-9, ckpt


@pytest.mark.parametrize("m", [12, 13, 18])
def test_kept_strides_and_little_memory(L, m):
    """Checkpoints that the forward kept (strides 2, 3 and 4, W_h among them or not), then with device memory for the
    full recurrence's blocks only (two of Lambda, the segment) and 130 bytes an entry: the same gradient."""
    import torch
    A = laplacian_2d(900, 0.1)
    dA = L.DeviceCSR.from_host(A)
    lo, hi = 0.1, 8.1
    blk = A.n * 60 * 8

    def grad(budget, spare):
        h = L.Handle()
        if budget:
            h.set_keep_budget(budget * blk)
        L.ll_logdet_forward(h, dA, lo, hi, L.options(degree=m, probes=90, seed=1, keep_for_backward=True))
        stride = h.info()["kept_w_stride"]
        fill = None
        if spare:
            torch.cuda.synchronize()
            need = (2 + stride - 1) * blk + 130 * A.nnz
            fill = torch.empty(torch.cuda.mem_get_info()[0] - need - (64 << 20), dtype=torch.uint8, device="cuda")
        try:
            return stride, L.ll_logdet_backward(h, dA, 1.0).cpu().numpy()
        finally:
            del fill
            torch.cuda.empty_cache()

    one, want = grad(0, False)
    assert one == 1
    for stride in (2, 3, 4):
        blocks = (m + stride - 1) // stride - 1
        for spare in (False, True):
            got_stride, got = grad(blocks, spare)
            assert got_stride == stride
            assert rel_err(got, want) < 1e-12, (stride, spare)

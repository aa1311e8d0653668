"""One handle per host thread, calls at the same time (needs a GB300 and the library)."""
from __future__ import annotations

import threading

import numpy as np
import pytest

from oracle import logdet as O
from synth import laplacian_2d
from tests.gpu_util import lib, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family", ["cluster", "step"])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_launches_of_one_kernel_with_different_shared_memory(family, prec):
    """A small and a larger shape of the same kernels in two threads: neither's launch may fail because the other
    one lowered the kernel's shared-memory limit, and both give what they give alone."""
    torch = need_gpu()
    L = lib()
    # (named kernels: what a choice by timing takes may differ from handle to handle, and with it the order of sums)
    kernel = "tma" if family == "step" else "auto"
    work = []
    for N, b in ((11, 2), (23, 10)):
        A = laplacian_2d(N, 0.1)
        lo, hi = O.gershgorin(A)
        V = torch.as_tensor(np.random.default_rng(N).standard_normal((A.n, b))).cuda()
        work.append((L.DeviceCSR.from_host(A, "f32" if prec == "f32" else "f64"), max(lo, 0.05), hi, V))

    def calls(w, count, stream, out):
        try:
            h = L.Handle()
            h.debug_family(family)
            h.set_step_config(kernel, 0, 0)
            for _ in range(count):
                P = L.ll_apply_poly(h, w[0], w[1], w[2], 6, w[3], prec, stream=stream)
                e = L.ll_logdet_forward(h, w[0], w[1], w[2], L.options(degree=6, probes=12, seed=1, precision=prec, use_graph=False,
                                                                       step_kernel=kernel, qr_gram="dfloat"), stream=stream)
            stream.synchronize()
            out.append((P, e))
        except Exception as e:   # (seen by the main thread)
            out.append(e)

    alone, both = [[], []], [[], []]
    torch.cuda.synchronize()
    for x in range(2):
        calls(work[x], 1, torch.cuda.Stream(), alone[x])
    ts = [threading.Thread(target=calls, args=(work[x], 300, torch.cuda.Stream(), both[x])) for x in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for x in range(2):
        assert not isinstance(both[x][0], Exception), both[x][0]
        assert torch.equal(both[x][0][0], alone[x][0][0]) and both[x][0][1] == alone[x][0][1]

"""The double-float Gram of FP64 blocks has no bias (needs a GB300 and the library)."""
from __future__ import annotations

import math

import numpy as np
import pytest

from tests.gpu_util import lib, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [10, 33])
def test_fp64_gram_squares_are_unbiased(k):
    """The mean over 2 k random columns of the signed relative error of their squared norms. A column's is the
    double-float sums' rounding, up to 2^-48 and independent of the others', so that the mean is within 2^-50;
    products without the trailing parts' product are 2.6e-15 too small in every column."""
    torch = need_gpu()
    L = lib()
    err = []
    for seed in (100, 101):
        X = np.random.default_rng(seed).standard_normal((100_000, k))
        got = L.ll_gram(L.Handle(), torch.as_tensor(X).cuda(), None, method="dfloat").cpu().numpy()
        for j in range(k):
            # exact products of the halves (24 and 29 bits) but for the smallest, added without rounding
            h = X[:, j].astype(np.float32).astype(np.float64)
            lo = X[:, j] - h
            want = math.fsum(np.concatenate([h * h, 2.0 * h * lo, lo * lo]))
            err.append((got[j, j] - want) / want)
    assert abs(np.mean(err)) <= 2.0 ** -50

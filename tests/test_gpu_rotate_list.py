"""The sliced rotation's list of elements to sum in FP64 holds what ordinary rows
put on it up to the largest D: a list that overflows has the FP64 kernel compute the
whole block, right but 25 times slower."""
import time

import numpy as np
import pytest
import torch

import oracle
import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [2048, 3072, 4096])
def test_ordinary_rows_fit_the_list(erq, D):
    n = 8192
    X, _ = S.mixture(n, D, 64, 11, normalize=True)
    X -= X.mean(0, keepdims=True)
    P = S.random_orthogonal(D, 12)
    Xd, Pd = to_dev(X), to_dev(P)
    out = erq.rotate(Xd, Pd, accurate=True)
    sub = np.arange(0, n, 401)
    np.testing.assert_array_equal(out[to_dev(sub)].cpu().numpy().view(np.uint32), oracle.rotate(X[sub], P).view(np.uint32))
    s = []
    for _ in range(3):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        erq.rotate(Xd, Pd, accurate=True, out=out)
        torch.cuda.synchronize()
        s.append(time.perf_counter() - t0)
    # FP64 multiply-adds alone take 2 n D^2 / 0.75e12 seconds (0.75 TFLOP/s)
    assert min(s) < 0.25 * 2 * n * D * D / 0.75e12

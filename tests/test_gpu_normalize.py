"""Unit rows: fl32(x / ||x||) of the FP64 quotient for rows of ordinary, tiny,
huge and mixed magnitudes, zeros, powers of two and lengths off the batches."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 192, 256, 320, 1600])
def test_unit_rows(erq, D):
    g = S.rng(D)
    N = 600
    X = g.standard_normal((N, D)).astype(np.float32)
    X[100:150] *= np.float32(1e-30)
    X[150:200] *= np.float32(1e30)
    X[200:250] *= np.exp2(g.integers(-60, 60, (50, D))).astype(np.float32)
    X[250:300] *= g.random((50, D)) < 0.1
    X[300:310] = 0.0
    X[310:330] = np.float32(0.5)
    X[330:340] = np.exp2(g.integers(-3, 4, (10, D))).astype(np.float32)
    X[340:345] = 0.0
    X[340:345, 3] = np.float32(-7.25)
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 5)), 4, 3, assign=to_dev(np.arange(N, dtype=np.int32) % 3),
                         normalize=True)
    got = ix.export("raw").numpy()
    X64 = X.astype(np.float64)
    nrm = np.sqrt((X64 * X64).sum(1, keepdims=True))
    want = np.divide(X64, nrm, out=np.zeros_like(X64), where=nrm > 0).astype(np.float32)
    # the two FP64 norms differ by a few ulps of FP64: a rounding to FP32 differs once in 2^26 elements
    assert (got != want).sum() <= 1
    np.testing.assert_allclose(got, want, rtol=1.2e-7, atol=0)

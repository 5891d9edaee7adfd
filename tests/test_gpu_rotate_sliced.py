"""The sliced tensor-core rotation against the FP64 sum, bit for bit: digits at
their largest everywhere (the accumulators' exact range), several drains of the
accumulators, ragged row counts, rows over a wide range of magnitudes, exact
zeros (more listed elements than the list holds) and rows that are not finite."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(erq, X, P):
    got = erq.rotate(to_dev(X), to_dev(P), accurate=True).cpu().numpy()
    ref = oracle.rotate(X, P)
    np.testing.assert_array_equal(got.view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("n,D", [(1, 64), (129, 576), (300, 1088), (40, 4096)])
@pytest.mark.parametrize("kind", ["gauss", "largest", "wide", "tiny", "sparse"])
def test_rotate_sliced_bit_exact(erq, kind, n, D):
    g = S.rng(100 * D + n)
    X = g.standard_normal((n, D))
    P = S.random_orthogonal(D, 5) if kind in ("gauss", "wide", "tiny") else None
    if kind == "largest":           # every digit of every product at 64 and of one sign
        X = np.full((n, D), 0.5 - 2.0 ** -8)
        P = np.full((D, D), 0.5 - 2.0 ** -8, np.float32)
    elif kind == "wide":
        X = X * np.exp2(g.uniform(-40, 40, (n, D)))
    elif kind == "tiny":
        X = X * 2.0 ** -120
    elif kind == "sparse":
        X = X * (g.random((n, D)) > 0.9)
        P = np.eye(D, dtype=np.float32)
    _check(erq, np.ascontiguousarray(X.astype(np.float32)), P)


def test_rotate_sliced_zero_and_non_finite_rows(erq):
    D = 128
    P = S.random_orthogonal(D, 6)
    X = S.mixture(200, D, 4, 7)[0]
    X[3] = 0.0
    _check(erq, X, P)
    X[9, 1] = np.inf
    got = erq.rotate(to_dev(X), to_dev(P), accurate=True).cpu().numpy()
    ok = np.arange(200) != 9
    np.testing.assert_array_equal(got[ok].view(np.uint32), oracle.rotate(X[ok], P).view(np.uint32))
    assert not np.isfinite(got[9]).any()

"""The encoder's bounded walk (range search, jumps, windows, oversized runs of
one key) against the FP64 oracle, bit for bit, on rows built to reach each
branch: one FP32 key shared by more events than a window holds, keys that
collide in FP32 but not exactly, heavy tails, magnitudes over 20 binades, and
one coordinate far above the rest."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


def _rows(kind, n, D, seed):
    g = S.rng(seed)
    sign = np.where(g.random((n, D)) < 0.5, -1.0, 1.0)
    if kind == "equal":                       # D events at every critical value
        x = np.full((n, D), 1.5) * sign
    elif kind == "near_equal":                # equal FP32 keys, different exact order
        x = (1.0 + g.integers(0, 4, (n, D)) * 2.0 ** -23) * sign
    elif kind == "ties":
        x = g.integers(-4, 5, (n, D)).astype(np.float64)
    elif kind == "cauchy":
        x = g.standard_cauchy((n, D))
    elif kind == "wide":
        x = np.exp2(g.uniform(-20, 0, (n, D))) * sign
    elif kind == "peak":
        x = g.standard_normal((n, D))
        x[:, 0] = 3000.0
    else:
        x = g.standard_normal((n, D))
    return np.ascontiguousarray(x.astype(np.float32))


@pytest.mark.parametrize("kind", ["gauss", "equal", "near_equal", "ties", "cauchy", "wide", "peak"])
@pytest.mark.parametrize("D,B,n", [(64, 10, 6), (576, 2, 24), (960, 5, 24), (1024, 8, 10), (1536, 3, 12),
                                   (4096, 9, 2)])
def test_encode_ranges_bit_exact(erq, kind, D, B, n):
    R = _rows(kind, n, D, 7000 + 10 * D + B)
    codes_o, st_o = oracle.quantize(R, B)
    fa_o, fr_o = oracle.stored_factors(st_o)
    codes, fa, fr, st = erq.encode(to_dev(R), B, with_stats=True)
    codes = codes.cpu().numpy().view(np.uint16 if B > 8 else np.uint8)
    np.testing.assert_array_equal(codes, codes_o.astype(codes.dtype))
    np.testing.assert_array_equal(st.cpu().numpy()[:, :2], np.asarray(st_o)[:, :2])
    np.testing.assert_array_equal(fa.cpu().numpy().view(np.uint32), fa_o.view(np.uint32))
    np.testing.assert_array_equal(fr.cpu().numpy().view(np.uint32), fr_o.view(np.uint32))


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_encode_refuses_non_finite_rows(erq, value):
    R = _rows("gauss", 3, 128, 7)
    R[1, 5] = value
    with pytest.raises(erq.ErqError):
        erq.encode(to_dev(R), 4)

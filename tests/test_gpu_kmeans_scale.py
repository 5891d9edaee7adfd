"""Lists of rows scaled by a power of two: every product, sum and distance scales
exactly, so the lists are the same.  Rows whose nearest centroids are close calls
(|x||c| far above the distances), at sizes whose squares' product leaves FP32's
range, with the product of norms on the tensor cores."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,D,nl", [(4000, 4096, 140), (40000, 256, 260)])
def test_lists_do_not_depend_on_the_scale(erq, N, D, nl):
    X = to_dev(S.mixture(N, D, 24, 93)[0] + np.float32(30.0))
    P = to_dev(S.random_orthogonal(D, 94))

    def lists(e):
        ix = erq.build_index(X * 2.0 ** e, P, 4, nl, kmeans_iters=1)
        out = ix.export("list_offsets"), ix.export("list_ids")
        ix.free()
        return out

    want = lists(0)
    for e in (-49, -30, 20, 45):
        for w, g in zip(want, lists(e)):
            assert torch.equal(w, g), e

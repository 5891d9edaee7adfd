"""Estimates of explicit ids on both sides of the sizes from which a block stages
its rows: a pair's estimate is the same sum in the same order either way, so one
large call and its parts agree bit for bit."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,B,nq,nc", [(64, 4, 2048, 32), (192, 9, 700, 131), (576, 3, 8200, 33), (1024, 8, 2049, 128),
                                       (1088, 5, 300, 40)])
@pytest.mark.parametrize("metric", ["l2", "ip"])
def test_a_large_call_equals_its_parts(erq, D, B, nq, nc, metric):
    N, nl = 900, 5
    X, lab = S.mixture(N, D, nl, 31, scale="aniso")
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 32)), B, nl, assign=to_dev(lab))
    Q = torch.randn(nq, D, device="cuda", generator=torch.Generator("cuda").manual_seed(33))
    ids = torch.randint(-1, N, (nq, nc), device="cuda", generator=torch.Generator("cuda").manual_seed(34))
    whole = ix.estimate(Q, ids, metric=metric)
    assert torch.equal(torch.isnan(whole), ids < 0)
    for a, b in ((0, 1), (nq // 2, nq // 2 + 7), (nq - 5, nq)):
        for j in (0, nc - 31):
            part = ix.estimate(Q[a:b].contiguous(), ids[a:b, j:j + 31].contiguous(), metric=metric)
            assert torch.equal(part.nan_to_num(7.0), whole[a:b, j:j + 31].nan_to_num(7.0))

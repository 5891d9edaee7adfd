"""The two-stage search's second stage where many rows of a list survive and where
few do, over coordinate counts that fill its lanes and that do not.  A row's estimate
is the same sum in the same order either way, so a search that prunes nothing and
one that prunes give a common candidate the same bits, and the first's candidates
are the best of all rows."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,B", [(64, 2), (128, 9), (640, 5), (1088, 2), (1536, 3), (2112, 8), (4096, 6), (192, 1)])
@pytest.mark.parametrize("nq,nprobe", [(3, 8), (300, 2)])
def test_estimates_do_not_depend_on_the_survivors(erq, D, B, nq, nprobe):
    N, nl, k = 2000, 8, 1000
    X, lab = S.mixture(N, D, nl, 61, scale="aniso")
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 62)), B, nl, assign=to_dev(lab))
    Q = to_dev(S.mixture(nq, D, nl, 63, comp_seed=61, scale="aniso")[0])
    kw = dict(rerank_k=k, nprobe=nprobe, return_candidates=True, return_stats=True)
    _, _, all_i, all_e, (rows, left) = ix.search_two_stage(Q, 10, eps0=1e4, **kw)
    assert left == rows                               # (bounds of 1e4 times the expected error prune nothing)
    got = torch.full((nq, N + 1), float("nan"), device="cuda")
    got.scatter_(1, torch.where(all_i >= 0, all_i, N), all_e)      # (absent candidates to the column past the rows)
    for k2, eps0 in ((20, 0.0), (20, 1.9), (5, 0.2)):
        _, _, cid, est, (_, fewer) = ix.search_two_stage(Q, 5, eps0=eps0, **dict(kw, rerank_k=k2))
        assert (cid >= 0).all() and fewer < rows
        assert torch.equal(est, got.gather(1, cid))
        if eps0 == 1.9:
            assert (cid[:, 0] == all_i[:, 0]).all()   # the best of all rows is kept

"""The block merge (k' > 32): per query the k smallest of many candidates, with
fills that reach and pass the sort buffer."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,k", [(1, 1), (31, 10), (33, 32), (8192, 20), (33, 33), (412, 100), (413, 100), (2000, 128),
                                 (8192, 1024)])
def test_merge_topk(erq, m, k):
    nq = 257
    g = S.rng(m + k)
    vals = g.standard_normal((nq, m)).astype(np.float32)
    ids = np.argsort(g.random((nq, m)), axis=1).astype(np.int64)
    got_i, got_v = erq.merge_topk(to_dev(ids), to_dev(vals), k)
    order = np.lexsort((ids, vals), axis=1)[:, :k]
    np.testing.assert_array_equal(got_i.cpu().numpy(), np.take_along_axis(ids, order, 1))
    np.testing.assert_array_equal(got_v.cpu().numpy(), np.take_along_axis(vals, order, 1))


@pytest.mark.parametrize("rerank_k,nq", [(20, 300), (20, 2500), (32, 1), (128, 300)])
def test_search_many_lists_per_query(erq, rerank_k, nq):
    """64 lists of every query: the full probe and re-rank give exact neighbours."""
    N, D, nl = 6000, 64, 64
    X, _ = S.mixture(N, D, 8, 51)
    P = S.random_orthogonal(D, 52)
    Q = S.mixture(nq, D, 8, 53, comp_seed=51)[0]
    ix = erq.build_index(to_dev(X), to_dev(P), 8, nl, assign=to_dev(S.random_assign(N, nl, 54)))
    sub = np.arange(min(nq, 300)) * (nq // min(nq, 300))
    ref = ((Q[sub, None, :].astype(np.float64) - X[None]) ** 2).sum(2)
    top = np.sort(ref, axis=1)[:, :10]
    for precision in ("fp32", "fp16"):
        _, d = ix.search(to_dev(Q), 10, rerank_k=rerank_k, nprobe=nl, precision=precision)
        np.testing.assert_allclose(d.cpu().numpy()[sub], top, rtol=1e-5)

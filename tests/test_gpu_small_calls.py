"""Calls of few (query, list) pairs: one planning kernel, no read-back of sizes,
narrow GEMM tiles.  The same queries in one large call take the general plan; a
query's estimates do not depend on its batch."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,nl,nprobe,step", [(64, 33, 33, 62), (192, 40, 7, 1), (320, 300, 64, 32), (64, 2, 2, 700)])
@pytest.mark.parametrize("precision", ["fp16", "fp32", "fp8"])
def test_small_calls_equal_the_large_one(erq, D, nl, nprobe, step, precision):
    N, nq = 5000, 2100
    X, _ = S.mixture(N, D, 8, 61)
    Q = to_dev(S.mixture(nq, D, 8, 62, comp_seed=61)[0])
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 63)), 5, nl,
                         assign=to_dev(S.random_assign(N, nl, 64)))
    npq = torch.randint(1, nprobe + 1, (nq,), dtype=torch.int32, device=Q.device)
    kw = dict(rerank_k=20, nprobe=nprobe, precision=precision)
    want = ix.search(Q, 10, nprobe_per_query=npq, return_candidates=True, **kw)
    for a in range(0, min(nq, 4 * step), step):
        got = ix.search(Q[a:a + step], 10, nprobe_per_query=npq[a:a + step], return_candidates=True, **kw)
        for g, w in zip(got, want):
            w = w[a:a + step]
            if g.dtype == torch.int64:
                assert torch.equal(g, w)
            else:
                np.testing.assert_allclose(g.cpu().numpy(), w.cpu().numpy(), rtol=2e-6)
        st = ix.stats()
        assert 0 < st["items"] <= st["lists"] <= st["pairs"] and 0 < st["rows"] <= N


@pytest.mark.parametrize("nq", [1, 40])
def test_small_call_reports_a_bad_probe_count(erq, nq):
    X, _ = S.mixture(500, 64, 4, 71)
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(64, 72)), 4, 8, assign=to_dev(S.random_assign(500, 8, 73)))
    Q = to_dev(X[:nq])
    bad = torch.full((nq,), 9, dtype=torch.int32, device=Q.device)
    for precision in ("fp16", "fp32"):
        with pytest.raises(Exception, match="(?i)bound|range|nprobe"):
            ix.search(Q, 5, nprobe=8, nprobe_per_query=bad, precision=precision)
        ix.search(Q, 5, nprobe=8, precision=precision)

"""FP32 precision ranks estimates that are not numbers, or infinite, last and by
id, on the tensor-core scan as on the CUDA-core one (k' above 128): a query with a
NaN in it, or one whose distances overflow, gets the lowest ids of its lists, and
the queries beside it what they get without it."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [5, 32, 33, 128, 160])
@pytest.mark.parametrize("nlist,nq", [(1, 1), (1, 70), (6, 3), (6, 600)])
@pytest.mark.parametrize("metric", ["l2", "ip"])
def test_nan_and_overflowing_queries(erq, k, nlist, nq, metric):
    N, D = 1300, 64
    X, _ = S.mixture(N, D, 6, 51)
    lab = np.arange(N, dtype=np.int32) % nlist
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 52)), 5, nlist, assign=to_dev(lab))
    Q = S.mixture(nq, D, 6, 53, comp_seed=51)[0]
    probe = to_dev(np.tile(np.arange(nlist, dtype=np.int32), (nq, 1)))[:, :max(1, nlist - 1)].contiguous()
    kw = dict(nprobe=probe.shape[1], precision="fp32", metric=metric)
    if nlist > 1:
        kw["probe"] = probe
    want_i, want_d = ix.search(to_dev(Q), k, **kw)
    bad = np.arange(0, nq, 3)
    lowest = torch.arange(N)[torch.from_numpy(lab) < probe.shape[1]][:k]
    for value in (np.nan, 1e30) if metric == "l2" else (np.nan,):
        B = Q.copy()
        B[bad] = np.float32(1.0)
        B[bad, 7 % D] = value
        ids, d = ix.search(to_dev(B), k, **kw)
        ids, d = ids.cpu(), d.cpu()
        assert torch.equal(ids[bad], lowest[None].expand(len(bad), -1))
        assert (torch.isnan(d[bad]) if np.isnan(value) else torch.isinf(d[bad])).all()
        ok = np.setdiff1d(np.arange(nq), bad)
        assert torch.equal(ids[ok], want_i.cpu()[ok]) and torch.equal(d[ok], want_d.cpu()[ok])

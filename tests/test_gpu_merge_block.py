"""The block merge over more keys than its sort buffer: both block sizes, keys
that spread over the counting intervals and keys that do not."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [3, 304, 305])
@pytest.mark.parametrize("kp", [33, 100, 128])
@pytest.mark.parametrize("kind", ["mixture", "few values"])
def test_many_keys_per_query(erq, nq, kp, kind):
    """96 lists of every query, all probed: the full re-rank of the merged candidates gives exact neighbours."""
    N, D, nl = 9600, 64, 96
    X, _ = S.mixture(N, D, 8, 81)
    if kind == "few values":
        X = X[np.arange(N) % 40]                # 240 copies of each row: a count of equal keys beyond any interval
    Q = S.mixture(nq, D, 8, 82, comp_seed=81)[0]
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 83)), 8, nl, assign=to_dev(S.random_assign(N, nl, 84)))
    ref = np.sort(((Q[:, None, :].astype(np.float64) - X[None]) ** 2).sum(2), axis=1)[:, :10]
    for precision in ("fp32", "fp16"):
        _, d = ix.search(to_dev(Q), 10, rerank_k=kp, nprobe=nl, precision=precision)
        np.testing.assert_allclose(d.cpu().numpy(), ref, rtol=1e-5)

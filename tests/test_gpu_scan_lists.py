"""The tensor-core scan's candidate lists where they fill: rows at one distance
(every candidate of a block ties, ordered by id), lists that outgrow their
shared part, items of one row block and of many, and the three precisions'
final results on the same index."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp16", "fp32", "fp8"])
@pytest.mark.parametrize("rr", [0, 256, 8192])
@pytest.mark.parametrize("kp,nq", [(20, 1), (32, 130), (20, 1000), (128, 40)])
def test_equal_rows_keep_the_lowest_ids(erq, precision, rr, kp, nq):
    """Copies of one row in two lists: every estimate of a list is the same
    number, so the k' candidates are the lowest ids of the nearer list."""
    D, N = 64, 3000
    g = S.rng(11)
    a, b = g.standard_normal((2, D)).astype(np.float32)
    lab = (np.arange(N) % 3 == 0).astype(np.int32)
    X = np.where(lab[:, None] == 1, a[None], b[None]).astype(np.float32)
    X[:2] += 0.25 * g.standard_normal((2, D)).astype(np.float32)       # (non-zero residuals)
    Q = (a[None] + 0.01 * g.standard_normal((nq, D))).astype(np.float32)
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 12)), 4, 2, assign=to_dev(lab))
    ix.set_scan_config(0, rr)
    _, _, ids, _ = ix.search(to_dev(Q), kp, nprobe=2, precision=precision, return_candidates=True)
    near = np.nonzero(lab == 1)[0]
    got = ids.cpu().numpy()
    ref = near[near >= 2][:kp] if kp < len(near) else near
    # the two perturbed rows have estimates of their own; all others tie
    for row in got:
        rest = [i for i in row if i >= 2]
        assert rest == sorted(rest) and set(rest) <= set(near.tolist())
        assert rest == ref[:len(rest)].tolist()


@pytest.mark.parametrize("B", [1, 3, 5, 9])
def test_precisions_agree_after_the_rerank(erq, B):
    N, D, nl = 9000, 192, 24
    X, lab = S.mixture(N, D, 6, 21, scale="aniso")
    Q = to_dev(S.mixture(700, D, 6, 22, comp_seed=21, scale="aniso")[0])
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 23)), B, nl, assign=to_dev(S.random_assign(N, nl, 24)))
    ref = None
    for qn, rr in ((0, 0), (32, 256), (64, 2048)):
        ix.set_scan_config(qn, rr)
        ids, d, cid, est = ix.search(Q, 10, rerank_k=32, nprobe=nl, precision="fp32", return_candidates=True)
        if ref is None:
            ref = (ids, d, cid, est)
        else:                                          # the item shape changes nothing
            for x, y in zip(ref, (ids, d, cid, est)):
                assert torch.equal(x, y)
    e = ix.estimate(Q, ref[2])
    assert ((ref[3] - e).abs() <= 2e-5 * e.abs()).all()

"""Candidates, all ranks of them: full lists of distinct ids in (estimate, id) order
with nothing better left out, where rows tie by the hundred, where a query's lists
hold more keys than the merge sorts at once (by counting, and chunk by chunk where
the counting interval of the k'-th ties as well), and in all three precisions."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(ix, Q, cid, est, group, k):
    """cid, est [nq, k]: every row of one group has one estimate; the candidates are
    the k smallest (estimate, id) pairs of all rows."""
    cid, est = cid.cpu().numpy(), est.cpu().numpy().astype(np.float64)
    assert (cid >= 0).all() and all(len(set(c)) == k for c in cid)
    d = np.diff(est, axis=1)
    assert (d >= 0).all() and (np.diff(cid, axis=1)[d == 0] > 0).all()
    ng = group.max() + 1
    rep = np.array([np.flatnonzero(group == g)[0] for g in range(ng)])
    e = ix.estimate(Q, to_dev(np.tile(rep, (len(cid), 1)))).cpu().numpy().astype(np.float64)    # each group's own value
    members = [np.sort(np.flatnonzero(group == g)) for g in range(ng)]
    for c, x, eg in zip(cid, est, e):
        mine = group[c]
        for g in range(ng):
            at = mine == g
            n = int(at.sum())
            if n == 0:                       # (FP32's and the estimate's sums agree to 2e-5)
                assert eg[g] >= x[-1] * (1 - 2e-5)
                continue
            assert len(set(x[at])) == 1 and abs(x[at][0] - eg[g]) <= 2e-5 * abs(eg[g])
            assert (np.sort(c[at]) == members[g][:n]).all()                   # the lowest ids of the group
            assert n == len(members[g]) or x[at][0] == x[-1]                  # all of them unless cut by the last rank


@pytest.mark.parametrize("distinct", [8, 40, 960])
@pytest.mark.parametrize("nq,k", [(3, 33), (3, 128), (305, 100), (305, 128)])
def test_merge_of_many_lists_with_equal_keys(erq, distinct, nq, k):
    """96 lists that hold the same rows: one centroid, so copies of a row tie in all of them."""
    nl, per, D = 96, 960 // 8, 64
    base = S.mixture(distinct, D, 4, 91)[0]
    if distinct == 960:                       # no ties: every list its own rows
        X = S.mixture(nl * per, D, 4, 91)[0]
        row = np.arange(nl * per)
    else:
        row = np.tile(np.arange(per) % distinct, nl)
        X = base[row]
    lab = np.repeat(np.arange(nl), per).astype(np.int32)
    p = S.rng(92).permutation(nl * per)
    X, lab, row = X[p], lab[p], row[p]
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 93)), 8, nl, assign=to_dev(lab))
    c = ix.export("centroids").numpy()
    if distinct != 960:
        assert (c == c[0]).all()
    Q = to_dev(S.mixture(nq, D, 4, 94, comp_seed=91)[0])
    _, _, cid, est = ix.search(Q, 10, rerank_k=k, nprobe=nl, precision="fp32", return_candidates=True)
    if distinct != 960:
        _check(ix, Q, cid, est, row, k)
        return
    e = ix.estimate(Q, torch.arange(nl * per, device="cuda")[None].expand(nq, -1).contiguous()).double()
    best = e.topk(k, largest=False).values
    assert (cid >= 0).all() and (cid.sort(1).values.diff(dim=1) > 0).all()
    assert ((est.double() - best).abs() <= 2e-5 * best.abs()).all()
    assert ((est.double() - e.gather(1, cid)).abs() <= 2e-5 * best.abs()).all()


@pytest.mark.parametrize("precision", ["fp16", "fp32", "fp8"])
@pytest.mark.parametrize("rr", [0, 256, 8192])
@pytest.mark.parametrize("kp,nq", [(20, 1), (32, 130), (20, 1000), (128, 40)])
def test_ties_fill_the_lists(erq, precision, rr, kp, nq):
    """Copies of one row in the nearer of two lists: the candidates are its kp lowest ids, none missing."""
    D, N = 64, 3000
    a, b = S.rng(11).standard_normal((2, D)).astype(np.float32)
    lab = (np.arange(N) % 3 == 0).astype(np.int32)
    X = np.where(lab[:, None] == 1, a[None], b[None]).astype(np.float32)
    last = np.array([N - 1, np.flatnonzero(lab == 1)[-1]])             # a row of each list away from the rest,
    X[last] += np.float32(8.0)                                         # so that residuals are not zero
    Q = (a[None] + 0.01 * S.rng(12).standard_normal((nq, D))).astype(np.float32)
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 13)), 4, 2, assign=to_dev(lab))
    ix.set_scan_config(0, rr)
    _, _, cid, est = ix.search(to_dev(Q), kp, nprobe=2, precision=precision, return_candidates=True)
    near = np.setdiff1d(np.flatnonzero(lab == 1), last)
    assert (cid.cpu().numpy() == near[None, :kp]).all()
    assert (est == est[:, :1]).all()


@pytest.mark.parametrize("B", [4, 6, 8])
@pytest.mark.parametrize("kp", [32, 128])
def test_three_precisions_find_the_neighbours(erq, B, kp):
    N, D, nl, nq = 3000, 192, 24, 300
    X, _ = S.mixture(N, D, 6, 21, scale="aniso")
    Q = S.mixture(nq, D, 6, 22, comp_seed=21, scale="aniso")[0]
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 23)), B, nl, assign=to_dev(S.random_assign(N, nl, 24)))
    ref = np.sort(((Q[:, None].astype(np.float64) - X[None]) ** 2).sum(2), axis=1)[:, :3]
    for precision in ("fp32", "fp16", "fp8"):
        _, d = ix.search(to_dev(Q), 3, rerank_k=kp, nprobe=nl, precision=precision)
        np.testing.assert_allclose(d.cpu().numpy(), ref, rtol=1e-5)

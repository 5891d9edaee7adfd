"""Cluster means and nearest centroids: the means equal the FP64 sums in stored
order, divided and rounded once, for sums that cancel, tiny, huge, zero and
single-row lists; the rows' lists are their nearest centroids, the lowest of
equal ones, on both sides of the size from which the product runs on the
tensor cores."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,D,nl", [(4000, 64, 7), (4000, 192, 300), (30000, 128, 2), (37, 64, 37)])
def test_means_are_the_ordered_sums(erq, N, D, nl):
    g = S.rng(N + D)
    X = (g.standard_normal((N, D)) * np.exp2(g.integers(-12, 12, (N, 1)))).astype(np.float32)
    X[:, 1] = np.where(np.arange(N) % 2 == 0, 1.0, -1.0) * np.abs(X[:, 1])       # cancels
    X[:, 2] = 0.0
    X[:, 3] *= np.float32(1e-30)
    X[:, 4] = np.float32(1.0) + np.float32(2.0 ** -23) * g.integers(0, 2, N).astype(np.float32)
    assign = S.random_assign(N, nl, 5)
    assign[assign == 1] = 0                                                      # an empty list
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 6)), 4, nl, assign=to_dev(assign))
    got = ix.export("centroids").numpy()
    for j in range(nl):
        rows = X[assign == j].astype(np.float64)
        want = (np.cumsum(rows, axis=0)[-1] / len(rows)).astype(np.float32) if len(rows) else np.zeros(D, np.float32)
        np.testing.assert_array_equal(got[j], want)


def _norms(X):
    """Row norms as a warp sums them: lane l takes coordinates 4 l .. 4 l + 3 of every 128."""
    N, D = X.shape
    acc = torch.zeros(N, 32, dtype=torch.float32, device=X.device)
    for k0 in range(0, D, 128):
        blk = torch.zeros(N, 128, dtype=torch.float64, device=X.device)
        blk[:, :min(128, D - k0)] = X[:, k0:k0 + 128].double()
        blk = blk.view(N, 32, 4)
        for i in range(4):
            acc = (acc.double() + blk[:, :, i] ** 2).float()
    lane = torch.arange(32, device=X.device)
    for o in (16, 8, 4, 2, 1):
        acc = acc + acc[:, lane ^ o]
    return acc[:, 0]


def _assign(X, C):
    """Argmin of the FP32 distances whose product is a chain of D fused multiply-adds."""
    acc = torch.zeros(X.shape[0], C.shape[0], dtype=torch.float32, device=X.device)
    for k in range(X.shape[1]):
        acc = (acc.double() + X[:, k].double()[:, None] * C[:, k].double()[None]).float()
    d = (_norms(X)[:, None] + _norms(C)[None]) - 2.0 * acc
    best = d.min(1, keepdim=True).values
    return (d == best).int().argmax(1).cpu().numpy()


@pytest.mark.parametrize("N,D,nl", [(3000, 64, 16), (40000, 256, 260), (21000, 448, 257)])
@pytest.mark.parametrize("kind", ["mixture", "offset", "copies"])
def test_lists_are_those_of_the_fp32_distances(erq, N, D, nl, kind):
    X, _ = S.mixture(N, D, 24, 91)
    if kind == "offset":
        X = X + np.float32(30.0)               # |x||c| far above the distances: every row is a close call
    if kind == "copies":
        X[N // 2:] = X[:N - N // 2]            # equal rows and equal initial centroids
        X[::5] = X[0]
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 92)), 4, nl, kmeans_iters=1)
    off, ids = ix.export("list_offsets").numpy(), ix.export("list_ids").numpy()
    lab = np.empty(N, np.int64)
    for j in range(nl):
        lab[ids[off[j]:off[j + 1]]] = j
    Xd = to_dev(X)
    C = X[(np.arange(nl) * float(N) / nl).astype(np.int64)].copy()
    first = _assign(Xd, to_dev(C))
    for j in range(nl):
        rows = X[first == j].astype(np.float64)
        if len(rows):
            C[j] = (np.cumsum(rows, axis=0)[-1] / len(rows)).astype(np.float32)
    want = _assign(Xd, to_dev(C))
    # (the emulated chain rounds twice: one step in 2^29 is off by a unit, so a tie may fall to the other side)
    assert (lab != want).sum() <= 2

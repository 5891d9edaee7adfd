"""Estimates and gradients of explicit ids at the sizes where their kernels'
blocks end: more ids than a staging pass, one id, a coordinate count below and
above one block's, 16-bit codes, ids that are absent, and queries that do not
start on a 16-byte boundary (gradient only: the estimate's rotation needs one)."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,B,nc", [(64, 4, 1), (192, 9, 33), (1024, 3, 128), (1088, 8, 129), (4096, 1, 40)])
@pytest.mark.parametrize("metric", ["l2", "ip"])
def test_estimate_and_backward_shapes(erq, D, B, nc, metric):
    N, nl, nq = 500, 4, 5
    X, lab = S.mixture(N, D, nl, 900 + D, scale="aniso")
    P = S.random_orthogonal(D, 901)
    ix = erq.build_index(to_dev(X), to_dev(P), B, nl, assign=to_dev(lab))
    Q = S.mixture(nq, D, nl, 902, comp_seed=900 + D, scale="aniso")[0]
    ids = S.rng(903).integers(0, N, (nq, nc)).astype(np.int64)
    ids[1, 0] = -1
    g = S.normal((nq, nc), 904)
    f = {k: ix.export(k).numpy() for k in ("centroids", "list_ids", "list_offsets", "f_add", "f_res")}
    codes = ix.export("codes").numpy().view(np.uint16 if B > 8 else np.uint8).astype(np.float64)
    row = np.empty(N, np.int64)
    row[f["list_ids"]] = np.arange(N)
    cl = np.searchsorted(f["list_offsets"], np.arange(N), side="right") - 1
    r = row[np.maximum(ids, 0)]
    c, y, fr = f["centroids"][cl[r]].astype(np.float64), codes[r] - (2 ** B - 1) / 2, f["f_res"][r].astype(np.float64)
    q, P64, w = Q.astype(np.float64)[:, None, :], P.astype(np.float64), np.where(ids >= 0, g, 0.0)
    if metric == "l2":
        e = ((q - c) ** 2).sum(2) + f["f_add"][r] + fr * (y * ((q - c) @ P64)).sum(2)
        gq = 2 * (w[..., None] * (q - c)).sum(1) + ((w * fr)[..., None] * y).sum(1) @ P64.T
    else:
        e = (c * q).sum(2) - 0.5 * fr * (y * (q @ P64)).sum(2)
        gq = (w[..., None] * c).sum(1) - 0.5 * ((w * fr)[..., None] * y).sum(1) @ P64.T
    est = ix.estimate(to_dev(Q), to_dev(ids), metric=metric).cpu().numpy()
    assert np.isnan(est[ids < 0]).all()
    ok = ids >= 0
    assert np.abs(est - e)[ok].max() <= 1e-5 * np.abs(e[ok]).max()
    flat = torch.zeros(nq * D + 1, device="cuda")
    flat[1:] = to_dev(Q).reshape(-1)
    for Qd in (to_dev(Q), flat[1:].view(nq, D)):
        got = ix.search_backward(Qd, to_dev(ids), to_dev(g), metric=metric).cpu().numpy()
        assert np.abs(got - gq).max() <= 2e-5 * np.abs(gq).max()

"""Selection of more than 32 lists per query: the lists with the smallest
(distance, list) pairs, over row lengths that end a register tile and value
distributions that do and do not spread over the counting intervals.  Whole
numbers below 2^24 throughout, so the distances are exact; one row per list, so
the probed lists are the candidates."""
import numpy as np
import pytest
import torch

from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nlist,p", [(33, 33), (40, 36), (1023, 100), (1024, 1024), (1025, 33), (4096, 256), (4097, 300),
                                     (16384, 1000), (16390, 64)])
@pytest.mark.parametrize("kind", ["spread", "ties", "outlier"])
def test_probe_lists(erq, nlist, p, kind):
    D, nq = 64, 37
    g = np.random.default_rng(nlist + p)
    span = 2 if kind == "ties" else 200
    X = g.integers(-span, span + 1, (nlist, D)).astype(np.float32)
    if kind == "outlier":
        X[nlist // 2] *= 200.0
    Q = g.integers(-span, span + 1, (nq, D)).astype(np.float32)
    ix = erq.build_index(to_dev(X), torch.eye(D, device="cuda"), 5, nlist,
                         assign=torch.arange(nlist, dtype=torch.int32, device="cuda"))
    out = ix.search_two_stage(to_dev(Q), p, nprobe=p, return_candidates=True)   # (takes p up to 1,024)
    cand = np.sort(out[2].cpu().numpy(), axis=1)
    d = ((Q[:, None, :].astype(np.int64) - X[None].astype(np.int64)) ** 2).sum(2)
    want = np.sort(np.argsort(d, axis=1, kind="stable")[:, :p], axis=1)
    np.testing.assert_array_equal(cand, want)

"""Rows of a scan work item where list sizes differ: the largest list is not cut
into more items than the chip has SMs, whatever the average list holds, and the
results are those of any other shape."""
import numpy as np
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [1, 16])
@pytest.mark.parametrize("precision", ["fp16", "fp32", "fp8"])
@pytest.mark.parametrize("async_mode", [False, True])
def test_one_large_list(erq, nq, precision, async_mode):
    N, D, nl = 200_000, 64, 256
    X = S.rng(71).standard_normal((N, D)).astype(np.float32)
    lab = np.where(np.arange(N) % 20 == 0, 1 + (np.arange(N) // 20) % (nl - 1), 0).astype(np.int32)   # 95 % in list 0
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 72)), 4, nl, assign=to_dev(lab))
    Q = to_dev(S.rng(73).standard_normal((nq, D)).astype(np.float32) * np.float32(0.1))
    kw = dict(rerank_k=20, nprobe=8, precision=precision, return_candidates=True)
    got = ix.search(Q, 10, async_mode=async_mode, **kw)
    torch.cuda.synchronize()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = ix.scan_config()[1]
    assert -(-190_000 // rows) <= sms
    ix.set_scan_config(0, 2048)
    for a, b in zip(got, ix.search(Q, 10, **kw)):
        assert torch.equal(a, b)

"""Shapes of scan work items.  Rows where list sizes differ: the largest list is
not cut into more items than the chip has SMs, whatever the average list holds, and
the results are those of any other shape.  Queries: 128 an item only where lists
have many queries and the chip has many items.  Tuning never leaves a shape much
slower than the untuned one."""
import time

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


@pytest.mark.parametrize("nlist,D,per_list,rows,want", [(256, 64, 80, 20, 64), (256, 64, 200, 20, 64), (512, 1536, 80, 20, 128),
                                                         (512, 1536, 60, 20, 64), (512, 960, 80, 20, 64), (4096, 192, 80, 4, 128),
                                                         (32, 64, 8192, 40, 128), (2048, 64, 80, 4, 128)])
def test_queries_of_an_item(erq, nlist, D, per_list, rows, want):
    N, np_ = nlist * rows, 16
    X, _ = S.mixture(N, D, 8, 74)
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 75)), 3, nlist, assign=to_dev(np.arange(N, dtype=np.int32) % nlist))
    Q = to_dev(np.resize(S.mixture(997, D, 8, 76, comp_seed=74)[0], (per_list * nlist // np_, D)))
    got = ix.search(Q, 10, rerank_k=20, nprobe=np_, precision="fp16")
    assert ix.scan_config()[0] == want
    ix.set_scan_config(192 - want, 0)                     # the other one gives the same
    for a, b in zip(got, ix.search(Q, 10, rerank_k=20, nprobe=np_, precision="fp16")):
        assert torch.equal(a, b)


@pytest.mark.parametrize("nlist,nq,np_", [(1, 100, 1), (1, 1, 1), (64, 1, 8), (64, 300, 16)])
def test_tuning_is_not_slower_than_the_default(erq, nlist, nq, np_):
    N, D = 10_000, 128
    X, _ = S.mixture(N, D, 8, 77)
    Q = to_dev(S.mixture(nq, D, 8, 78, comp_seed=77)[0])
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(D, 79)), 4, nlist, assign=to_dev(np.arange(N, dtype=np.int32) % nlist))
    kw = dict(rerank_k=20, nprobe=np_, precision="fp16")
    plain = ix.search(Q, 10, **kw)
    shape = ix.scan_config()

    def us():
        best = []
        for _ in range(7):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(20):
                ix.search(Q, 10, async_mode=True, **kw)
            torch.cuda.synchronize()
            best.append((time.perf_counter() - t0) / 20 * 1e6)
        return min(best)

    before = us()
    tuned = ix.autotune(Q, 10, reps=5, **kw)
    for a, b in zip(plain, ix.search(Q, 10, **kw)):
        assert torch.equal(a, b)
    assert ix.scan_config() == tuned
    assert tuned == shape or us() <= 1.1 * before

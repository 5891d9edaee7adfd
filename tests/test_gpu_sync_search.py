"""A synchronous search of few (query, list) pairs returns once its planning is
checked, with its scan in flight: a scan held up for 20 ms (the test stall of the
bounded waits) is still running when the call returns, and what it reports then
comes with the next status read, as for larger searches."""
import pytest
import torch

import synthetic as S
from gpu_common import erq, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp16", "fp32", "fp8"])
@pytest.mark.parametrize("nq,nlist", [(1, 8), (300, 4), (5, 1)])
def test_small_search_returns_with_its_scan_in_flight(erq, precision, nq, nlist):
    X, _ = S.mixture(4000, 64, 8, 66)
    ix = erq.build_index(to_dev(X), to_dev(S.random_orthogonal(64, 67)), 4, nlist,
                         assign=to_dev(S.random_assign(4000, nlist, 68)))
    Q = to_dev(X[:nq])
    kw = dict(rerank_k=20, nprobe=nlist, precision=precision)
    want = ix.search(Q, 10, **kw)
    torch.cuda.synchronize()
    ix.set_wait_limit(20_000_000, stall_stage=0)
    ix.search(Q, 10, **kw)
    assert not torch.cuda.current_stream().query()
    with pytest.raises(erq.ErqError) as ei:
        ix.status()
    assert ei.value.code == erq.ERQ_ETIMEOUT
    ix.set_wait_limit(0)
    for w, g in zip(want, ix.search(Q, 10, **kw)):
        assert torch.equal(w, g)
    ix.status()

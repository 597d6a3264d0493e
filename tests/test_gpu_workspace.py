"""Searches whose filter finds no room for its scratch (needs a GB300): they run
the CUDA-core select alone, as exact, and without allocating in every call."""
import numpy as np
import pytest

import oracle
from paper_0804_1448_gb300 import inputs
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def knn():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0804_1448_gb300 import knn as mod
    return mod


def stages(ix, Q, k, metric="l2"):
    ix.set_profiling(True)
    ix.search(Q, k, metric)
    names = set(ix.profile())
    ix.set_profiling(False)
    return names


def check(dist, idx, R, Q, k, metric="l2"):
    o_dist, o_idx = oracle.knn(R, Q, parity.oracle_k(k, R.shape[0]), metric)
    parity.compare(dist.cpu().numpy(), idx.cpu().numpy(), o_dist, o_idx, k, R.shape[0])


@pytest.mark.parametrize("metric", ["l2", "l1"])
def test_a_refused_filter_is_not_tried_again_in_every_search(knn, monkeypatch, metric):
    import torch
    R, Q, k = inputs.uniform(60000, 64, seed=401), inputs.uniform(3000, 64, seed=402), 10
    Rd, Qd = torch.from_numpy(R).cuda(), torch.from_numpy(Q).cuda()
    ix = knn.Index(0, "fp32")
    ix.set_reference(Rd)
    need = ix.workspace_size(3000, k, metric)
    # a search in between needs less than the filter and more than nothing
    monkeypatch.setenv("KNN_FAULT_INJECT_OOM", str(need - 1))
    dist, idx = ix.search(Qd, k, metric)
    ix.sync()
    check(dist, idx, R, Q, k, metric)
    assert "cc_select" in stages(ix, Qd, k, metric)
    held = ix.stats()["workspace_bytes"]
    assert 0 < held < need
    # the next one neither waits for other work nor touches the workspace
    busy, done = torch.cuda.Stream(), torch.cuda.Event()
    s = torch.cuda.Stream()
    with torch.cuda.stream(busy):
        torch.cuda._sleep(400_000_000)      # 0.2 s
        done.record(busy)
    ix.search_into(Qd, k, dist, idx, metric, stream=s)
    assert not done.query()
    torch.cuda.synchronize()
    assert ix.stats()["workspace_bytes"] == held
    check(dist, idx, R, Q, k, metric)
    # memory is there again
    monkeypatch.delenv("KNN_FAULT_INJECT_OOM")
    assert "cc_select" not in stages(ix, Qd, k, metric)
    dist, idx = ix.search(Qd, k, metric)
    ix.sync()
    check(dist, idx, R, Q, k, metric)
    ix.close()

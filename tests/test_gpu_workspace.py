"""Searches whose filter finds no room for its scratch (needs a GB300): the
handle's limit, a device short of memory, and a stream under capture.  They run
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


@pytest.mark.parametrize("form", ["pair", "small", "l1", "bf16", "self"])
def test_search_under_capture(knn, form):
    """A captured search, chained kernels and all, replayed on other queries."""
    import torch
    n, m, d, k = (700, 3000, 8, 10) if form == "small" else (700, 9000, 40, 10)
    R = inputs.uniform(m, d, seed=411)
    ix = knn.Index(0, "bf16" if form == "bf16" else "fp32")
    ix.set_reference(torch.from_numpy(R).cuda())
    metric = "l1" if form == "l1" else "l2"
    rows = m if form == "self" else n
    Q = torch.zeros((n, d), device="cuda")
    s = torch.cuda.Stream()
    dist = torch.empty((rows, k), device="cuda")
    idx = torch.empty((rows, k), device="cuda", dtype=torch.int32)

    def run():
        if form == "self":
            knn._lib.knn_search_self(ix.h, k, 0, dist.data_ptr(), idx.data_ptr(), s.cuda_stream)
        else:
            ix.search_into(Q, k, dist, idx, metric, stream=s)
    run()                                    # sizes the workspace
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
        run()
    for seed in (412, 413):
        Qh = R[:n] if form == "self" else inputs.uniform(n, d, seed=seed)
        Q.copy_(torch.from_numpy(Qh))
        dist.fill_(-1)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        if form == "self":
            o_dist, o_idx = oracle.knn(R, R[:n], parity.oracle_k(k + 1, m), "l2")
            own = o_idx[:, 0] == np.arange(n)
            assert own.all()
            np.testing.assert_allclose(dist[:n].cpu().numpy(), o_dist[:, 1:k + 1], rtol=1e-5)
        else:
            check(dist, idx, R, Qh, k, metric)
    ix.sync()
    ix.close()


def test_capture_with_room_for_the_select_only(knn):
    import torch
    R, n, k = inputs.uniform(9000, 40, seed=421), 700, 10
    Rd = torch.from_numpy(R).cuda()
    whole = knn.Index(0, "fp32")
    whole.set_reference(Rd)
    need = whole.workspace_size(n, k)
    few = knn.Index(0, "fp32", workspace_limit=need - 1)
    few.set_reference(Rd)
    select = few.workspace_size(n, k)
    assert select < need
    whole.reserve(select * 4 // 5)           # grows by a quarter: still under the filter's
    whole.reserve(select)
    assert select <= whole.stats()["workspace_bytes"] < need
    Qh = inputs.uniform(n, 40, seed=422)
    Q = torch.from_numpy(Qh).cuda()
    dist = torch.empty((n, k), device="cuda")
    idx = torch.empty((n, k), device="cuda", dtype=torch.int32)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    held = whole.stats()["workspace_bytes"]
    with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
        whole.search_into(Q, k, dist, idx, "l2", stream=s)
    graph.replay()
    torch.cuda.synchronize()
    check(dist, idx, R, Qh, k)
    assert whole.stats()["workspace_bytes"] == held
    few.close()
    whole.close()


# ---- the select itself, which searches with room for a filter no longer reach

def limited(knn, R, n, k, metric="l2"):
    """A handle with room for the select but not for the filter."""
    import torch
    Rd = torch.from_numpy(R).cuda()
    free = knn.Index(0, "fp32")
    free.set_reference(Rd)
    need = free.workspace_size(n, k, metric)
    free.close()
    ix = knn.Index(0, "fp32", workspace_limit=need - 1)
    ix.set_reference(Rd)
    assert ix.workspace_size(n, k, metric) < need
    return ix


@pytest.mark.parametrize("offset", [0.0, 1000.0])
def test_select_far_from_the_origin(knn, offset):
    """Its lower bounds of the expanded distance keep their slack at the scale
    of the points' spread, so no query needs the exact fallback."""
    import torch
    R = inputs.uniform(6000, 32, seed=431) + np.float32(offset)
    Q = inputs.uniform(300, 32, seed=432) + np.float32(offset)
    ix = limited(knn, R, 300, 20)
    Qd = torch.from_numpy(Q).cuda()
    assert "cc_select" in stages(ix, Qd, 20)
    dist, idx = ix.search(Qd, 20)
    ix.sync()
    check(dist, idx, R, Q, 20)
    assert ix.stats()["fallback_queries"] == 0
    ix.close()


@pytest.mark.parametrize("metric", ["l2", "l1", "linf"])
@pytest.mark.parametrize("n,m,d,k", [(8192, 5000, 17, 20), (8193, 9001, 6, 5), (9000, 6000, 33, 60)])
def test_select_of_many_queries(knn, metric, n, m, d, k):
    """The shape of 128 queries a CTA, which starts at 8192."""
    import torch
    R, Q = inputs.uniform(m, d, seed=441), inputs.uniform(n, d, seed=442)
    ix = limited(knn, R, n, k, metric)
    Qd = torch.from_numpy(Q).cuda()
    assert "cc_select" in stages(ix, Qd, k, metric)
    dist, idx = ix.search(Qd, k, metric)
    ix.sync()
    check(dist, idx, R, Q, k, metric)
    ix.close()

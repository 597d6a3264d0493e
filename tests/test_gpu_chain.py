"""Kernels of a search launched in a chain (needs a GB300): the chain must not
cost the kernels their place on the GPU."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def knn():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0804_1448_gb300 import knn as mod
    return mod


def test_exact_fallback_keeps_its_speed_in_the_chain(knn):
    """Every point stored 100 times, so that all 2048 queries take the exact
    fallback.  With stage profiling on, an event lies between every two
    kernels, and none can start before its predecessor has ended; the chained
    search may not take longer than that one's stages together (1.9 times, when
    the fallback's CTAs were let in early and shared SMs; 1.25 leaves room for
    the clock)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(3)
    R = torch.rand((200, 96), generator=g, device="cuda").repeat(100, 1)
    Q = torch.rand((2048, 96), generator=g, device="cuda")
    ix = knn.Index(0, "fp32")
    torch.cuda.synchronize()
    ix.set_reference(R)
    s = torch.cuda.Stream()
    dist = torch.empty((2048, 10), device="cuda")
    idx = torch.empty((2048, 10), device="cuda", dtype=torch.int32)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    whole, stages = [], []
    for _ in range(4):
        ix.set_profiling(False)
        a.record(s)
        ix.search_into(Q, 10, dist, idx, "l2", stream=s)
        b.record(s)
        s.synchronize()
        whole.append(a.elapsed_time(b))
        ix.set_profiling(True)
        ix.search_into(Q, 10, dist, idx, "l2", stream=s)
        s.synchronize()
        stages.append(sum(ix.profile().values()))
    assert ix.stats()["fallback_queries"] == 8 * 2048
    ix.close()
    assert min(whole[1:]) < 1.25 * min(stages[1:]), (whole, stages)

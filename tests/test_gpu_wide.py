"""Searches of up to 304 queries finish one query per CTA (needs a GB300): the
largest such search and the smallest of the other kind agree with the oracle,
with many short lists per query (many reference splits) and a few long ones
(few splits), in every precision and distance that has lists."""
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


@pytest.mark.parametrize("precision,metric", [("bf16", "l2"), ("tf32", "l2"), ("fp32", "l2"),
                                              ("fp32", "l1"), ("fp32", "linf")])
@pytest.mark.parametrize("n,m,d,k", [
    (1, 200000, 32, 20),      # 146 splits and more
    (64, 100000, 50, 1),
    (304, 20011, 24, 100),
    (304, 4500, 40, 20),
    (305, 4500, 40, 20),
])
def test_few_queries(knn, precision, metric, n, m, d, k):
    import torch
    R = inputs.uniform(m, d, seed=801 + m)
    Q = inputs.uniform(n, d, seed=802 + n)
    ix = knn.Index(0, precision)
    ix.set_reference(torch.from_numpy(R).cuda())
    dist, idx = ix.search(torch.from_numpy(Q).cuda(), k, metric)
    ix.sync()
    ix.close()
    o_dist, o_idx = oracle.knn(R, Q, parity.oracle_k(k, m), metric)
    parity.compare(dist.cpu().numpy(), idx.cpu().numpy(), o_dist, o_idx, k, m)

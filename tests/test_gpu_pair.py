"""Float32 Euclidean searches through the operand-pair filter (m > 4096; needs
a GB300): parity with the oracle at the edges of its row layout (the extra
words inside the padding of d or in a K step of their own), of its tiles
(reference sets one row around whole tiles, query sets around 128) and of its
range of d, on shuffled and on cluster-ordered sets; and the queue of queries
it leaves to the CUDA-core select.

The rule is tests/parity.py's, which the other float32 tests use: the filter
only chooses candidates, and the finalize certifies them.
"""
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


def search(knn, R, Q, k):
    import torch
    ix = knn.Index(0, "fp32")
    ix.set_reference(torch.from_numpy(R).cuda())
    dist, idx = ix.search(torch.from_numpy(Q).cuda(), k)
    ix.sync()
    st = ix.stats()
    ix.close()
    return dist.cpu().numpy(), idx.cpu().numpy(), st


def check(knn, R, Q, k):
    assert knn.explain_plan(Q.shape[0], R.shape[0], R.shape[1], k, precision="fp32")["k_blocks"] > 0
    dist, idx, st = search(knn, R, Q, k)
    o_dist, o_idx = oracle.knn(R, Q, parity.oracle_k(k, R.shape[0]), "l2")
    parity.compare(dist, idx, o_dist, o_idx, k, R.shape[0])
    return st


@pytest.mark.parametrize("n,m,d,k", [
    (300, 4352, 11, 10),     # the extra words just fit the padding of d; 17 whole tiles
    (300, 4353, 12, 10),     # they no longer do; one row past
    (129, 5119, 16, 20),
    (128, 5120, 27, 1),
    (127, 6001, 28, 20),
    (1000, 20011, 50, 10),
    (333, 9000, 59, 33),
    (200, 9001, 60, 20),
    (257, 8192, 96, 100),
    (200, 6000, 128, 20),
    (130, 5000, 187, 20),
    (2000, 30000, 3, 5),
    (500, 120000, 8, 64),
])
def test_uniform(knn, n, m, d, k):
    st = check(knn, inputs.uniform(m, d, seed=31 + m), inputs.uniform(n, d, seed=32 + n), k)
    assert st["fallback_queries"] == 0


def test_cluster_ordered_set(knn):
    """100 tight clusters stored one after the other, queries in a few of them:
    a query's neighbours are neighbours in storage too."""
    rng = np.random.default_rng(5)
    centres = rng.uniform(0, 1, (100, 24))
    R = (np.repeat(centres, 300, 0) + 0.02 * rng.standard_normal((30000, 24))).astype(np.float32)
    Q = (np.repeat(centres[::10], 30, 0) + 0.02 * rng.standard_normal((300, 24))).astype(np.float32)
    st = check(knn, R, Q, 20)
    assert st["fallback_queries"] == 0


@pytest.mark.parametrize("n", [20, 200])
def test_queries_left_to_the_select(knn, n):
    """Half of the set so far out that its squared norms overflow float32: the
    filter lists those references for every query and its lists overflow.
    More than 32 such queries go to the CUDA-core select, which certifies them;
    20 go straight to the exact fallback."""
    R = inputs.uniform(12000, 20, seed=71)
    R[1::2] = np.float32(3e19)
    Q = inputs.uniform(n, 20, seed=72)
    st = check(knn, R, Q, 10)
    assert st["fallback_queries"] == (n if n <= 32 else 0)


def test_select_leaves_ties_to_the_fallback(knn):
    """5000 equal references: neither the filter nor the select can certify."""
    R = np.concatenate([np.full((5000, 6), 0.5, np.float32), inputs.uniform(5000, 6, seed=73) + 4])
    Q = inputs.uniform(60, 6, seed=74)
    dist, idx, st = search(knn, R, Q, 12)
    assert idx.tolist() == [list(range(12))] * 60
    assert st["fallback_queries"] == 60

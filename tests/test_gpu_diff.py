"""Manhattan and Chebyshev searches with a pilot threshold and hit lists (m >
4096, d <= 128; needs a GB300): parity with the oracle at the edges of the CTA
shapes (16, 64 and 128 queries), of the reference tiles (whole tiles, one row
past, missing last columns) and of the coordinate stages (fewer than four, one
past a stage), on shuffled and on sorted sets, and the queries left to the
heap select and to the exact fallback.  The rule is tests/parity.py's.
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


def search(knn, R, Q, k, metric):
    import torch
    ix = knn.Index(0, "fp32")
    ix.set_reference(torch.from_numpy(R).cuda())
    dist, idx = ix.search(torch.from_numpy(Q).cuda(), k, metric)
    ix.sync()
    st = ix.stats()
    ix.close()
    return dist.cpu().numpy(), idx.cpu().numpy(), st


def check(knn, R, Q, k, metric):
    dist, idx, st = search(knn, R, Q, k, metric)
    o_dist, o_idx = oracle.knn(R, Q, parity.oracle_k(k, R.shape[0]), metric)
    parity.compare(dist, idx, o_dist, o_idx, k, R.shape[0])
    return st


@pytest.mark.parametrize("metric", ["l1", "linf"])
@pytest.mark.parametrize("n,m,d,k", [
    (1, 4097, 1, 1),
    (16, 4224, 3, 5),         # 33 whole tiles
    (17, 4225, 4, 20),        # one row past
    (64, 5000, 16, 10),
    (65, 5001, 17, 10),
    (129, 20011, 33, 10),
    (300, 30000, 96, 40),
    (1000, 9000, 128, 20),
    (200, 9000, 129, 20),     # rows too long: the heap select
    (2000, 60000, 20, 100),
])
def test_uniform(knn, metric, n, m, d, k):
    check(knn, inputs.uniform(m, d, seed=131 + m), inputs.uniform(n, d, seed=132 + n), k, metric)


@pytest.mark.parametrize("metric", ["l1", "linf"])
def test_sorted_set(knn, metric):
    """Points in the order of their first coordinate, clusters one after another."""
    rng = np.random.default_rng(6)
    centres = np.sort(rng.uniform(0, 1, (100, 10)), 0)
    R = (np.repeat(centres, 200, 0) + 0.01 * rng.standard_normal((20000, 10))).astype(np.float32)
    Q = (np.repeat(centres[::20], 40, 0) + 0.01 * rng.standard_normal((200, 10))).astype(np.float32)
    assert check(knn, R, Q, 10, metric)["fallback_queries"] == 0


@pytest.mark.parametrize("metric", ["l1", "linf"])
@pytest.mark.parametrize("n", [20, 100])
def test_ties_reach_the_fallback(knn, metric, n):
    """5000 equal references: the lists overflow, and the heap select (more than
    32 queries) cannot certify either."""
    R = np.concatenate([np.full((5000, 6), 0.5, np.float32), inputs.uniform(5000, 6, seed=173) + 4])
    Q = inputs.uniform(n, 6, seed=174)
    dist, idx, st = search(knn, R, Q, 12, metric)
    assert idx.tolist() == [list(range(12))] * n
    assert st["fallback_queries"] == n


@pytest.mark.parametrize("n", [20, 100])
def test_few_finite_distances(knn, n):
    """Six references at a finite Manhattan distance, fewer than the filter's
    candidates: the lists stay short, and the other forms answer."""
    R = np.full((6000, 5), np.float32(3e38))
    R[::1000] = inputs.uniform(6, 5, seed=175)
    Q = inputs.uniform(n, 5, seed=176)
    dist, idx, _ = search(knn, R, Q, 1, "l1")
    want = np.abs(Q[:, None].astype(np.float64) - R[None, ::1000].astype(np.float64)).sum(-1)
    np.testing.assert_array_equal(idx[:, 0], want.argmin(1) * 1000)
    np.testing.assert_allclose(dist[:, 0], want.min(1), rtol=1e-5)

"""What a float32 filter cannot certify (needs a GB300): the length of the queue
that skips the CUDA-core select, and the select over a queue at the edges of its
CTA shapes.  The rule is tests/parity.py's."""
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


def ladders(m, n, n_ladder, d=16, rungs=100, step=5e-7, seed=5):
    """Uniform points; around each of n_ladder of the queries `rungs` references
    at squared distances 0.01 + i step: more of them within the operand pairs'
    slack (some 7e-5 here) than the filter keeps.  The select keeps as many in
    every one of its splits, over which they are spread."""
    rng = np.random.default_rng(seed)
    Q = inputs.uniform(n, d, seed=seed + 1)
    R = inputs.uniform(m, d, seed=seed + 2)
    at = rng.permutation(m)[:n_ladder * rungs].reshape(n_ladder, rungs)
    who = rng.permutation(n)[:n_ladder]
    s = np.sqrt(0.01 + step * np.arange(rungs))
    for q, rows in zip(who, at):
        u = rng.standard_normal((rungs, d))
        u /= np.linalg.norm(u, axis=1, keepdims=True)
        R[rows] = (Q[q].astype(np.float64) + s[:, None] * u).astype(np.float32)
    return R, Q


def check(knn, R, Q, k, rows=None):
    import torch
    ix = knn.Index(0, "fp32")
    ix.set_reference(torch.from_numpy(R).cuda())
    dist, idx = ix.search(torch.from_numpy(Q).cuda(), k)
    ix.sync()
    st = ix.stats()
    ix.close()
    dist, idx = dist.cpu().numpy(), idx.cpu().numpy()
    if rows is not None:
        dist, idx, Q = dist[rows], idx[rows], Q[rows]
    o_dist, o_idx = oracle.knn(R, Q, parity.oracle_k(k, R.shape[0]), "l2")
    parity.compare(dist, idx, o_dist, o_idx, k, R.shape[0])
    return st


@pytest.mark.parametrize("m,direct", [(20000, True), (600000, False)])
def test_short_queues_of_a_large_set_take_the_select(knn, m, direct):
    """16 queries that the filter cannot certify: among 20000 references the
    exact fallback spreads them over the GPU; among 600000 it would spread 6 and
    read the whole set through one CTA for each of the others, and the select,
    which certifies them all, is the faster form."""
    R, Q = ladders(m, 16, 16)
    st = check(knn, R, Q, 10)
    if direct:
        assert st["fallback_queries"] > 8
    else:
        assert st["fallback_queries"] == 0


@pytest.mark.parametrize("where", ["first", "middle", "huge", "nan"])
@pytest.mark.parametrize("d", [8, 32, 96])
def test_outliers_do_not_move_the_centre(knn, d, where):
    """A row far from all others, or one that is no point at all, wherever it is
    stored: the filter still certifies (what 20 queries among 20000 references
    leave uncertified goes to the exact fallback)."""
    R = inputs.uniform(20000, d, seed=91)
    Q = inputs.uniform(20, d, seed=92)
    if where == "first":
        R[0] += np.float32(30.0)
    elif where == "middle":
        R[10000:10010] -= np.float32(1000.0)
    elif where == "huge":
        R[0] = np.float32(1e30)
    else:
        R[0] = np.nan
    if where == "nan":   # the oracle has no order for it: the other rows, moved up by one
        import torch
        ix = knn.Index(0, "fp32")
        ix.set_reference(torch.from_numpy(R).cuda())
        dist, idx = ix.search(torch.from_numpy(Q).cuda(), 10)
        ix.sync()
        st = ix.stats()
        ix.close()
        o_dist, o_idx = oracle.knn(R[1:], Q, parity.oracle_k(10, 19999), "l2")
        parity.compare(dist.cpu().numpy(), idx.cpu().numpy() - 1, o_dist, o_idx, 10, 19999)
    else:
        st = check(knn, R, Q, 10)
    assert st["fallback_queries"] == 0


def test_centre_of_a_whitened_set(knn):
    """Mahalanobis searches run on whitened rows, which have a centre of their own."""
    import torch
    d = 24
    R = inputs.uniform(20000, d, seed=93) + np.float32(50.0)
    R[0] += np.float32(30.0)
    Q = inputs.uniform(20, d, seed=94) + np.float32(50.0)
    M = np.diag(np.linspace(1.0, 4.0, d))
    ix = knn.Index(0, "fp32")
    ix.set_reference(torch.from_numpy(R).cuda())
    ix.set_mahalanobis(M)
    dist, idx = ix.search(torch.from_numpy(Q).cuda(), 10, "mahalanobis")
    ix.sync()
    st = ix.stats()
    ix.close()
    o_dist, o_idx = oracle.knn_mahalanobis(R, Q, M, parity.oracle_k(10, 20000))
    parity.compare(dist.cpu().numpy(), idx.cpu().numpy(), o_dist, o_idx, 10, 20000)
    assert st["fallback_queries"] == 0


@pytest.mark.parametrize("n", [16, 300])
@pytest.mark.parametrize("m,d,k", [(20000, 1, 10), (100000, 2, 10), (1000000, 2, 10),
                                   (1000000, 3, 10), (4000000, 3, 5)])
def test_dense_points(knn, n, m, d, k):
    """Points so dense that a filter with the select's candidates could not
    certify: it keeps more, or is not planned; at most a query in a hundred
    reaches the exact fallback (16 of 16 did at d = 1)."""
    st = check(knn, inputs.uniform(m, d, seed=95), inputs.uniform(n, d, seed=96), k,
               rows=np.arange(0, n, max(1, n // 32)))
    assert st["fallback_queries"] <= n // 100


def test_bound_near_the_float32_limit(knn):
    """Squared distances within 3e-5 of the largest float32, queries at the
    centre: the threshold passes half that limit, and twice it must not become a
    bound of +inf, which would certify whatever the cut left.  Each far row has
    its length in two coordinates with large remainders, which the filter's
    slack counts as nearness; the ten nearest have theirs in one, with none."""
    d, m = 16, 4352
    g = np.random.default_rng(21)
    R = np.zeros((m, d))
    pair = g.integers(0, d // 2, m)
    top = 3.40281e38
    a = np.float32(1.0 + 2.0 ** -8 - 2.0 ** -17) * 2.0 ** 63          # just past a bf16 half unit
    b = np.sqrt(top * (1 - 8e-6 * g.random(m)) - a.astype(np.float64) ** 2)
    rows = np.arange(m)
    R[rows, 2 * pair] = g.choice([-1.0, 1.0], m) * a
    R[rows, 2 * pair + 1] = g.choice([-1.0, 1.0], m) * b
    near = 100 + 400 * np.arange(10)
    R[near] = 0
    R[near, 2 * pair[near]] = 2.0 ** 64 * (1 - 8e-6 - 4e-7 * np.arange(10))
    R = R.astype(np.float32)
    assert np.all(np.isfinite((R * R).sum(1, dtype=np.float32)))
    Q = np.zeros((16, d), np.float32)
    check(knn, R, Q, 10)


@pytest.mark.parametrize("n,left", [(8192, 150), (9000, 400)])
def test_queue_of_a_large_search(knn, n, left):
    """Part of 8192 or more queries left over: the select of 128 queries a CTA
    over a queue that fills no whole number of them.  It certifies most, though
    with few splits its own margin of 8 candidates is narrow here."""
    R, Q = ladders(60000, n, left)
    st = check(knn, R, Q, 10)
    assert st["fallback_queries"] < left // 2

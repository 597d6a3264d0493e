"""Where a float32 Euclidean search plans the operand-pair filter
(knn_explain_plan; no GPU): not where points are so dense on the scale of their
spread that its answers cannot be certified, and with more candidates on the way
there; no different elsewhere."""
import numpy as np
import pytest

from paper_0804_1448_gb300 import knn

U = 2.0 ** -24


def plan(n, m, d, k):
    return knn.explain_plan(n, m, d, k, precision="fp32", num_sms=152)


@pytest.mark.parametrize("m,d,k", [(20000, 1, 10), (100000, 1, 1), (4000000, 1, 100),
                                   (1000000, 2, 10), (20000000, 2, 100), (2000000000, 3, 10)])
@pytest.mark.parametrize("n", [1, 300, 4096])
def test_dense_points_take_the_select(n, m, d, k):
    p = plan(n, m, d, k)
    assert p["k_blocks"] == 0 and p["candidates"] == k + max(8, k // 4)


@pytest.mark.parametrize("m,d,k", [(5000, 2, 10), (20000, 3, 5), (38400, 3, 5), (38400, 8, 20),
                                   (38400, 96, 20), (20011, 50, 10), (1000000, 8, 10),
                                   (4000000, 8, 10), (1048576, 128, 100), (4194304, 96, 20)])
def test_sparse_points_keep_the_filter_as_it_was(m, d, k):
    p = plan(4096, m, d, k)
    assert p["k_blocks"] > 0 and p["candidates"] == k + max(8, k // 4)


def slack(d, rows):
    hs = (d + 15) // 16
    acc = 17.0 * U * (3 * hs + (0 if d + 5 <= 16 * hs else 1))
    common = 1.0004 * 2.0 ** -18 + (d + 16) * U
    left = 0.23 * 2.0 ** -16
    return (2 * (common + 0.51 * acc) + 2 * (common + 1.02 * acc) + acc + 4 * left) * rows


@pytest.mark.parametrize("m,d,k", [(5000, 1, 100), (100000, 2, 1), (100000, 2, 10), (100000, 3, 20),
                                   (1000000, 3, 10), (20000, 8, 10)])
def test_candidates_reach_past_the_slack(m, d, k):
    """Uniform points: all but a few queries have fewer references within the
    slack of their k-th distance than the plan keeps.  (The slack of a query near
    its neighbours: 2 eq n_q + 2 er n_r + a |t|, n_q, n_r and 2 |t| about the
    query's squared distance from the centre; a |t| counts twice.)"""
    g = np.random.default_rng(7)
    R = g.random((m, d))
    Q = g.random((100, d))
    keep = plan(100, m, d, k)["candidates"]
    short = 0
    for q in Q:
        D = ((R - q) ** 2).sum(1)
        kth = np.partition(D, k - 1)[k - 1]
        short += np.count_nonzero(D <= kth + slack(d, ((q - 0.5) ** 2).sum())) > keep
    assert short <= 1

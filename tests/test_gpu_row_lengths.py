"""Tensor-core searches in bf16 and tf32 (needs a GB300) at row lengths around
every change of the operand rows' layout: rows padded to whole MMA K steps, so
that the last 128-byte block is read in part; whole-tile stages (up to two blocks)
and single-block ones (three to seven); raw hit staging and codes; and query
counts around whole tiles.  The float32 form's row lengths are in
tests/test_gpu_pair.py.

The rule is tests/test_gpu_tc.py's: every row the oracle's under
tests/parity.py, every distance exact within 1e-5.
"""
import pytest

import oracle
from paper_0804_1448_gb300 import inputs
from tests import parity
from tests.test_gpu_tc import check_all_rows, knn, run   # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,d", [("bf16", 60), ("bf16", 61), ("bf16", 124), ("bf16", 188),
                                         ("bf16", 252), ("bf16", 300), ("bf16", 380), ("bf16", 444),
                                         ("tf32", 28), ("tf32", 60), ("tf32", 92), ("tf32", 124),
                                         ("tf32", 156), ("tf32", 188), ("tf32", 220)])
@pytest.mark.parametrize("n,m", [(129, 9001), (257, 5000)])
def test_row_lengths(knn, precision, d, n, m):
    R = inputs.uniform(m, d, seed=5000 + d)
    Q = inputs.uniform(n, d, seed=6000 + n)
    assert knn.explain_plan(n, m, d, 10, precision=precision)["tensor_cores"] == 1
    g_dist, g_idx = run(knn, R, Q, 10, precision)
    o_dist, o_idx = oracle.knn(R, Q, parity.oracle_k(10, m), "l2")
    check_all_rows(R, Q, g_dist, g_idx, o_dist, o_idx, 10)


@pytest.mark.parametrize("precision", ["bf16", "tf32"])
@pytest.mark.parametrize("n", [128, 129, 384, 2500])
def test_query_tiles(knn, precision, n):
    R = inputs.uniform(20011, 50, seed=7001)
    Q = inputs.uniform(n, 50, seed=7002)
    g_dist, g_idx = run(knn, R, Q, 20, precision)
    o_dist, o_idx = oracle.knn(R, Q, parity.oracle_k(20, R.shape[0]), "l2")
    check_all_rows(R, Q, g_dist, g_idx, o_dist, o_idx, 20)


def test_longer_rows_run_in_float32(knn):
    assert knn.explain_plan(300, 9000, 445, 10, precision="bf16")["tensor_cores"] == 0
    assert knn.explain_plan(300, 9000, 221, 10, precision="tf32")["tensor_cores"] == 0

"""What the tensor cores make of a sum (needs a GB300): every certificate of a
float32 Euclidean search allows an MMA step, 16 exact products added to the
accumulator, an error of 17 * 2^-24 of the largest among its products and the
sums before and after it.  Checked on operands of the search's kind and on
operands made to lose as much as possible, against float64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0804_1448_gb300 import knn
    ix = knn.Index(0, "fp32")

    def run(A, B, steps):
        A = np.ascontiguousarray(A, np.float32)
        B = np.ascontiguousarray(B, np.float32)
        D = np.empty((128, 256), np.float32)
        assert A.shape == (128, 64) and B.shape == (256, 64)
        assert knn.knn_selftest_mma(ix.h, A.ctypes.data, B.ctypes.data, steps, D.ctypes.data) == 0
        return D
    yield run
    assert knn.knn_selftest_mma(ix.h, None, None, 1, None) == 1
    ix.close()


def bf16(x):
    b = np.ascontiguousarray(x, np.float32).view(np.uint32).astype(np.uint64)
    b = (b + 0x7fff + ((b >> 16) & 1)) & 0xffff0000
    return b.astype(np.uint32).view(np.float32).astype(np.float64)


def worst(D, A, B, steps):
    """The largest error over what the steps are allowed together."""
    a, b = bf16(A), bf16(B)
    s = np.zeros((128, 256))
    allowed = np.zeros((128, 256))
    for i in range(steps):
        p = a[:, None, 16 * i:16 * i + 16] * b[None, :, 16 * i:16 * i + 16]
        t = s + p.sum(-1)
        allowed += 17 * 2.0 ** -24 * np.maximum(np.abs(p).max(-1), np.maximum(np.abs(s), np.abs(t)))
        s = t
    return np.max(np.abs(D - s) / np.maximum(allowed, 1e-300))


def operands(kind, g):
    if kind == "normal":
        return g.standard_normal((128, 64)), g.standard_normal((256, 64))
    if kind == "positive":
        return g.random((128, 64)), g.random((256, 64))
    if kind == "wide":
        return (g.standard_normal((128, 64)) * 2.0 ** g.integers(-12, 1, (128, 64)),
                g.standard_normal((256, 64)) * 2.0 ** g.integers(-12, 1, (256, 64)))
    # one product of 1 (a first one, or the sum so far) and others near 2^-e
    e, sign, where = kind
    A = 2.0 ** -e * (1 + g.integers(0, 128, (128, 64)) / 128)
    B = 1 + g.integers(0, 128, (256, 64)) / 128
    A *= sign
    for s in range(4):
        A[:, 16 * s:16 * s + 16] *= 2.0 ** -(s % 2)
    if where == "last":
        A[:, :48] *= 2.0 ** -3
        A[:, 48], B[:, 48] = 1, 1
    else:
        A[:, 0], B[:, 0] = 1, 1
    return A, B


@pytest.mark.parametrize("steps", [1, 2, 4])
@pytest.mark.parametrize("kind", ["normal", "positive", "wide"] +
                         [(e, s, w) for e in (20, 22, 23, 24, 25, 26, 27) for s in (1, -1)
                          for w in ("first", "last")], ids=str)
def test_steps_stay_within_the_bound(probe, kind, steps):
    A, B = operands(kind, np.random.default_rng(11))
    assert worst(probe(A, B, steps), A, B, steps) <= 1.0


def test_layout(probe):
    """Integers, whose sums are exact."""
    g = np.random.default_rng(12)
    A, B = g.integers(-8, 9, (128, 64)), g.integers(-8, 9, (256, 64))
    for steps in (1, 3, 4):
        np.testing.assert_array_equal(probe(A, B, steps), A[:, :16 * steps] @ B[:, :16 * steps].T)

"""The operand-pair filter's bound, in numpy: with q' and r' taken relative to
a centre and written as pairs of bf16 words, acc = h.h + l.h + h.l - (1/2 - er)
n_r + t and the query's bound b = (1 - 2 eq) n_q + 2 t - 2 a |t|, every
reference has ||q - r||^2 >= b - 2 acc.  Checked against float64 distances with
the accumulation the slack allows for (every MMA step of 16 products cutting
each of its 17 addends at 2^-23 of the largest, towards the side that hurts) on
large offsets, near duplicates and far outliers.  No GPU."""
import numpy as np
import pytest

U = 2.0 ** -24


def bf16(x):
    b = np.ascontiguousarray(x, np.float32).view(np.uint32).astype(np.uint64)
    b = (b + 0x7fff + ((b >> 16) & 1)) & 0xffff0000
    return b.astype(np.uint32).view(np.float32)


def slack(d):
    acc = 34.0 * U * (3 * ((d + 15) // 16) + 1)
    common = 1.505 * 2.0 ** -16 + (d + 16) * U
    return common + 0.51 * acc, common + 1.02 * acc, acc   # eq, er, a


def cut_sum(products, acc):
    """acc + the 16 products of one MMA step, each addend cut downwards at
    2^-23 of the largest (less acc means a larger bound: the unsafe side)."""
    top = np.maximum(np.abs(products).max(-1), np.abs(acc))
    quantum = 2.0 ** (np.floor(np.log2(np.maximum(top, 1e-300))) - 23)
    return (np.floor(products / quantum[..., None]).sum(-1) + np.floor(acc / quantum)) * quantum


def bounds(Q, R, c, t):
    d = Q.shape[1]
    pad = (-d) % 16
    def words(X):
        x = (X - c).astype(np.float32)
        n = (x * x).sum(1, dtype=np.float32)
        h = bf16(x)
        l = bf16(x - h)
        z = np.zeros((X.shape[0], pad), np.float32)
        return np.hstack([h, z]).astype(np.float64), np.hstack([l, z]).astype(np.float64), n
    qh, ql, nq = words(Q)
    rh, rl, nr = words(R)
    eq, er, a = slack(d)
    acc = np.zeros((Q.shape[0], R.shape[0]))
    for s in range(0, d + pad, 16):
        for A, B in ((qh, rh), (ql, rh), (qh, rl)):
            acc = cut_sum(A[:, None, s:s + 16] * B[None, :, s:s + 16], acc)
    v = (-(np.float32(0.5) - np.float32(er)) * nr).astype(np.float32)
    w1 = bf16(v)
    w2 = bf16(v - w1)
    w3 = bf16((v - w1) - w2)
    aug = np.broadcast_to(np.stack([w1, w2, w3], 1)[None].astype(np.float64), acc.shape + (3,))
    acc = cut_sum(np.concatenate([aug, np.full(acc.shape + (1,), t)], -1), acc)
    nq = nq.astype(np.float64)
    b = nq * (1 - 2 * eq - 8 * U) + 2 * t - (2 * a + 16 * U) * abs(t) - 1e-33
    return b[:, None] - 2 * acc


@pytest.mark.parametrize("d", [3, 11, 12, 33, 96, 187])
@pytest.mark.parametrize("offset", [0.0, 1000.0, -3.5e4])
def test_bound_never_exceeds_the_distance(d, offset):
    g = np.random.default_rng(50 + d)
    R = (g.random((150, d)) + offset).astype(np.float32)
    R[140:] += np.float32(300.0)                                # far outliers
    Q = (g.random((40, d)) + offset).astype(np.float32)
    Q[:10] = R[:10]
    Q[10:20] = (R[10:20] + np.float32(1e-3) * g.standard_normal((10, d))).astype(np.float32)
    D = ((Q[:, None].astype(np.float64) - R[None].astype(np.float64)) ** 2).sum(-1)
    for t in (0.0, -0.25 * d, 40.0):
        L = bounds(Q, R, R[0], t)
        assert np.all(L <= D), np.max(L - D)
        near = D[:, :140]                                       # tight: a few 1e-4 of the norms
        assert np.max((near - L[:, :140]) / (near + d + 2 * abs(t))) < 2e-3


def test_every_reference_has_one_row():
    """The order of the copy: row p, column c of tile g, is reference
    ((c mod 64) 4 + c / 64) T + g, and the filter's index of column 64 g4 + x is
    (4 x + g4) T + g."""
    for m in (1, 255, 256, 4097, 20011):
        T = (m + 255) // 256
        p = np.arange(T * 256)
        g, c = p // 256, p % 256
        j = ((c % 64) * 4 + c // 64) * T + g
        assert sorted(j) == list(range(T * 256))
        g4, x = c // 64, c % 64
        np.testing.assert_array_equal(j, (4 * x + g4) * T + g)

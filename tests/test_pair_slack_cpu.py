"""The operand-pair filter's bound with the rows' own remainders, in numpy.

acc = h.h + l.h + h.l - (1/2 - er) n_r + w_r + t and b = (n_q - 2 w_q) (1 - 2 eq)
+ 2 t - 2 a |t|, w = 1.504 |x - h|^2 of a row x = h + l + e: every reference has ||q - r||^2 >= b - 2 acc, with the accumulation the slack allows
for (17 addends a step, each cut at 2^-24 of the largest, towards the side that
hurts).  No GPU."""
import numpy as np
import pytest

U = 2.0 ** -24


def bf16(x):
    b = np.ascontiguousarray(x, np.float32).view(np.uint32).astype(np.uint64)
    b = (b + 0x7fff + ((b >> 16) & 1)) & 0xffff0000
    return b.astype(np.uint32).view(np.float32)


def steps(d):
    hs = (d + 15) // 16
    return 3 * hs + (0 if d + 5 <= 16 * hs else 1)


def slack(d):
    acc = 17.0 * U * steps(d)
    common = 64.01 * U + (d + 16) * U
    return common + 0.51 * acc, common + 1.02 * acc, acc   # eq, er, a


def cut_sum(products, acc):
    """acc + the products of one MMA step, each addend cut downwards at 2^-24 of
    the largest (less acc means a larger bound: the unsafe side)."""
    top = np.maximum(np.abs(products).max(-1), np.abs(acc))
    quantum = 2.0 ** (np.floor(np.log2(np.maximum(top, 1e-300))) - 24)
    return (np.floor(products / quantum[..., None]).sum(-1) + np.floor(acc / quantum)) * quantum


def words(X, c):
    x = (X - c).astype(np.float32)
    n = (x * x).sum(1, dtype=np.float32)
    h = bf16(x)
    l = bf16(x - h)
    e = (x - h) - l
    assert np.all(h.astype(np.float64) + l + e == x)
    assert np.all(np.abs(e) <= 2.0 ** -8 * np.abs(x - h))
    w = 1.506 * ((x - h).astype(np.float64) ** 2).sum(1)
    pad = np.zeros((X.shape[0], (-X.shape[1]) % 16), np.float32)
    return np.hstack([h, pad]).astype(np.float64), np.hstack([l, pad]).astype(np.float64), n, \
        w.astype(np.float32)


def bounds(Q, R, c, t):
    d = Q.shape[1]
    qh, ql, nq, wq = words(Q, c)
    rh, rl, nr, wr = words(R, c)
    eq, er, a = slack(d)
    v = ((np.float32(er) - np.float32(0.5)) * nr + wr).astype(np.float32)
    w1 = bf16(v)
    w2 = bf16(v - w1)
    extra = np.stack([w1, w2, (v - w1) - w2], 1).astype(np.float64)
    acc = np.zeros((Q.shape[0], R.shape[0]))
    extra = np.concatenate([np.broadcast_to(extra[None], acc.shape + (3,)),
                            np.full(acc.shape + (1,), t)], -1)
    hs = (d + 15) // 16
    inside = d + 5 <= 16 * hs
    sl = [slice(16 * s, 16 * s + 16) for s in range(hs)]
    prod = lambda A, B, s: A[:, None, s] * B[None, :, s]
    for s in range(hs):                       # the order of the MMA issuer
        p = prod(qh, rh, sl[s])
        if inside and s == hs - 1:
            p = np.concatenate([p, extra], -1)
        acc = cut_sum(p, acc)
        acc = cut_sum(prod(ql, rh, sl[s]), acc)
    for s in range(hs):
        acc = cut_sum(prod(qh, rl, sl[s]), acc)
    if not inside:
        acc = cut_sum(extra, acc)
    b = (nq - 2 * wq).astype(np.float64) * (1 - 2 * eq - 10 * U) + 2 * t \
        - (2 * a + 16 * U) * abs(t) - 1e-33
    return b[:, None] - 2 * acc


def worst_rows(g, rows, d):
    """Coordinates whose lower words and rests are as large as they get: just
    past half a unit of the upper word, and of the lower."""
    x = 1.0 + 2.0 ** -8 - 2.0 ** -17 - 2.0 ** -23 + np.zeros((rows, d))
    return (x * g.choice([-1.0, 1.0], (rows, 1)) * 2.0 ** g.integers(-2, 3, (rows, 1))).astype(np.float32)


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
        L = bounds(Q, R, np.median(R, 0), t)
        assert np.all(L <= D), np.max(L - D)
        near = D[:, :140]
        assert np.max((near - L[:, :140]) / (near + d + 2 * abs(t))) < 1e-3


@pytest.mark.parametrize("d", [3, 16, 96, 187])
def test_rows_with_the_largest_remainders(d):
    g = np.random.default_rng(60 + d)
    R, Q = worst_rows(g, 60, d), worst_rows(g, 20, d)
    D = ((Q[:, None].astype(np.float64) - R[None].astype(np.float64)) ** 2).sum(-1)
    zero = np.zeros(d, np.float32)
    for t in (0.0, 0.5 * d):
        assert np.all(bounds(Q, R, zero, t) <= D)
    *_, n, w = words(R, zero)
    assert np.all(w < 1.51 * 2.0 ** -16 * n) and np.all(w > 1.2 * 2.0 ** -16 * n)


def test_ordinary_rows_leave_little():
    X = np.random.default_rng(9).random((500, 24)).astype(np.float32)
    *_, n, w = words(X, np.float32(0.5))
    assert np.mean(w / n) < 0.25 * 2.0 ** -16

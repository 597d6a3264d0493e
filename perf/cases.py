"""Timed work of the library: what its users have it do, through the public
binding (paper_0804_1448_gb300.knn), over the range of sizes, dimensions,
precisions, distances and forms it serves.

Every case is one call on inputs already in hand: a search of n queries among
m resident references, a self-join, or a batch of independent searches.
Points are uniform in [0, 1)^d or drawn from a Gaussian mixture, the
distributions of the library's workloads (inputs.py).
"""
from __future__ import annotations

import math

import torch

from paper_0804_1448_gb300 import knn

# n * m * d of the largest listed searches: Euclidean in bf16 / tf32, and
# float32 (which also serves the Manhattan and Chebyshev distances)
_MOST_TENSOR = 16384 * 1048576 * 128
_MOST_FP32 = 38400 * 38400 * 96
_MOST_POINTS = 4194304 * 96          # m * d of the largest resident reference set


def _search(name, n, m, d, k, precision="fp32", metric="l2", data="uniform", io="device"):
    return dict(name=name, kind="search", n=n, m=m, d=d, k=k, precision=precision, metric=metric,
                data=data, io=io)


def listed():
    return [
        # the smallest problem of the paper's Table 1, at the binding's default
        # precision: launches and latency
        _search("small_n1200_d8_fp32", 1200, 1200, 8, 20),
        # an ordinary default-precision search at sizes nobody picked for a tile
        _search("ragged_n4999_m20011_d50_fp32", 4999, 20011, 50, 10),
        # the largest problem of Table 1 in float32 ...
        _search("table1_n38400_d96_fp32", 38400, 38400, 96, 20),
        # ... in bf16, the workload the library is quoted on ...
        _search("table1_n38400_d96_bf16", 38400, 38400, 96, 20, "bf16"),
        # ... and the same search from and to pinned host memory, copies included
        _search("host_n38400_d96_bf16", 38400, 38400, 96, 20, "bf16", io="host"),
        # the paper's other distance, at a middle size of Table 1
        _search("manhattan_n19200_d80", 19200, 19200, 80, 20, "fp32", "l1"),
        # Chebyshev distances, few queries, odd sizes, rows that are no whole float4s
        _search("chebyshev_n3001_m30011_d33", 3001, 30011, 33, 10, "fp32", "linf"),
        # descriptor-like clustered points, a large set, many neighbours
        _search("mixture_n16384_m1048576_d128_k100_bf16", 16384, 1048576, 128, 100, "bf16",
                data="mixture"),
        # serving: one small request against a resident set of four million points
        _search("serve_n64_m4194304_d96_bf16", 64, 4194304, 96, 20, "bf16"),
        # Mahalanobis distances in tf32: whitening and the second tensor-core precision
        _search("mahalanobis_n9600_m19200_d64_tf32", 9600, 19200, 64, 20, "tf32", "mahalanobis"),
        # the neighbours among the other points that the entropy estimate reads
        dict(name="selfjoin_m20000_d3_fp32", kind="self", m=20000, d=3, k=4, precision="fp32",
             metric="l2"),
        # many uneven independent searches handed over at once
        dict(name="batch_32_bf16", kind="batch", count=32, precision="bf16", n_max=4096,
             m_max=200000, shapes=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["search", "self", "batch"], [10, 1, 1])[0]
    if kind == "self":
        d = _log_int(rng, 3, 16)
        return dict(kind="self", m=_log_int(rng, 2000, 38400), d=d, k=rng.randint(1, 20),
                    precision=rng.choice(["fp32", "bf16"]), metric="l2")
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 32), precision=rng.choice(["bf16", "tf32"]),
                    n_max=_log_int(rng, 256, 4096), m_max=_log_int(rng, 8000, 200000),
                    shapes=rng.randrange(1 << 20))
    precision = rng.choice(["fp32", "fp32", "bf16", "bf16", "tf32"])
    metric = rng.choices(["l2", "l1", "linf", "mahalanobis"], [7, 1, 1, 1])[0]
    fp32 = precision == "fp32" or metric in ("l1", "linf")
    most = _MOST_FP32 if fp32 else (_MOST_TENSOR if precision == "bf16" else _MOST_TENSOR // 2)
    while True:
        n, m = _log_int(rng, 1, 38400), _log_int(rng, 1200, 4194304)
        d, k = _log_int(rng, 8, 128), _log_int(rng, 1, 100)
        # short rows cost a search as much as rows of 32 coordinates
        if n * m * max(d, 32) <= most and m * d <= _MOST_POINTS and n * k <= 16384 * 100:
            break
    return dict(kind="search", n=n, m=m, d=d, k=k, precision=precision, metric=metric,
                data=rng.choice(["uniform", "uniform", "mixture"]),
                io="host" if n <= 38400 and rng.random() < 0.15 else "device")


# ---------------------------------------------------------------------- inputs

def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _uniform(rows, d, seed, salt):
    return torch.rand((rows, d), generator=_gen(seed, salt), device="cuda", dtype=torch.float32)


def _mixture(rows, d, centres, seed, salt):
    g = _gen(seed, salt)
    x = torch.randn((rows, d), generator=g, device="cuda", dtype=torch.float32).mul_(0.05)
    which = torch.randint(0, centres.shape[0], (rows,), generator=g, device="cuda")
    return x.add_(centres[which])


def _points(case, seed):
    """(R, Q) of a search, on the GPU."""
    n, m, d = case["n"], case["m"], case["d"]
    if case["data"] == "mixture":
        centres = _uniform(1024, d, seed, 1)
        return _mixture(m, d, centres, seed, 2), _mixture(n, d, centres, seed, 3)
    return _uniform(m, d, seed, 2), _uniform(n, d, seed, 3)


def _inverse_covariance(case, seed):
    """A symmetric positive definite matrix with eigenvalues from 1 to 30."""
    d = case["d"]
    a = torch.randn((d, d), generator=_gen(seed, 4), device="cuda", dtype=torch.float64)
    rot, _ = torch.linalg.qr(a)
    ev = torch.linspace(1.0, 30.0, d, device="cuda", dtype=torch.float64)
    s = (rot * ev) @ rot.T
    return 0.5 * (s + s.T)


def _instance_shapes(case):
    """The batching workload's shapes (d in {32, 64, 128}, k in {1, 10, 50}),
    fixed by the case."""
    g = torch.Generator().manual_seed(case["shapes"])
    def pick(lo, hi):
        return int(torch.randint(lo, hi + 1, (1,), generator=g))
    return [(pick(16, case["n_max"]), pick(1000, case["m_max"]), (32, 64, 128)[pick(0, 2)],
             (1, 10, 50)[pick(0, 2)]) for _ in range(case["count"])]


def prepare(case, seed):
    if case["kind"] == "batch":
        inst = []
        for i, (n, m, d, k) in enumerate(_instance_shapes(case)):
            inst.append(dict(R=_uniform(m, d, seed, 100 + 2 * i), Q=_uniform(n, d, seed, 101 + 2 * i),
                             k=k, dist=torch.empty((n, k), device="cuda"),
                             idx=torch.empty((n, k), device="cuda", dtype=torch.int32)))
        return dict(case=case, index=knn.Index(0, case["precision"]), instances=inst)
    ix = knn.Index(0, case["precision"])
    if case["kind"] == "self":
        R, Q = _uniform(case["m"], case["d"], seed, 2), None
    else:
        R, Q = _points(case, seed)
    torch.cuda.current_stream().synchronize()   # set_reference reads R on the handle's own stream
    ix.set_reference(R)
    if case["kind"] == "self":
        return dict(case=case, index=ix)
    if case["metric"] == "mahalanobis":
        ix.set_mahalanobis(_inverse_covariance(case, seed).cpu().numpy())
    st = dict(case=case, index=ix, Q=Q)
    if case["io"] == "host":
        n, k = case["n"], case["k"]
        st["Q"] = Q.cpu().pin_memory()
        st["dist"] = torch.empty((n, k), dtype=torch.float32).pin_memory()
        st["idx"] = torch.empty((n, k), dtype=torch.int32).pin_memory()
    return st


def run(state):
    case, ix = state["case"], state["index"]
    stream = torch.cuda.current_stream()
    if case["kind"] == "batch":
        ix.search_batch(state["instances"], stream=stream)
        return [dict(dist=x["dist"], idx=x["idx"]) for x in state["instances"]]
    if case["kind"] == "self":
        dist, idx = ix.search_self(case["k"], case["metric"], stream=stream)
        return dict(dist=dist, idx=idx)
    if case["io"] == "host":
        ix.search_into(state["Q"], case["k"], state["dist"], state["idx"], case["metric"],
                       stream=stream)
        return dict(dist=state["dist"], idx=state["idx"])
    dist, idx = ix.search(state["Q"], case["k"], case["metric"], stream=stream)
    return dict(dist=dist, idx=idx)


# ------------------------------------------------------------------------ work

def _search_work(n, m, d, k, metric, ref_bytes):
    # the resident references in the precision the distances are formed in, the
    # float32 queries, the outputs; one multiply-add (or difference and
    # accumulation) per coordinate pair
    return (ref_bytes * m * d + 4 * n * d + 8 * n * k, 2 * n * m * d)


def work(case):
    ref_bytes = 2 if case["precision"] == "bf16" else 4
    if case["kind"] == "batch":
        parts = [_search_work(n, m, d, k, "l2", 4) for n, m, d, k in _instance_shapes(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if case["metric"] in ("l1", "linf"):
        ref_bytes = 4
    n = case["m"] if case["kind"] == "self" else case["n"]
    b, f = _search_work(n, case["m"], case["d"], case["k"], case["metric"], ref_bytes)
    if case["metric"] == "mahalanobis":
        f += n * case["d"] * (case["d"] + 1)       # whitening the queries
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------- 64-bit answer

def _nearest(Q, R, k, metric, skip_self=False):
    """The k nearest rows of R to each row of Q (float64), ascending by
    (distance, index): a few spare candidates from one pass over all distances,
    then their distances from coordinate differences."""
    n, m = Q.shape[0], R.shape[0]
    keep = min(m, k + 8 + (1 if skip_self else 0))
    dist = torch.empty((n, k), device=Q.device, dtype=torch.float64)
    idx = torch.empty((n, k), device=Q.device, dtype=torch.int32)
    nr = (R * R).sum(1)
    rows = max(1, min(n, (1 << 28) // m))
    for a in range(0, n, rows):
        q = Q[a:a + rows]
        if metric == "l2":
            key = torch.addmm(nr[None, :], q, R.T, alpha=-2.0)
        else:
            key = torch.cdist(q, R, p=1.0 if metric == "l1" else float("inf"))
        if skip_self:
            i = torch.arange(q.shape[0], device=Q.device)
            key[i, a + i] = float("inf")
        cand = torch.topk(key, keep, dim=1, largest=False).indices
        del key
        cand, _ = torch.sort(cand, dim=1)
        for b in range(0, q.shape[0], 4096):
            c = cand[b:b + 4096]
            diff = (R[c] - q[b:b + 4096, None, :]).abs_()
            e = (diff.square_().sum(2) if metric == "l2"
                 else diff.sum(2) if metric == "l1" else diff.amax(2))
            if skip_self:
                own = torch.arange(a + b, a + b + c.shape[0], device=Q.device)
                e[c == own[:, None]] = float("inf")
            e, order = torch.sort(e, dim=1, stable=True)
            e = e[:, :k]
            lo = a + b
            dist[lo:lo + c.shape[0]] = e.sqrt() if metric == "l2" else e
            idx[lo:lo + c.shape[0]] = torch.gather(c, 1, order)[:, :k].int()
    return dist, idx


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for i, (n, m, d, k) in enumerate(_instance_shapes(case)):
            dist, idx = _nearest(_uniform(n, d, seed, 101 + 2 * i).double(),
                                 _uniform(m, d, seed, 100 + 2 * i).double(), k, "l2")
            out.append(dict(dist=dist, idx=idx))
        return out
    if case["kind"] == "self":
        R = _uniform(case["m"], case["d"], seed, 2).double()
        dist, idx = _nearest(R, R, case["k"], "l2", skip_self=True)
        return dict(dist=dist, idx=idx)
    R, Q = _points(case, seed)
    R, Q = R.double(), Q.double()
    metric = case["metric"]
    if metric == "mahalanobis":
        L = torch.linalg.cholesky(_inverse_covariance(case, seed))
        R, Q, metric = R @ L, Q @ L, "l2"
    dist, idx = _nearest(Q, R, case["k"], metric)
    if case["io"] == "host":
        dist, idx = dist.cpu(), idx.cpu()
    return dict(dist=dist, idx=idx)

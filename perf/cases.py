"""Timed cases of the SpKAdd library: B = A_1 + ... + A_k through its public entry points.

Kinds of inputs, after the library's own workloads:

  er         Erdos-Renyi columns: `d` distinct uniform rows in every column of
             every input, or (ragged) a Poisson number with mean `d`.
  rmat       R-MAT graphs of 2^scale vertices, 16 edges per vertex, quadrant
             probabilities .57, .19, .19, .05: a few huge columns, many tiny.
  spgemm     partial products of a sparse matrix product: column j has 4 L_j
             candidate rows and every input holds about L_j of them, so that
             the inputs overlap heavily.
  unordered  partial products whose rows come in no order inside a column
             (option input_order = 1).
  tall       few columns of a very long row range (k sparse vectors, or a
             block of them, of millions of rows).
  batch      many independent problems of mixed k, shape and type in one call.
  stream     a running sum on the device, inputs added a few at a time.
"""
import json
import math
import zlib

import numpy as np
import torch

import paper_2112_10223_gb300 as spk

DTYPES = {"f32": torch.float32, "f64": torch.float64}
RMAT = (0.57, 0.19, 0.19, 0.05)
EDGE_FACTOR = 16


def listed():
    return [
        # A small system assembled from four parts: the latency of one call.
        dict(name="er_small", kind="er", k=4, m=1024, n=1024, d=8, ragged=False, dtype="f64", values="int",
             method="twopass"),
        # An ordinary sum of a handful of matrices, odd sizes, into buffers of the input's size.
        dict(name="er_onepass", kind="er", k=7, m=300007, n=300007, d=11, ragged=True, dtype="f32", values="uniform",
             method="onepass"),
        # The paper's Erdos-Renyi experiment at the largest size (32 inputs of 2^20 x 2^20, 16 per column).
        dict(name="er_large", kind="er", k=32, m=1 << 20, n=1 << 20, d=16, ragged=False, dtype="f64",
             values="uniform", method="twopass"),
        # Summing small graphs (snapshots of an evolving network).
        dict(name="rmat_small", kind="rmat", k=16, scale=14, dtype="f64", method="twopass"),
        # The paper's R-MAT experiment at the largest size.
        dict(name="rmat_large", kind="rmat", k=64, scale=20, dtype="f32", method="twopass"),
        # Stage sums of a distributed sparse product (SUMMA): equal column lengths, large overlap.
        dict(name="spgemm_stages", kind="spgemm", k=64, m=1 << 17, n=1 << 17, L_lo=32, L_hi=32, ragged=False,
             dtype="f32", method="twopass"),
        # Many stages of a smaller product: ragged columns of thousands of entries.
        dict(name="spgemm_many", kind="spgemm", k=250, m=20011, n=20011, L_lo=4, L_hi=64, ragged=True, dtype="f64",
             method="twopass"),
        # Products straight from a hash SpGEMM, whose columns are not sorted.
        dict(name="unordered_products", kind="unordered", k=24, m=65537, n=65537, L_lo=8, L_hi=64, ragged=True,
             dtype="f32", method="twopass"),
        # Sparse vectors of millions of rows (index sets touched by workers), a block of columns at once.
        dict(name="tall_vectors", kind="tall", k=24, m=3000017, n=96, d=20011, dtype="f32", method="twopass"),
        # Many independent sums of mixed sizes and types, one call.
        dict(name="batch_mixed", kind="batch", count=20, k_lo=2, k_hi=64, n_lo=1024, n_hi=16384, L_lo=4, L_hi=64),
        # Products that arrive in groups and do not fit together: a running sum.
        dict(name="stream_sum", kind="stream", k=32, group=8, m=1 << 16, n=1 << 16, L_lo=32, L_hi=32, ragged=False,
             dtype="f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fit(k, n, d, limit):
    """n, lowered so that k * n * d stays below `limit` entries."""
    return max(1, min(n, int(limit / (k * max(d, 1)))))


def draw(rng):
    kind = rng.choice(["er", "er", "rmat", "spgemm", "spgemm", "unordered", "tall", "batch", "stream"])
    dtype = rng.choice(["f32", "f64"])
    method = rng.choice(["twopass", "twopass", "onepass"])
    if kind == "er":
        k, d = _log(rng, 2, 64), _log(rng, 2, 64)
        m = _log(rng, 1000, 1 << 20)
        return dict(kind=kind, k=k, m=m, n=_fit(k, m, d, 2.5e8), d=d, ragged=rng.random() < 0.5, dtype=dtype,
                    values=rng.choice(["uniform", "int"]), method=method)
    if kind == "rmat":
        scale = rng.randint(10, 19)
        return dict(kind=kind, k=_log(rng, 2, 64), scale=scale, dtype=dtype, method=method)
    if kind in ("spgemm", "unordered"):
        k, lo = _log(rng, 4, 300), rng.randint(2, 32)
        hi = rng.randint(lo, 64)
        m = _log(rng, 1000, 1 << 18)
        return dict(kind=kind, k=k, m=m, n=_fit(k, m, (lo + hi) / 2, 6e7 if kind == "unordered" else 1.2e8), L_lo=lo,
                    L_hi=hi, ragged=kind == "unordered" or rng.random() < 0.5, dtype=dtype, method=method)
    if kind == "tall":
        k, n = _log(rng, 3, 64), _log(rng, 1, 256)
        m = _log(rng, 1 << 18, 1 << 23)
        d = max(64, min(m // 16, _log(rng, 2000, 60000), int(4e7 / (k * n))))
        return dict(kind=kind, k=k, m=m, n=n, d=d, dtype=dtype, method=method)
    if kind == "batch":
        return dict(kind=kind, count=_log(rng, 4, 20), k_lo=2, k_hi=_log(rng, 8, 80), n_lo=1024,
                    n_hi=_log(rng, 2048, 16384), L_lo=rng.randint(2, 8), L_hi=rng.randint(16, 64))
    k, lo = _log(rng, 8, 48), rng.randint(4, 32)
    hi = rng.randint(lo, 40)
    m = _log(rng, 2000, 1 << 17)
    return dict(kind="stream", k=k, group=rng.randint(3, 9), m=m, n=_fit(k, m, (lo + hi) / 2, 8e7), L_lo=lo, L_hi=hi,
                ragged=rng.random() < 0.5, dtype=dtype)


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------
def _values(g, count, dtype, kind="uniform"):
    if kind == "int":
        x = torch.randint(0, 16, (count,), generator=g, device="cuda", dtype=torch.int8)
        return torch.where(x < 8, x - 8, x - 7).to(dtype)
    return torch.rand(count, generator=g, device="cuda", dtype=dtype) * 2 - 1


def _counts_to_ptr(counts):
    ptr = torch.zeros(counts.numel() + 1, dtype=torch.int32, device="cuda")
    torch.cumsum(counts, 0, out=ptr[1:])
    return ptr


def _from_keys(keys, m, n):
    """CSC pattern of sorted distinct keys col * m + row."""
    cols = torch.div(keys, m, rounding_mode="floor")
    rows = (keys - cols * m).to(torch.int32)
    bounds = torch.arange(n + 1, device="cuda", dtype=torch.int64) * m
    return torch.searchsorted(keys, bounds).to(torch.int32), rows


def _uniform_rows(g, n, d, m):
    """(n, d) int32: d distinct uniform rows per column, ascending."""
    rows = torch.randint(0, m, (n, d), generator=g, device="cuda", dtype=torch.int32).sort(dim=1).values
    while True:
        bad = (rows[:, 1:] == rows[:, :-1]).any(dim=1).nonzero().squeeze(1)
        if bad.numel() == 0:
            return rows
        rows[bad] = torch.randint(0, m, (bad.numel(), d), generator=g, device="cuda",
                                  dtype=torch.int32).sort(dim=1).values


def _er(g, k, m, n, d, ragged):
    d = min(d, m // 2)
    out = []
    for _ in range(k):
        if ragged:
            keys = torch.randint(0, n * m, (n * d,), generator=g, device="cuda", dtype=torch.int64)
            cp, ri = _from_keys(torch.unique(keys), m, n)
        else:
            ri = _uniform_rows(g, n, d, m).reshape(-1)
            cp = torch.arange(n + 1, device="cuda", dtype=torch.int32) * d
        out.append((cp, ri))
    return out


def _rmat(g, k, scale):
    m = 1 << scale
    a, b, c, _ = RMAT
    out = []
    for _ in range(k):
        rows = torch.zeros(EDGE_FACTOR * m, dtype=torch.int32, device="cuda")
        cols = torch.zeros_like(rows)
        for _ in range(scale):
            u = torch.rand(rows.numel(), generator=g, device="cuda")
            low = u >= a + b
            rows.mul_(2).add_(low)
            cols.mul_(2).add_((u >= a + b + c) | ((u >= a) & ~low))
        out.append(_from_keys(torch.unique(cols.to(torch.int64) * m + rows), m, m))
    return out


def _products(g, k, m, n, lo, hi, ragged, shuffle=False):
    """Inputs drawn from 4 L_j candidate rows per column: one of every four
    candidates, or (ragged) each candidate with probability 1/4."""
    lo, hi = min(lo, m // 8), min(hi, m // 8)
    L = torch.randint(lo, hi + 1, (n,), generator=g, device="cuda", dtype=torch.int64)
    # Candidates: one uniform row in each of 4 L_j equal ranges of the column's rows.
    col = torch.repeat_interleave(torch.arange(n, device="cuda"), 4 * L)
    start = torch.zeros(n, dtype=torch.int64, device="cuda")
    start[1:] = torch.cumsum(4 * L, 0)[:-1]
    t = torch.arange(col.numel(), device="cuda") - start[col]
    w = 4 * L[col]
    x0, x1 = t * m // w, (t + 1) * m // w
    u = torch.rand(col.numel(), generator=g, device="cuda", dtype=torch.float64)
    cand = torch.minimum(x0 + (u * (x1 - x0)).to(torch.int64), x1 - 1).to(torch.int32)
    del t, w, x0, x1, u
    out = []
    for _ in range(k):
        if ragged:
            pick = (torch.rand(cand.numel(), generator=g, device="cuda") < 0.25).nonzero().squeeze(1)
            cp = _counts_to_ptr(torch.bincount(col[pick], minlength=n))
        else:
            pick = torch.arange(cand.numel() // 4, device="cuda") * 4
            pick += torch.randint(0, 4, (pick.numel(),), generator=g, device="cuda")
            cp = _counts_to_ptr(L)
        if shuffle:
            key = col[pick].to(torch.float64) + torch.rand(pick.numel(), generator=g, device="cuda",
                                                           dtype=torch.float64) * 0.999
            pick = pick[key.argsort()]
        out.append((cp, cand[pick]))
    return out


def _filled(patterns, g, dtype, kind="uniform"):
    """The inputs of one seed: the case's patterns in another order, with their
    columns rotated and values of their own.  Every seed then has the same
    nnz(B), and so outputs of the same sizes."""
    n = patterns[0][0].numel() - 1
    order = torch.randperm(len(patterns), generator=g, device="cuda").tolist()
    shift = int(torch.randint(0, n, (1,), generator=g, device="cuda"))
    out = []
    for i in order:
        cp, ri = patterns[i]
        p = int(cp[shift])
        cp = torch.cat([cp[shift:] - p, cp[1:shift + 1] + (ri.numel() - p)])
        ri = torch.cat([ri[p:], ri[:p]])
        out.append((cp, ri, _values(g, ri.numel(), dtype, kind)))
    return out


def _batch_params(case):
    """The problems of a batch: k and n log-uniform, either family, either type."""
    r = np.random.default_rng(case["count"])
    out = []
    for _ in range(case["count"]):
        k = int(round(math.exp(r.uniform(math.log(case["k_lo"]), math.log(case["k_hi"])))))
        n = int(round(math.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        out.append((k, n, "er" if r.random() < 0.5 else "spgemm", "f32" if r.random() < 0.5 else "f64"))
    return out


def prepare(case, seed):
    same = json.dumps({key: v for key, v in case.items() if key != "name"}, sort_keys=True)
    shape = torch.Generator(device="cuda")  # the patterns belong to the case
    shape.manual_seed(zlib.crc32(same.encode()))
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    if kind == "batch":
        problems = []
        for k, n, family, dt in _batch_params(case):
            if family == "er":
                P = _er(shape, k, n, n, (case["L_lo"] + case["L_hi"]) // 2, True)
            else:
                P = _products(shape, k, n, n, case["L_lo"], case["L_hi"], False)
            problems.append((_filled(P, g, DTYPES[dt]), n))
        return dict(kind=kind, problems=problems)
    dtype = DTYPES[case["dtype"]]
    m = 1 << case["scale"] if kind == "rmat" else case["m"]
    if kind in ("er", "tall"):
        P = _er(shape, case["k"], m, case["n"], case["d"], case.get("ragged", True))
    elif kind == "rmat":
        P = _rmat(shape, case["k"], case["scale"])
    else:
        P = _products(shape, case["k"], m, case["n"], case["L_lo"], case["L_hi"], case["ragged"],
                      shuffle=kind == "unordered")
    state = dict(kind=kind, A=_filled(P, g, dtype, case.get("values", "uniform")), m=m,
                 method=case.get("method", "twopass"), options=None)
    if kind == "unordered":
        state["options"] = spk.default_options(input_order=1)
    if kind == "stream":
        state.update(n=case["n"], dtype=dtype, group=case["group"])
    return state


def run(state):
    if state["kind"] == "batch":
        return spk.spkadd_batch(state["problems"])
    if state["kind"] == "stream":
        s = spk.SpkaddStream(state["m"], state["n"], dtype=state["dtype"])
        for i in range(0, len(state["A"]), state["group"]):
            s.add(state["A"][i:i + state["group"]])
        out = s.result()
        s.close()
        return out
    return spk.spkadd(state["A"], state["m"], options=state["options"], method=state["method"])


# ---------------------------------------------------------------------------
# What a pass cannot do without, and what it should return.
# ---------------------------------------------------------------------------
def _er_counts(k, m, n, d):
    d = min(d, m // 2)
    return k * n * d, n * m * -math.expm1(k * math.log1p(-d / m))


def _product_counts(k, m, n, lo, hi):
    lo, hi = min(lo, m // 8), min(hi, m // 8)
    mean = (lo + hi) / 2
    return k * n * mean, 4 * mean * n * (1 - 0.75 ** k)


def _rmat_counts(k, scale):
    """Expected distinct edges of one matrix (times k) and of the union: the
    cells of equal probability a^i b^j d^l are counted together."""
    a, b, _, d = RMAT
    edges = EDGE_FACTOR * 2.0 ** scale
    one = union = 0.0
    for i in range(scale + 1):
        for j in range(scale + 1 - i):
            l = scale - i - j
            cells = math.factorial(scale) / (math.factorial(i) * math.factorial(j) * math.factorial(l)) * 2.0 ** j
            p = a ** i * b ** j * d ** l
            one += cells * -math.expm1(-edges * p)
            union += cells * -math.expm1(-k * edges * p)
    return k * one, union


def _bytes(k, n, nnz_in, nnz_out, dtype):
    entry = 4 + (4 if dtype == "f32" else 8)
    return (nnz_in + nnz_out) * entry + k * (n + 1) * 4 + (n + 1) * 8


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total = adds = 0
        for k, n, family, dt in _batch_params(case):
            if family == "er":
                i, o = _er_counts(k, n, n, (case["L_lo"] + case["L_hi"]) // 2)
            else:
                i, o = _product_counts(k, n, n, case["L_lo"], case["L_hi"])
            total += _bytes(k, n, i, o, dt)
            adds += i
        return {"bytes": int(total), "flops": int(adds)}
    if kind in ("er", "tall"):
        i, o = _er_counts(case["k"], case["m"], case["n"], case["d"])
        n = case["n"]
    elif kind == "rmat":
        i, o = _rmat_counts(case["k"], case["scale"])
        n = 1 << case["scale"]
    else:
        i, o = _product_counts(case["k"], case["m"], case["n"], case["L_lo"], case["L_hi"])
        n = case["n"]
    return {"bytes": int(_bytes(case["k"], n, i, o, case["dtype"])), "flops": int(i)}


def tolerance(case):
    """Column pointers and rows are whole numbers and exact.  Sums of small
    integers are exact; others differ by the rounding of their order.
    Measured against 64-bit sums (float) and against sums in another order
    (double), times four."""
    if case["kind"] == "er" and case["values"] == "int":
        return "exact"
    if case["kind"] == "batch":
        return {"rel": 6e-7}
    return {"rel": 6e-7 if case["dtype"] == "f32" else 2e-15}


def _exact_sum(A, m):
    """The sum in 64 bits, a range of columns at a time."""
    n = A[0][0].numel() - 1
    ptrs = [a[0].to(torch.int64) for a in A]
    total = torch.stack(ptrs).sum(0)
    out_cp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rows, vals = [], []
    c0 = 0
    while c0 < n:
        limit = total[c0] + (1 << 27)
        c1 = int(torch.searchsorted(total, limit, right=True)) - 1
        c1 = min(n, max(c0 + 1, c1))
        keys, terms = [], []
        for p, (_, ri, va) in zip(ptrs, A):
            lo, hi = int(p[c0]), int(p[c1])
            col = torch.repeat_interleave(torch.arange(c1 - c0, device="cuda"), p[c0 + 1:c1 + 1] - p[c0:c1],
                                          output_size=hi - lo)
            keys.append(col * m + ri[lo:hi])
            terms.append(va[lo:hi].to(torch.float64))
        key, order = torch.cat(keys).sort()
        term = torch.cat(terms)[order]
        del keys, terms, order
        uniq, count = torch.unique_consecutive(key, return_counts=True)
        group = torch.repeat_interleave(torch.arange(uniq.numel(), device="cuda"), count, output_size=key.numel())
        s = torch.zeros(uniq.numel(), dtype=torch.float64, device="cuda").index_add_(0, group, term)
        bounds = torch.arange(1, c1 - c0 + 1, device="cuda", dtype=torch.int64) * m
        out_cp[c0 + 1:c1 + 1] = out_cp[c0] + torch.searchsorted(uniq, bounds)
        rows.append((uniq % m).to(torch.int32))
        vals.append(s)
        c0 = c1
    return out_cp, torch.cat(rows), torch.cat(vals)


def exact(case, seed):
    state = prepare(case, seed)
    if state["kind"] == "batch":
        return [_exact_sum(A, m) for A, m in state["problems"]]
    return _exact_sum(state["A"], state["m"])

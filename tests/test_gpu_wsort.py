"""Light columns sorted in registers: key counts, segment tables, row limits, and the one-pass tiles.

Small-integer values: indices and sums must match the oracle exactly in either type.
"""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_2112_10223_gb300 as spk
from spk_testlib import compare, run_gpu, to_np
from test_gpu_items import _columns

pytestmark = pytest.mark.gpu

# 32 E keys hold a column, E = 1, 2, 4, 8, 10, 12 or 16.
LENGTHS = [0, 1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 288, 289, 300, 319, 320, 321, 383, 384, 385,
           511, 512]


def _check(A, m, dtype, **opt):
    want = oracle.add(to_np(A))
    s = sum(a[0].cpu().diff() for a in A).numpy()
    unique = int(((np.diff(want["col_ptr"]) == s) & (s > 0)).sum())
    launches = {}
    for method in ("twopass", "onepass"):
        out = run_gpu(A, m, dtype=dtype, options=spk.default_options(**opt), info=True, method=method)
        compare(tuple(t.cpu().numpy() for t in out[:3]), want, dtype, exact=True)
        assert out[3]["onepass"] == (method == "onepass") and out[3]["cols_unique"] == unique
        launches[method] = out[3]["kernel_launches"]
    outs = spk.spkadd_batch([([tuple(t.cuda() for t in a) for a in A], m)] * 2, options=spk.default_options(**opt))
    for o in outs:
        compare(tuple(t.cpu().numpy() for t in o), want, dtype, exact=True)
    return launches


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("m", [600, 1 << 16, 65537, 1 << 23, (1 << 23) + 1])  # bitmaps 2^16 rows, keys below 2^23
def test_key_counts_and_row_limits(m, dtype):
    A = _columns(29, m, LENGTHS, 4, dtype)
    _check(A, m, dtype)


@pytest.mark.parametrize("k", [1, 31, 32, 33, 63, 64, 65, 130])  # tables hold 64 inputs, two per lane
def test_segment_tables(k):
    lengths = [min(s, 40 * k) for s in LENGTHS]
    A = _columns(k, 4000, lengths, 5, torch.float64, [max(120, s // 2) for s in lengths])
    _check(A, 4000, torch.float64)
    _check(A, 4000, torch.float64, input_order=1, sort_mode=1)


def test_equal_runs_and_last_rows():
    """Every input the same: runs of k equal rows; rows up to the last."""
    m = (1 << 23) - 1
    rows = torch.arange(m - 25, m, dtype=torch.int32)
    cp = torch.tensor([0, 25, 25, 50], dtype=torch.int32)
    A = [(cp, torch.cat([rows, rows - 70]), torch.arange(50, dtype=torch.float64) - i) for i in range(20)]
    _check(A, m, torch.float64)


@pytest.mark.parametrize("d", [2, 9, 20, 40])  # columns per warp and tile follow the longest column
def test_onepass_columns_per_warp(d):
    n = 8 * 16 * 152 * 12 + 77  # enough columns for the largest tiles, and a ragged last one
    g = torch.Generator().manual_seed(d)
    A = []
    for _ in range(3):
        keep = torch.rand(n, d, generator=g) < 0.5
        col, at = keep.nonzero(as_tuple=True)
        cp = torch.zeros(n + 1, dtype=torch.int32)
        cp[1:] = torch.cumsum(keep.sum(1), 0)
        va = torch.randint(-8, 9, (at.numel(),), generator=g).to(torch.float64)
        A.append((cp, (at * 7).to(torch.int32), va))
    want = oracle.add(to_np(A))
    out = run_gpu(A, 7 * d, info=True, method="onepass")
    assert out[3]["onepass"] == 1
    compare(tuple(t.cpu().numpy() for t in out[:3]), want, torch.float64, exact=True)


def _dealt(k, m, lengths, n, dtype, seed):
    """k inputs; n columns of each length, dealt evenly to the inputs.  The rows of every other length lie close
    together (many repeats across the inputs), those of the others anywhere."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    rows, counts = [[] for _ in range(k)], [[] for _ in range(k)]
    for at, s in enumerate(lengths):
        for i in range(k):
            L = s // k + (i < s % k)
            step = max(1, (m if at % 2 else 3 * max(1, s // k)) // max(L, 1))
            r = torch.arange(L, device="cuda") * step + torch.randint(0, step, (n, L), generator=g, device="cuda")
            rows[i].append(r.reshape(-1).to(torch.int32))
            counts[i].append(torch.full((n,), L, device="cuda"))
    out = []
    for i in range(k):
        cp = torch.zeros(n * len(lengths) + 1, dtype=torch.int32, device="cuda")
        cp[1:] = torch.cumsum(torch.cat(counts[i]), 0)
        ri = torch.cat(rows[i])
        out.append((cp, ri, torch.randint(-8, 9, (ri.numel(),), generator=g, device="cuda").to(dtype)))
    return out


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("k", [5, 32, 33, 70])  # inputs in registers, one chunk, two halves of a table, two tables
def test_short_and_long_columns_in_kernels_of_their_own(k, dtype):
    """Enough columns of both lengths that each is summed by its own kernel, at every network's edges; and by one."""
    m = 60000
    both = _dealt(k, m, [s for s in LENGTHS if s >= 31], 3200, dtype, k)
    assert _check(both, m, dtype)["twopass"] == 7  # bins, three counts, scan, two light sums
    few = _dealt(k, m, [s for s in LENGTHS if s >= 31], 50, dtype, k)
    assert _check(few, m, dtype)["twopass"] == 6
    long = _dealt(k, m, [s for s in LENGTHS if s > 288], 300, dtype, k)
    assert _check(long, m, dtype)["twopass"] == 6
    for rows in (m, 70000):  # a mean above 384: no networks of 320 and 384 keys
        assert _check(_dealt(k, rows, [256, 385, 511, 512, 500], 60, dtype, k), rows, dtype)["twopass"] == 6


def test_columns_just_above_the_short_ones():
    """Columns of 257 to 288 entries of few repeats go to the buckets when there are many."""
    m, n = 40000, 16400  # (mean 149: too many repeats expected for all long columns to go there)
    near = _dealt(6, m, [20, 257, 20, 288, 20, 289], n, torch.float64, 1)
    assert _check(near, m, torch.float64)["twopass"] == 8  # bins, three counts, scan, sort of short and long, buckets
    repeats = _dealt(6, m, [257, 20, 288, 20, 289, 20], n, torch.float64, 1)
    assert _check(repeats, m, torch.float64)["twopass"] == 7
    assert _check(_dealt(6, m, [20, 257, 20, 288, 20, 289], 100, torch.float64, 1), m, torch.float64)["twopass"] == 6


def test_columns_split_between_sort_and_buckets():
    """Few repeats expected (large m): the long columns go to the buckets, those that repeat after all to the sort."""
    m = 1 << 22
    lengths = [300, 512, 257, 256, 100, 400] * 20
    pool = [400 if j % 6 == 1 else m for j in range(len(lengths))]
    A = _columns(16, m, lengths, 6, torch.float64, pool)
    for mode in (0, 1):  # bins, heavy and CTA counts, two light ones, scan, two light sums
        assert _check(A, m, torch.float64, sort_mode=mode)["twopass"] == 8
    far = _columns(16, m, lengths, 6, torch.float64)  # hardly a repeat: every long column stays in the buckets
    assert _check(far, m, torch.float64)["twopass"] == 8
    short = _columns(16, 1 << 17, lengths, 6, torch.float64)  # repeats expected: all to the sort
    assert _check(short, 1 << 17, torch.float64)["twopass"] == 6


def test_float_runs_round_once_and_keep_infinities():
    """Runs of equal rows are summed as if in double: cancellation, overflow on the way, infinities and NaN."""
    inf, big = float("inf"), 3.0e38
    runs = [[1.0, 2.0 ** -30, -1.0], [big, big, -big], [big, big, big], [inf, 1.0, big], [inf, -inf, 1.0],
            [float("nan"), 1.0, 2.0], [-0.0, 0.0, -0.0], [1.0e-45, 1.0e-45, -1.0e-45], [1.0e8, 1.0, -1.0e8],
            [big, -inf, big], [16777216.0, 1.0, 1.0]]
    g = torch.Generator().manual_seed(3)
    runs += [(torch.randn(3, generator=g) * 10.0 ** torch.randint(-20, 20, (3,), generator=g)).tolist() for _ in range(400)]
    n, per = 41, len(runs) // 41 + 1
    cp = torch.arange(n + 1, dtype=torch.int32) * per
    v = torch.zeros(n * per, 3, dtype=torch.float32)
    v[:len(runs)] = torch.tensor(runs, dtype=torch.float64).to(torch.float32)
    rows = (torch.arange(per, dtype=torch.int32) * 3).repeat(n)
    A = [(cp, rows, v[:, i].contiguous()) for i in range(3)]
    d = v.double()
    want = ((d[:, 0] + d[:, 1]) + d[:, 2]).to(torch.float32)
    for method in ("twopass", "onepass"):
        got = run_gpu(A, 3 * per, method=method)[2].cpu()
        assert torch.equal(torch.isnan(got), torch.isnan(want))
        ok = ~torch.isnan(want)
        assert torch.equal(got[ok], want[ok])


@pytest.mark.parametrize("n", [2, 3, 9, 64, 256, 512])
def test_float_runs_are_as_exact_as_double_sums(n):
    """Long runs that cancel: what a sum of n floats may lose is n^3 u^3 sum|terms| (u = 2^-24), at most 2^-45 of it,
    besides its rounding to float; in all no more than a sum in double loses.  A run of minus zeros is minus zero."""
    rng, cols = np.random.default_rng(n), 240
    v = np.zeros((cols, n), dtype=np.float32)
    for c in range(cols):
        half = (rng.standard_normal(n // 2) * 2.0 ** rng.integers(-13, 13, n // 2)).astype(np.float32)
        x = np.concatenate([half, -half, rng.standard_normal(n % 2).astype(np.float32)])
        at = rng.integers(0, n, max(1, n // 8))
        x[at] += (rng.standard_normal(at.size) * (0.0, 1e-10, 1e-6, 1e-3, 1.0)[c % 5]).astype(np.float32)
        v[c] = x[rng.permutation(n)]
    v[7::40] = -0.0
    cp = torch.arange(cols + 1, dtype=torch.int32)
    A = [(cp, torch.zeros(cols, dtype=torch.int32), torch.from_numpy(v[:, i].copy())) for i in range(n)]
    exact = np.array([math.fsum(row) for row in v.astype(np.float64)])
    size = np.abs(v.astype(np.float64)).sum(1)
    acc = np.zeros(cols)
    for i in range(n):
        acc += v[:, i]
    by_double = np.abs(acc.astype(np.float32).astype(np.float64) - exact)
    for method in ("twopass", "onepass"):
        got = run_gpu(A, 5, method=method)[2].cpu().numpy()
        err = np.abs(got.astype(np.float64) - exact)
        bound = 0.5 * np.spacing(np.abs(exact).astype(np.float32)).astype(np.float64) + n ** 3 * 2.0 ** -72 * size
        assert (err <= bound).all(), (method, (err - bound).max())
        assert err.sum() <= by_double.sum()
        assert np.signbit(got[7::40]).all()

"""Thread-block items in registers: the sizes where their chunks, slots, segment tables and layouts end.

Small-integer values: indices and sums must match the oracle exactly in either type.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2112_10223_gb300 as spk
from spk_testlib import check_full, compare, to_np

pytestmark = pytest.mark.gpu


def _columns(k, m, lengths, seed, dtype, pool=None):
    """k inputs; column j has lengths[j] entries dealt to the inputs at random (some inputs get none),
    from the first pool[j] rows of a random row order when given (repeats across inputs)."""
    r = np.random.default_rng(seed)
    n = len(lengths)
    cols = [[] for _ in range(k)]
    for j, s in enumerate(lengths):
        owner = np.sort(r.integers(0, k, s))
        rows = np.empty(s, dtype=np.int64)
        cand = None if pool is None else r.choice(m, pool[j], replace=False)
        for i in np.unique(owner):
            at = owner == i
            c = int(at.sum())
            src = m if cand is None else cand
            rows[at] = np.sort(r.choice(src, c, replace=False))
        for i in range(k):
            cols[i].append(rows[owner == i])
    out = []
    for i in range(k):
        cp = np.zeros(n + 1, dtype=np.int32)
        cp[1:] = np.cumsum([len(c) for c in cols[i]])
        ri = np.concatenate(cols[i]).astype(np.int32) if cp[-1] else np.zeros(0, np.int32)
        va = r.integers(-8, 9, ri.size)
        out.append((torch.from_numpy(cp), torch.from_numpy(ri), torch.from_numpy(va).to(dtype)))
    return out


# 256 threads of 16 slots hold 4096 entries, 384 hold 6144; slots come in pairs.
LENGTHS = [1, 255, 256, 257, 511, 513, 1023, 1025, 4095, 4096, 4097, 6143, 6144, 6145, 8193, 12289]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("m", [5000, 1 << 17, (1 << 17) + 1, 1 << 20, (1 << 20) + 77])
def test_chunk_and_slot_edges(m, dtype):
    pool = [min(m, max(s // 3, 40)) for s in LENGTHS]
    A = _columns(37, m, LENGTHS, 1, dtype, pool) if m == 5000 else _columns(37, m, LENGTHS, 1, dtype)
    for opt in (None, spk.default_options(warp_max=32, block_accumulator=2),
                spk.default_options(warp_max=32, input_order=1)):
        check_full(A, m, dtype, exact=True, options=opt)


@pytest.mark.parametrize("k", [1, 2, 63, 64, 65, 255, 256, 257, 511, 512, 513, 1100])
def test_segment_table_edges(k):
    """Tables hold 512 inputs; sums of more than 167 inputs go in phases of 128 (float)."""
    lengths = [600, 1500, 3000, 5000, 9000]
    lengths = [min(s, 400 * k) for s in lengths]
    for dtype in (torch.float32, torch.float64):
        A = _columns(k, 3001, lengths, k, dtype, [min(3001, max(500, s // 2)) for s in lengths])
        check_full(A, 3001, dtype, exact=True, options=spk.default_options(warp_max=64, cta_max=2048))


def test_few_distinct_rows_many_terms():
    """Items whose entries meet on a handful of rows, and whole columns of 4096 distinct rows."""
    A = _columns(300, 4096, [1000, 4000, 20000], 3, torch.float32, [40, 90, 400])
    check_full(A, 4096, torch.float32, exact=True)
    r = torch.arange(4096, dtype=torch.int32)
    full = [(torch.tensor([0, 4096], dtype=torch.int32), r + 7, torch.ones(4096, dtype=torch.float64))]
    check_full(full, 5000, torch.float64, exact=True)
    check_full([(full[0][0], r, full[0][2])], 4096, torch.float64, exact=True)
    check_full([(full[0][0], r + ((1 << 20) - 4096), full[0][2])], 1 << 20, torch.float64, exact=True)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("k,L,m", [(40, 16, 5000), (33, 32, 1 << 23), (200, 6, 9001), (70, 64, (1 << 23) + 1)])
def test_many_columns_on_few_rows(k, L, m, dtype):
    """Enough columns on few rows for the warp-per-column table where the problem has at most 2^20 rows (others stay
    with the block items), one and several segment tables, ragged and equal inputs, in and out of order."""
    import synth
    n = 8300
    A = synth.spgemm_like(k, m, n, L, seed=9, dtype=dtype, value_kind="int8")
    A[1] = (torch.zeros(n + 1, dtype=torch.int32), A[1][1][:0], A[1][2][:0])  # an empty input: lengths differ
    check_full(A, m, dtype, exact=True)
    flipped = []
    for cp, ri, va in A:
        e = torch.arange(ri.numel())
        col = torch.repeat_interleave(torch.arange(n), (cp[1:] - cp[:-1]).long())
        at = (cp[:-1].long()[col] + cp[1:].long()[col] - 1 - e)
        flipped.append((cp, ri[at], va[at]))
    check_full(flipped, m, dtype, exact=True, options=spk.default_options(input_order=1))


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n, parts", [(3, 1), (200, 4), (1400, 1)])
def test_empty_last_window(n, parts, dtype):
    """The last cut (a multiple of 4032 distinct rows) falls into the last 64-row word, which leaves an empty
    window behind it; with more items than resident blocks, those that follow it must still be summed."""
    m, u = 1 << 18, parts * 4032 + 2
    rows = torch.cat([torch.arange(u - 10, dtype=torch.int64) * ((m - 64) // (u - 10)), torch.arange(m - 10, m)])
    ri = rows.to(torch.int32).cuda().repeat(n)
    cp = torch.arange(n + 1, dtype=torch.int32, device="cuda") * u
    va = torch.arange(u * n, device="cuda").remainder(1000).to(dtype)
    B_cp, B_ri, B_va = spk.spkadd([(cp, ri, va), (cp, ri, va)], m)
    assert torch.equal(B_cp, cp.to(torch.int64)) and torch.equal(B_ri, ri)
    assert torch.equal(B_va, 2 * va)


@pytest.mark.parametrize("n", [100, 8300])
def test_columns_on_few_rows_beyond_the_stated_nnz(n):
    """Column pointers that end past the stated nnz (the arrays behind are long enough here): more columns on few rows
    than their list, sized by nnz, holds.  The call is refused and the next one is right."""
    k, L, m = 40, 16, 64
    rows = torch.arange(L, dtype=torch.int32, device="cuda").repeat(n)
    cp = torch.arange(n + 1, dtype=torch.int32, device="cuda") * L
    va = torch.ones(L * n, dtype=torch.float64, device="cuda")
    with pytest.raises(spk.SpkaddError) as e:
        spk.spkadd([(cp, rows[:L * 10], va[:L * 10])] * k, m)
    assert e.value.name == "SPKADD_ERR_INTERNAL"
    B_cp, B_ri, B_va = spk.spkadd([(cp, rows, va)] * k, m)
    assert torch.equal(B_cp, cp.to(torch.int64)) and torch.equal(B_ri, rows) and bool((B_va == k).all())


def test_symbolic_again_after_it_failed():
    """A symbolic phase that found no memory for the windows' offsets starts over when it is called again."""
    lengths = [600] * 3000 + [30000, 200, 5000]
    A = _columns(20, 1 << 16, lengths, 11, torch.float64, [100] * 3000 + [1 << 16, 300, 700])
    Ad = [tuple(t.cuda() for t in a) for a in A]
    live, full = {}, []

    @spk.ALLOC_FN
    def alloc(nbytes, stream, ctx):
        if live and not full:  # the workspace is the first; the second is refused once
            full.append(nbytes)
            return None
        t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        live[t.data_ptr()] = t
        return t.data_ptr()

    @spk.FREE_FN
    def free(ptr, stream, ctx):
        live.pop(ptr, None)

    o = spk.default_options()
    o.alloc, o.free = alloc, free
    want = [t.cpu() for t in spk.spkadd(Ad, 1 << 16)]
    fresh = spk.spkadd(Ad, 1 << 16, info=True)[3]
    h = spk.spkadd_plan(Ad, 1 << 16, options=o)
    with pytest.raises(spk.SpkaddError) as e:
        spk.spkadd_symbolic(h)
    assert e.value.status == 6 and len(full) == 1
    nnz = spk.spkadd_symbolic(h)
    B = [torch.empty(len(lengths) + 1, dtype=torch.int64, device="cuda"), torch.empty(nnz, dtype=torch.int32, device="cuda"),
         torch.empty(nnz, dtype=torch.float64, device="cuda")]
    spk.spkadd_numeric(h, *B)
    info = spk.spkadd_get_info(h)
    spk.spkadd_destroy(h)
    assert info["status"] == "SPKADD_OK"
    for key in ("windows", "windows_split", "cols_unique"):
        assert info[key] == fresh[key], key
    assert all(torch.equal(x.cpu(), y) for x, y in zip(B, want))


def _few_rows(k, m, groups, seed, dtype):
    """k inputs of the columns of groups [(n, P, L)]: n columns, L rows out of P in every input (on the GPU)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    at = [torch.randint(0, m - 3 * P + 1, (n, 1), generator=g, device="cuda") for n, P, _ in groups]
    cp = torch.zeros(sum(n for n, _, _ in groups) + 1, dtype=torch.int32, device="cuda")
    cp[1:] = torch.cumsum(torch.cat([torch.full((n,), L, device="cuda") for n, _, L in groups]), 0)
    out = []
    for _ in range(k):
        pick = [torch.rand(n, P, generator=g, device="cuda").topk(L, dim=1).indices.sort(dim=1).values for n, P, L in groups]
        ri = torch.cat([(a + 3 * p).reshape(-1) for a, p in zip(at, pick)]).to(torch.int32)
        out.append((cp, ri, torch.randint(-8, 9, (ri.numel(),), generator=g, device="cuda").to(dtype)))
    return out


def _launches(problems, wants=None, **opt):
    """Kernels launched for the problems, whose sums are checked."""
    outs, info = spk.spkadd_batch(problems, info=True, options=spk.default_options(**opt))
    for (A, _), B, want in zip(problems, outs, wants or [oracle.add(to_np(A)) for A, _ in problems]):
        compare(tuple(t.cpu().numpy() for t in B), want, A[0][2].dtype, exact=True)
    return info["kernel_launches"]


def _flipped(A):
    """The inputs with every column's entries in the opposite order."""
    out = []
    for cp, ri, va in A:
        col = torch.repeat_interleave(torch.arange(cp.numel() - 1, device=cp.device), (cp[1:] - cp[:-1]).long())
        at = cp[:-1].long()[col] + cp[1:].long()[col] - 1 - torch.arange(ri.numel(), device=cp.device)
        out.append((cp, ri[at], va[at]))
    return out


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("k, m, P, L, beside, table", [
    (40, 5000, 31, 15, 60, True),        # one key a lane in the final sort, entries of several inputs in a round
    (600, 5000, 64, 1, 6, True),         # two keys; ten tables of 64 inputs, one entry to an input
    (40, 1 << 20, 128, 32, 60, True),    # four keys; rows up to 2^20
    (20, 9001, 255, 60, 100, True),      # eight keys
    (5, 4096, 255, 255, 700, True),      # the most distinct rows a column may have, and one more
    (5, 4096, 256, 256, 700, True),
    (5, 4096, 257, 257, 700, False),
    (130, 5000, 60, 30, 30, True),       # tables of 1920 positions: one start-bit map
    (64, 5000, 80, 48, 60, True),        # of 3072: two
    (100, 5000, 200, 50, 300, True),     # heavy columns (5000 entries), listed by k_sym_heavy
])
def test_table_of_few_rows_edges(k, m, P, L, beside, table, dtype):
    """Columns that reach the warp-per-column table, of equal and of mixed segment lengths, in and out of order.  One
    column on many rows, of the same class, goes to the block items in any case, so the table is one launch more than
    the flat accumulator makes."""
    groups = [(8300, P, L), (1, 1000, beside)]
    A = _few_rows(k, m, groups, 3, dtype)
    shorter = _few_rows(k, m, [(8300, P, max(1, L - 3)), groups[1]], 3, dtype)
    empty = (torch.zeros_like(A[0][0]), A[0][1][:0], A[0][2][:0])
    for inputs in (A, A[:k - k // 3] + shorter[:k // 3 - 1] + [empty] if P < 255 and L > 3 else A):
        want = [oracle.add(to_np(inputs))]
        for B, order in ((inputs, 0), (_flipped(inputs), 1)):
            flat = _launches([(B, m)], want, block_accumulator=1, input_order=order)
            assert _launches([(B, m)], want, input_order=order) - flat == table


def test_table_of_few_rows_in_batches():
    """One launch of the table for each problem kind; and in a batch with a problem of more than 2^20 rows, whose own
    columns are never listed, the heavy columns of the others are."""
    P = [(_few_rows(k, 4096, [(8300, 60, 15), (1, 1000, 3000 // k)], k, dt), 4096)
         for k, dt in ((40, torch.float32), (200, torch.float32), (40, torch.float64))]
    wants = [oracle.add(to_np(A)) for A, _ in P]
    assert _launches(P, wants) - _launches(P, wants, block_accumulator=1) == 3
    tall = _few_rows(30, 1 << 22, [(30, 200, 100), (10, 255, 200)], 4, torch.float64)
    P = [(_few_rows(100, 5000, [(8300, 200, 50), (1, 1000, 300)], 5, torch.float64), 5000), (tall, 1 << 22)]
    wants = [oracle.add(to_np(A)) for A, _ in P]
    assert _launches(P, wants) - _launches(P, wants, block_accumulator=2) == 1


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("more, launches", [
    ([], 0),               # all in the table: one launch, as when the block items (block_accumulator 1) take them all
    ([(1, 1000, 40)], 1),  # beside them a column on many rows: the block items' launch as well
    ([(1, 255, 55)], 0),   # 2200 entries, below the 2430 that one column may have
    ([(1, 255, 100)], 1),  # 4000 entries: to the block items
    ([(1, 255, 200)], 0),  # 8000 entries: to the block items, whose flat form launches once more, for the heavy class
])
def test_large_columns_on_few_rows_stay_out_of_the_table(more, launches, dtype):
    """A column on few rows that has many times the entries of the others is not left to one warp."""
    A = _few_rows(40, 4096, [(8300, 60, 15), *more], 5, dtype)
    assert _launches([(A, 4096)]) - _launches([(A, 4096)], block_accumulator=1) == launches


def test_few_columns_of_a_kind_stay_out_of_the_table():
    """Columns on few rows are counted kind by kind: 8300 of one kind go to the table, 5000 of another do not."""
    many = _few_rows(40, 4096, [(8300, 60, 15), (1, 1000, 40)], 6, torch.float64)
    few = _few_rows(40, 4096, [(5000, 60, 15), (1, 1000, 40)], 7, torch.float32)
    a, b = (many, 4096), (few, 4096)
    flat = _launches([a, b], block_accumulator=1)
    assert _launches([a, b]) == flat + 1  # k_num_items for either kind, and k_num_dup for one


@pytest.mark.parametrize("acc", [0, 1, 2])
@pytest.mark.parametrize("m", [1 << 17, 1 << 20, (1 << 20) + 5000])
def test_rows_out_of_order_stay_inside_the_inputs(m, acc):
    """Unordered columns stated to be ordered: B is unspecified, but every segment of a split window stays inside its
    input, and the next call is right.  (Starts of consecutive windows, found by binary search, may lie in either
    order; segments of negative length would shift the other inputs' positions past their ends.)"""
    k, L = 8, 20000
    g = torch.Generator(device="cuda").manual_seed(m)
    cp = torch.tensor([0, L, 2 * L], dtype=torch.int32, device="cuda")
    A = [(cp, torch.cat([torch.randperm(m, generator=g, device="cuda")[:L] for _ in range(2)]).to(torch.int32),
          torch.ones(2 * L, dtype=torch.float64, device="cuda")) for _ in range(k)]
    h = spk.spkadd_plan(A, m, options=spk.default_options(block_accumulator=acc))
    nnz = spk.spkadd_symbolic(h)
    B = [torch.empty(3, dtype=torch.int64, device="cuda"), torch.full((nnz,), -1, dtype=torch.int32, device="cuda"),
         torch.empty(nnz, dtype=torch.float64, device="cuda")]
    spk.spkadd_numeric(h, *B)
    info = spk.spkadd_get_info(h)
    spk.spkadd_destroy(h)
    assert info["windows_split"] > 8 and info["status"] in ("SPKADD_OK", "SPKADD_ERR_INTERNAL")
    in_order = [(c, torch.cat([r[:L].sort().values, r[L:].sort().values]), v) for c, r, v in A]
    assert check_full(in_order, m, torch.float64, exact=True)[0]["status"] == "SPKADD_OK"


def _spread(k, m, n, L, seed, dtype):
    """k inputs of n columns of L rows each, one in each of L equal ranges."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    step = m // L
    cp = torch.arange(n + 1, dtype=torch.int32, device="cuda") * L
    out = []
    for _ in range(k):
        ri = torch.arange(L, device="cuda") * step + torch.randint(0, step, (n, L), generator=g, device="cuda")
        ri = ri.reshape(-1).to(torch.int32)
        out.append((cp, ri, torch.randint(-8, 9, (ri.numel(),), generator=g, device="cuda").to(dtype)))
    return out


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("k, L", [(3, 4000), (16, 800), (40, 300), (41, 300), (200, 45), (180, 130)])
@pytest.mark.parametrize("m", [40000, 1 << 20, (1 << 21) + 3])
def test_heavy_windows_of_several_chunks(k, L, m, dtype):
    """Windows of more entries than a chunk holds, few (one block in two takes none) and more than four to an SM, in
    and out of order: walked in runs where their segments are long, chunk by chunk where they are not."""
    for n in (20, 330):
        A = _spread(k, m, n, L, k, dtype)
        want = oracle.add(to_np(A))
        for B, order in ((A, 0), (_flipped(A), 1)):
            out = spk.spkadd(B, m, info=True, options=spk.default_options(input_order=order))
            compare(tuple(t.cpu().numpy() for t in out[:3]), want, dtype, exact=True)
            assert out[3]["cols_heavy"] == n and out[3]["windows"] >= 2 * n


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_columns_over_several_slabs(dtype):
    """CTA-class columns of problems past 2^20 rows: every slab takes the rows inside it, ends of slabs among them."""
    m = (1 << 22) + 9
    A = _spread(7, m, 200, 300, 2, dtype)
    edge = torch.tensor([0, (1 << 20) - 1, 1 << 20, (1 << 21) - 1, 1 << 21, (1 << 22) - 1, 1 << 22, m - 1], dtype=torch.int32)
    cp = torch.arange(201, dtype=torch.int32, device="cuda") * 8
    A.append((cp, edge.cuda().repeat(200), torch.ones(1600, dtype=dtype, device="cuda")))
    for B, opt in ((A, {}), (_flipped(A), dict(input_order=1)), (A, dict(block_accumulator=2))):
        info, _ = check_full([tuple(t.cpu() for t in a) for a in B], m, dtype, exact=True, options=spk.default_options(**opt))
        assert info["cols_cta"] == 200

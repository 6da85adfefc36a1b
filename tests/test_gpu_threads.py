"""Distinct handles are independent: host threads with problems of other sizes, each on a stream of its own.

The problems take the same kernels with other amounts of dynamic shared memory (rows of the bitmaps, entries of the
longest column), so a launch that depended on another thread's size would be refused.
"""
import ctypes
import threading

import pytest
import torch

import paper_2112_10223_gb300 as spk

pytestmark = pytest.mark.gpu

# (method, k, m, n, entries of an input's column)
JOBS = [("onepass", 4, 900, 700, 3), ("onepass", 8, 4000, 700, 60), ("twopass", 20, 1500, 300, 40),
        ("twopass", 20, 1 << 17, 300, 40), ("twopass", 12, 1200, 60, 500), ("twopass", 12, 1 << 17, 60, 500),
        ("twopass", 12, 1 << 16, 500, 20), ("twopass", 12, 1000, 500, 20)]


def _inputs(k, m, n, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for _ in range(k):
        step = m // d
        rows = torch.arange(d, device="cuda") * step + torch.randint(0, step, (n, d), generator=g, device="cuda")
        cp = torch.arange(n + 1, dtype=torch.int32, device="cuda") * d
        out.append((cp, rows.to(torch.int32).reshape(-1),
                    torch.randint(-8, 9, (n * d,), generator=g, device="cuda").to(torch.float64)))
    return out


def test_handles_of_several_threads():
    lib = spk.library()
    problems = [(_inputs(k, m, n, d, q), m, method) for q, (method, k, m, n, d) in enumerate(JOBS)]
    want = [spk.spkadd(A, m, method=method) for A, m, method in problems]
    torch.cuda.synchronize()
    start, wrong = threading.Barrier(len(problems)), []

    def compute(h, method, B, again):
        """Calls without Python between them (ctypes lets the other threads run meanwhile): first the status that is not OK."""
        nnz, ptrs = ctypes.c_int64(), [t.data_ptr() for t in B]
        for _ in range(again):
            s = lib.spkadd_onepass(h.ptr, *ptrs, B[1].numel(), ctypes.byref(nnz)) if method == "onepass" else \
                lib.spkadd_numeric(h.ptr, *ptrs)
            if s != 0:
                return s
        return 0

    def work(q):
        A, m, method = problems[q]
        with torch.cuda.stream(torch.cuda.Stream()):
            B = [torch.empty_like(t) if method == "twopass" else
                 torch.empty(t.numel() if i == 0 else sum(a[1].numel() for a in A), dtype=t.dtype, device="cuda")
                 for i, t in enumerate(want[q])]
            for _ in range(20):
                start.wait()
                h = spk.spkadd_plan(A, m)
                try:
                    if method == "twopass":
                        spk.spkadd_symbolic(h)
                    status = compute(h, method, B, 100)
                    torch.cuda.current_stream().synchronize()
                except spk.SpkaddError as e:
                    status = str(e)
                spk.spkadd_destroy(h)
                if status != 0:
                    wrong.append((JOBS[q], status))
                elif not all(torch.equal(x[:y.numel()], y) for x, y in zip(B, want[q])):
                    wrong.append((JOBS[q], "B differs"))

    threads = [threading.Thread(target=work, args=(q,)) for q in range(len(problems))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong

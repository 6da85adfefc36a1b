"""bench.py's host logic without a GPU: the max-over-ranks reduction and
barrier on a 2-rank gloo group, the reference arm launched under torchrun
(rank 0 alone prints one JSON line), and the memory-sized wave plan of the
batched workload."""
import json
import os
import socket
import subprocess
import sys

import pytest
import torch
import torch.multiprocessing as mp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def _free_port():
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        return s.getsockname()[1]


def _rank_main(rank, world, port, out):
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port), RANK=str(rank), WORLD_SIZE=str(world),
                      LOCAL_RANK=str(rank))
    w, r, _ = bench.dist_setup()
    assert (w, r) == (world, rank)
    v = bench.reduce_max(1.5 + rank, w)
    bench.barrier(w)
    out.put((rank, v))
    import torch.distributed as dist

    dist.destroy_process_group()


def test_reduce_max_over_two_gloo_ranks():
    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    port = _free_port()
    procs = [ctx.Process(target=_rank_main, args=(r, 2, port, q)) for r in range(2)]
    for p in procs:
        p.start()
    got = sorted(q.get(timeout=120) for _ in range(2))
    for p in procs:
        p.join(timeout=60)
        assert p.exitcode == 0
    assert got == [(0, 2.5), (1, 2.5)]


def test_reference_arm_under_torchrun_prints_one_line():
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node", "2", "--master-addr",
           "127.0.0.1", "--master-port", str(_free_port()), "bench.py", "--impl", "reference", "--gpus", "2",
           "--workload", "er_k4_m1024_d8_f64int", "--steps", "1", "--warmup", "1", "--oracle-cols", "256"]
    r = subprocess.run(cmd, cwd=ROOT, capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [ln for ln in r.stdout.splitlines() if ln.startswith("{")]
    assert len(lines) == 1, r.stdout
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["n_gpus"] == 2 and d["value"] > 0
    assert d["cpu_baseline"]["kind"] == "oracle" and d["e2e"]["h2d_bytes_per_step"] == 0


def test_wave_plan_respects_the_budget_and_order():
    import synth

    params = synth.batch_instance_params(300, seed=0)
    budget = 20 * 10 ** 9
    waves = bench.plan_waves(params, budget)
    assert [q for w in waves for q in w] == list(range(300))
    for w in waves:
        used = sum(bench._instance_bytes(params[q]) for q in w)
        assert used <= budget or len(w) == 1


@pytest.mark.parametrize("m, n, mean, onepass, above, want", [
    (1 << 20, 1 << 20, 512, 0, 0, "k_warp_col<numeric>"),
    (1 << 20, 1 << 20, 512, 1, 0, "k_warp_onepass"),
    (1 << 20, 1 << 20, 100, 0, 0, "k_warp_sort and k_warp_col<numeric>"),
    (1 << 20, 1 << 20, 100, 1, 0, "k_sort_onepass"),
    (1024, 1024, 32, 0, 0, "k_warp_sort<numeric>"),
    (1024, 1024, 32, 1, 0, "k_sort_onepass"),
    ((1 << 23) + 1, 1000, 32, 0, 0, "k_warp_col<numeric>"),
    ((1 << 23) + 1, 1000, 32, 1, 0, "k_warp_onepass"),
    (1 << 20, 1 << 20, 1000, 0, 5, "spkadd_numeric: k_warp_sort, k_num_items"),
])
def test_kernel_label_follows_the_library_rules(m, n, mean, onepass, above, want):
    info = {"m": m, "n": n, "nnz_in": mean * n, "cols_cta": above, "cols_heavy": 0, "onepass": onepass}
    assert bench.kernel_label(info, "onepass" if onepass else "twopass").startswith(want)

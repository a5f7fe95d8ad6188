"""Host-side logic of the benchmark with more than one rank, on CPU: the path has no cross-GPU exchange
(every rank runs a replica), so what has to be right is the barrier / MAX-over-ranks timing, the whole-job
aggregation and that only rank 0 of the reference arm prints.  Two gloo ranks stand in for two GPUs."""
import json
import os
import socket
import subprocess
import sys

import torch
import torch.distributed as dist
import torch.multiprocessing as mp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _free_port():
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        return s.getsockname()[1]


def _rank_main(rank, world, port, out):
    sys.path.insert(0, ROOT)
    import bench
    dist.init_process_group("gloo", init_method=f"tcp://127.0.0.1:{port}", rank=rank, world_size=world)
    try:
        dist.barrier()
        local = 0.25 if rank == 0 else 0.40                  # rank 1 is the slow one
        slowest = bench.max_over_ranks(local, dist, "cpu")
        value = bench.whole_job_value(tokens_per_layer=640, layers=32, steps=5, world=world, seconds=slowest)
        out.put((rank, slowest, value))
        dist.barrier()
    finally:
        dist.destroy_process_group()


def test_max_over_ranks_and_whole_job_value_two_gloo_ranks():
    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    port = _free_port()
    procs = [ctx.Process(target=_rank_main, args=(r, 2, port, q)) for r in range(2)]
    for p in procs:
        p.start()
    got = sorted(q.get(timeout=120) for _ in procs)
    for p in procs:
        p.join(timeout=60)
        assert p.exitcode == 0
    for rank, slowest, value in got:
        assert slowest == 0.40                               # every rank reports the slowest rank's time
        assert value == 2 * 640 * 32 * 5 / 0.40              # both replicas count, divided by that time


def test_single_rank_needs_no_process_group():
    sys.path.insert(0, ROOT)
    import bench
    assert bench.max_over_ranks(0.5, None, "cpu") == 0.5
    assert bench.whole_job_value(608, 1, 3, 1, 0.5) == 608 * 3 / 0.5


def test_reference_arm_prints_on_rank_zero_only():
    cmd = [sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--workload", "C1", "--steps", "1",
           "--warmup", "0", "--gpus", "2"]
    env = dict(os.environ, WORLD_SIZE="2", MASTER_ADDR="127.0.0.1", MASTER_PORT=str(_free_port()))
    r1 = subprocess.run(cmd, env=dict(env, RANK="1", LOCAL_RANK="1"), capture_output=True, text=True, timeout=300)
    assert r1.returncode == 0 and r1.stdout.strip() == ""
    r0 = subprocess.run(cmd, env=dict(env, RANK="0", LOCAL_RANK="0"), capture_output=True, text=True, timeout=300)
    assert r0.returncode == 0
    line = json.loads(r0.stdout.strip().splitlines()[-1])
    assert line["impl"] == "reference" and line["n_gpus"] == 2 and line["value"] > 0
    assert line["cpu_baseline"]["kind"] == "oracle" and line["e2e"]["h2d_bytes_per_step"] == 0
    assert line["config"]["workload"] == "C1" and line["unit"] == "tokens/s/layer"


def test_the_result_line_is_short_enough_to_be_kept_whole():
    # with every field at its longest the line stays below the 3000 characters that are kept of the end of an output
    sys.path.insert(0, ROOT)
    import argparse
    import bench
    f, i = 12345678.901234567, 123456789012
    args = argparse.Namespace(steps=20, warmup=5, policy="keydiff", hybrid=True, proxy=32, mode="graph")
    cfg = bench.CONFIGS["C5"]
    step = dict(value=f, ms_per_step=f, ms_per_step_in_order=f, roofline_step={"frac": f})
    m = dict(step, launches_per_step=i, kernel_ms_sum=f, output_check=dict(max_abs_err=f, tolerance=f, elements=i, ok=True, sample="x" * 60),
             clocks=dict(sm_mhz=f, sm_max_mhz=f, reasons=["sw_power_cap"], samples=99, power_w_max=f),
             config=bench.config_dict(cfg, 32, args, 8, {"compress": "x" * 50, "l2": "inputs exceed L2"}),
             kv_bytes={k: i for k in ("logical_budget", "physical_allocated", "uncompressed", "blobs_incl_positions")},
             e2e=dict(value=f, unit=bench.UNIT, h2d_bytes_per_step=i, d2h_bytes_per_step=i, steps=5, ms_per_step=f),
             cpu_baseline=dict(value=f, unit=bench.UNIT, cores=16, kind="oracle", sample="x" * 70, seconds=f),
             roofline=dict({k: f for k in bench.ROOFLINE_KEYS}, timing="x" * 300), kernels={"attention": {k: f for k in "abcdefghij"}})
    line = bench.result_line(args, cfg, 1, m, {name: step for name in bench.EXTRA_WORKLOADS})
    assert len(line) < 2800 and "\n" not in line
    got = json.loads(line)
    assert got["value"] == 12345700.0 and got["gpu_launches"] == 20 * i and got["workloads"]["T4"]["roofline_step_frac"] == 12345700.0

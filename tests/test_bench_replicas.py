"""bench.py with N > 1 runs independent replicas: no collective on the data path, only the timing is
shared (max over ranks) and the throughput is the whole job's.  Checked here with two gloo ranks on CPU."""
import os
import socket
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _rank(rank, world, port, out):
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port), RANK=str(rank), WORLD_SIZE=str(world))
    sys.path.insert(0, ROOT)
    import torch.distributed as dist
    import bench
    dist.init_process_group("gloo", rank=rank, world_size=world)
    try:
        ms = bench.max_over_ranks(10.0 + 5.0 * rank, world, "cpu")      # rank 1 is the slow one
        out.put((rank, ms, bench.whole_job_images_per_s(64, world, 30, ms)))
        dist.barrier()
    finally:
        dist.destroy_process_group()


def test_two_replicas_report_the_slowest_rank_and_the_whole_job():
    import torch.multiprocessing as mp
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        port = s.getsockname()[1]
    ctx = mp.get_context("spawn")
    out = ctx.Queue()
    procs = [ctx.Process(target=_rank, args=(r, 2, port, out)) for r in range(2)]
    for p in procs:
        p.start()
    got = sorted(out.get(timeout=120) for _ in procs)
    for p in procs:
        p.join(timeout=60)
        assert p.exitcode == 0
    for rank, ms, value in got:
        assert ms == 15.0
        assert value == pytest.approx(2 * 64 * 30 / 15e-3)


def test_single_rank_needs_no_process_group():
    sys.path.insert(0, ROOT)
    import bench
    assert bench.max_over_ranks(7.5, 1, "cpu") == 7.5
    assert bench.whole_job_images_per_s(64, 1, 30, 300.0) == pytest.approx(6400.0)


def test_result_line_is_short_and_whole():
    """All of the line is within the last 1,500 characters of the output, whatever the record behind it holds."""
    import json
    sys.path.insert(0, ROOT)
    import bench
    from paper_2502_12499_b200 import workloads as wl
    big = {"per_shape": [{"shape": [64, 224, 224, 64, 64, 3, 1], "ms": 0.123456789}] * 40}
    config = {"workload": bench.workload_name(wl.config(2)), "parallelism": "single GPU", "submission": "CUDA graph replay of the recorded step",
              "l2": "inputs larger than L2 (every step streams > 1 GB of activations); single kernels rotate over buffer sets beyond the L2",
              "timing": "median of 3 regions of 30 steps"}
    record = dict(metric=bench.METRIC, value=7812.3456789012, unit=bench.UNIT, n_gpus=8, steps=30, warmup=5, ms_per_step=8.1923456789012,
                  higher_is_better=True, scaling="weak", vs_baseline=None, dtype="bf16", data="synthetic", config=config,
                  e2e=dict(value=7790.123456789, unit=bench.UNIT, h2d_bytes_per_step=19267840, d2h_bytes_per_step=12), gpu_launches=12345,
                  clocks=dict(sm_mhz=1890.0, sm_max_mhz=1965.0, reasons=["sw_power_cap", "sw_thermal_slowdown"], samples=123), peak_bytes=10 ** 10,
                  predicted_bytes=10 ** 10, recompute_overhead_pct=22.773410403630567, loss=6.9, planner_us=big,
                  roofline=dict(big, kernel="k" * 100, bound="tensor", achieved=1234.56789012, peak=1714.512345, unit="TFLOP/s", frac=0.72012345678),
                  configs={wl.config(i)["name"]: dict(big, ms_per_step=56.843123456789) for i in (2, 3, 4, 5)},
                  cpu_baseline=dict(value=0.58941223, unit=bench.UNIT, cores=16, kind="oracle", sample="s" * 200))
    line = json.dumps(bench.result_line(record))
    assert len(line) < 1450 and "\n" not in line, len(line)
    back = json.loads(line)
    assert back["value"] == pytest.approx(record["value"], rel=1e-5) and back["e2e"]["h2d_bytes_per_step"] == 19267840
    assert back["config"] == config and back["gpu_launches"] == 12345 and len(back["configs_ms"]) == 4

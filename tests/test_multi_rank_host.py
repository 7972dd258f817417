"""Host-side logic of the multi-GPU bench (N independent replicas, one layer per rank, no collective on the data
path): per-rank seeds, max-over-ranks timing and whole-job throughput, run as two gloo ranks on the CPU."""
import os
import socket
import sys
import time

import pytest
import torch
import torch.distributed as dist
import torch.multiprocessing as mp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def _free_port():
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        return s.getsockname()[1]


def _rank_main(rank, world, port, out):
    import bench
    os.environ["MASTER_ADDR"] = "127.0.0.1"
    os.environ["MASTER_PORT"] = str(port)
    dist.init_process_group("gloo", rank=rank, world_size=world)
    try:
        spec = bench.bench_spec(rank)
        my_ms = 10.0 + 5.0 * rank                       # rank 1 is the slower replica
        ms = bench.max_over_ranks(my_ms, world, "cpu")
        value = bench.aggregate_value(spec.weights, world, ms)
        out.put((rank, spec.seed, ms, value))
    finally:
        dist.destroy_process_group()


def test_two_replicas_take_the_slowest_rank_and_add_the_work():
    import bench
    world, port = 2, _free_port()
    ctx = mp.get_context("spawn")
    out = ctx.Queue()
    procs = [ctx.Process(target=_rank_main, args=(r, world, port, out)) for r in range(world)]
    for p in procs:
        p.start()
    got = sorted(out.get(timeout=120) for _ in range(world))
    for p in procs:
        p.join(timeout=60)
        assert p.exitcode == 0
    weights = bench.bench_spec(0).weights
    assert [g[1] for g in got] == [bench.bench_spec(0).seed, bench.bench_spec(0).seed + 100]   # different layers per rank
    for _, _, ms, value in got:
        assert ms == 15.0                                # the maximum over the ranks, on every rank
        assert value == world * weights / 15.0e-3


def test_reference_arm_runs_on_rank_zero_only(monkeypatch):
    import bench

    class Args:
        gpus, steps, warmup = 2, 1, 0
    monkeypatch.setenv("RANK", "1")
    assert bench.run_reference(Args()) == 0              # other ranks return at once, without work or output


def test_the_bench_line_keeps_its_keys_and_stays_short():
    """Where only the last few kilobytes of the output are kept, a line with the per-layer tables cannot be read back."""
    import json
    import bench
    x = 123456.78901234567
    kernel = {"bound": "alu", "achieved": x, "peak": x, "unit": "TFLOP/s", "frac": x, "ms_per_step": x,
              "launches_per_step": 2, "peak_source": "p" * 140}
    layer = {"layer": "c3.layer4.0.downsample", "ms": x, "stages_ms": {k: x for k in "abcdef"}, "roofline_frac": {"a": x}}
    one_set = {"n_layers": 54, "weights": 25502912, "total_ms": x, "weights_per_s": x, "graph_total_ms": x,
               "overlapped_8_streams_cta_limited_ms": x, "layers": [layer] * 54, "stage_total_ms": {k: x for k in "abcdef"}}
    report = {
        "metric": bench.METRIC, "value": x, "unit": bench.UNIT, "n_gpus": 8, "steps": 100, "warmup": 3, "ms_per_step": x,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": bench.workload_config(bench.bench_spec(), 8),
        "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": ["hw_slowdown", "sw_power_cap"], "samples": 100},
        "e2e": {"value": x, "unit": bench.UNIT, "h2d_bytes_per_step": 40108032, "d2h_bytes_per_step": 589832,
                "ms_per_step": x},
        "gpu_launches": 2000,
        "roofline": dict(kernel, kernel="gram_i8_tcgen05", traffic=x, launch_ms=x, algorithmic_work_per_launch=x,
                         sweep_ns_per_column=x, per_kernel={f"kernel{i}": kernel for i in range(8)}),
        "cpu_baseline": {"value": x, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 60,
                         "codes_equal_to_gpu": True, "order_equal_to_gpu": True},
        "stages_ms": {k: x for k in ("hessian", "inverse", "grid", "order", "sweep")},
        "kernels": {f"kernel{i}": {"ms_per_step": x, "launches_per_step": 2} for i in range(20)},
        "fp64_peak": {"dfma_tflops": x, "dmma_tflops": x, "fp64_tflops": x},
        "layer_sets": {f"c{i}_resnet50_w4": one_set for i in range(4)}, "context": "c" * 90}
    line = bench.bench_line(report)
    assert len(line) <= bench.LINE_LIMIT
    got = json.loads(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "roofline", "cpu_baseline"):
        assert key in got, key
    assert got["value"] == x and got["ms_per_step"] == x and got["e2e"] == report["e2e"] and got["config"] == report["config"]
    assert "layer_sets_ms" in got and "per_kernel" not in got["roofline"]
    report["roofline"]["peak_source"] = "p" * 500
    assert len(bench.bench_line(report)) <= bench.LINE_LIMIT


@pytest.mark.parametrize("region", [0.3, 0.0])
def test_clocks_are_sampled_however_late_the_first_line_and_however_short_the_region(tmp_path, monkeypatch, region):
    """A stand-in for nvidia-smi that prints its first line after 0.4 s and another one every 50 ms, idle clocks first."""
    tool = tmp_path / "nvidia-smi"
    tool.write_text("#!/bin/bash\nsleep 0.4\nmhz=345\nwhile true; do\n"
                    "echo \"0, $mhz, 1965, 100.0, 0x0, Not Active, Not Active, Not Active, Active\"\nsleep 0.05; mhz=1900\ndone\n")
    tool.chmod(0o755)
    monkeypatch.setenv("PATH", f"{tmp_path}:{os.environ['PATH']}")
    import bench
    sampler = bench.ClockSampler(0)
    sampler.start()
    time.sleep(0.3)                     # the warm-up
    sampler.mark()
    time.sleep(region)
    out = sampler.stop()
    assert out["samples"] >= 1 and out["sm_mhz"] == 1900.0 and out["sm_max_mhz"] == 1965.0
    assert out["reasons"] == ["sw_power_cap"]

"""Host logic of the multi-GPU benchmark path, on CPU with two gloo ranks.

The decoding path shards by series with no exchange step: every rank decodes its own batch.
What the ranks share is bookkeeping only -- distinct series per rank, the max-over-ranks time,
the whole-job throughput, and the rule that the CPU-reference arm runs on rank 0 alone."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest
import torch
import torch.distributed as dist
import torch.multiprocessing as mp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def _worker(rank, world, port, out_dir):
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port), RANK=str(rank), WORLD_SIZE=str(world))
    dist.init_process_group("gloo", rank=rank, world_size=world)
    import bench
    from tsfm_inputs import make_series, workload
    wl = bench.rank_workload(workload("C0", batch=3, series_recipe="c1"), rank)
    s = make_series(wl)
    ms = bench.max_over_ranks(10.0 + 5.0 * rank, world, device="cpu")       # rank 1 is the slow one
    value = bench.whole_job_value(world, wl.batch, wl.n_patches, 4, ms)
    json.dump({"ms": ms, "value": value, "checksum": float(np.abs(s).sum()), "first": s[0, :4].tolist()},
              open(os.path.join(out_dir, f"r{rank}.json"), "w"))
    dist.barrier()
    dist.destroy_process_group()


def test_two_ranks_decode_different_series_and_agree_on_the_job_time(tmp_path):
    world, port = 2, 29500 + os.getpid() % 2000
    mp.spawn(_worker, args=(world, port, str(tmp_path)), nprocs=world, join=True)
    r = [json.load(open(tmp_path / f"r{i}.json")) for i in range(world)]
    assert r[0]["ms"] == r[1]["ms"] == 15.0                       # max over ranks, seen by both
    assert r[0]["value"] == r[1]["value"] == 2 * 3 * 4 * 4 / 15e-3    # all ranks' patches / slowest time
    assert r[0]["first"] != r[1]["first"]                          # each rank has its own series


def test_reference_arm_runs_on_rank_zero_only():
    env = dict(os.environ, RANK="1", WORLD_SIZE="2", LOCAL_RANK="1")
    res = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--workload", "C0",
                          "--steps", "1", "--warmup", "0", "--gpus", "2"], env=env, capture_output=True, text=True,
                         timeout=300)
    assert res.returncode == 0 and res.stdout.strip() == ""
    env["RANK"] = "0"
    res = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--workload", "C0",
                          "--steps", "1", "--warmup", "0", "--gpus", "2"], env=env, capture_output=True, text=True,
                         timeout=300)
    line = json.loads(res.stdout.strip().splitlines()[-1])
    assert line["impl"] == "reference" and line["cpu_baseline"]["kind"] == "oracle" and line["value"] > 0
    assert line["e2e"]["h2d_bytes_per_step"] == 0 and line["n_gpus"] == 2


def test_result_line_is_short_and_strict_json():
    """The headline survives a reader that keeps the last 3000 characters, whatever else was measured."""
    import bench
    from tsfm_inputs import workload
    nan = float("nan")
    kernel = {k: 1 / 3 for k in ("share", "launches_per_step", "ms_per_step", "GB/s", "frac_hbm")}
    m = {"ms_per_step": 12.3456789012345, "target_only": {"ms_per_step": 2 / 3}, "speedup_vs_target_only": nan,
         "phases_ms": {f"ms_{p}": 1 / 3 for p in ("prefill", "draft", "verify", "accept")}, "kernels": {f"kernel_{i}": kernel for i in range(12)},
         "roofline": dict.fromkeys(bench.ROOFLINE_KEYS, 1 / 3), "mse_vs_truth": {"speculative": nan}}
    wl = workload("C4")
    r = dict(m, metric=bench.METRIC, value=123456.789012345, unit=bench.UNIT, n_gpus=1, steps=20, warmup=5, higher_is_better=True,
             scaling="weak", vs_baseline=None, dtype="bf16", data="synthetic", config=bench.bench_config(wl, wl.K, wl.tau),
             e2e={"value": 1 / 3, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2}, gpu_launches=12345,
             clocks={"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": ["sw_power_cap"], "samples": 99},
             cpu_baseline={"value": 1 / 3, "unit": bench.UNIT, "cores": 64, "kind": "oracle", "sample": "x" * 400},
             workloads={n: dict(m) for n, _, _, _ in bench.other_workloads(["C2", "C1", "C3", "C5"])} | {"bad": {"error": "e" * 500}})
    line = bench.result_line(r)
    assert len(line) < 3000 and "\n" not in line
    back = json.loads(line, parse_constant=lambda c: pytest.fail(f"not strict JSON: {c}"))
    assert back["value"] == r["value"] and back["ms_per_step"] == r["ms_per_step"] and set(bench.LINE_KEYS) <= set(back)

"""The N > 1 path on CPU: the benchmark's replicas share nothing but the clock, so what there is to test
is the max-over-ranks reduction (gloo, world size 2) and that the reference arm under torchrun prints
exactly one line, from rank 0."""
import json
import os
import subprocess
import sys

import torch
import torch.distributed as dist
import torch.multiprocessing as mp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _worker(rank, world, port, out):
    sys.path.insert(0, ROOT)
    import bench
    os.environ["MASTER_ADDR"] = "127.0.0.1"
    os.environ["MASTER_PORT"] = str(port)
    dist.init_process_group("gloo", rank=rank, world_size=world)
    try:
        slowest = bench.reduce_max_over_ranks(10.0 + 5.0 * rank, world)
        dist.barrier()
        out[rank] = (slowest, bench.aggregate_value(2.0e9, world, slowest))
    finally:
        dist.destroy_process_group()


def test_max_over_ranks_and_aggregate_gloo():
    world = 2
    with mp.Manager() as m:
        out = m.dict()
        mp.spawn(_worker, args=(world, 29541, out), nprocs=world, join=True)
        res = dict(out)
    assert res[0] == res[1]
    slowest, value = res[0]
    assert slowest == 15.0                                  # the slower replica sets the clock
    assert abs(value - 2 * 2.0e9 / 15.0e-3 / 1e9) < 1e-9     # both replicas' work over that time


def test_reference_arm_under_torchrun_prints_one_line():
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node", "2", "--master-addr", "127.0.0.1",
           "--master-port", "29543", os.path.join(ROOT, "bench.py"), "--impl", "reference", "--gpus", "2", "--steps", "1",
           "--warmup", "0"]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [ln for ln in r.stdout.splitlines() if ln.startswith("{")]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["n_gpus"] == 2 and d["e2e"]["h2d_bytes_per_step"] == 0
    assert d["cpu_baseline"]["kind"] == "oracle" and d["value"] > 0


def test_headline_is_short_whatever_the_tables():
    """The line on stdout holds the metric, the end-to-end figure, clocks, roofline and CPU baseline in under 1500 characters; tables of any
    length are the other part."""
    import json

    import bench

    third, long = 1000.0 / 3.0, [{"layer": "wrn_s1_32@32", "ms": 1.0 / 3.0}] * 500
    line = {"metric": bench.METRIC, "value": third * 1e3, "unit": bench.UNIT, "n_gpus": 8, "steps": 20, "warmup": 5, "ms_per_step": third, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32+tf32", "data": "synthetic",
            "config": {"workload": bench.WORKLOAD, "layers_per_step": 90, "batch": 128, "groups": [1, 2, 4, 8, 16], "parallelism": "replicas only (8)",
                       "launch": "cuda graph of the step", "l2": "every layer instance owns its x/y buffers: 1.82 GB cycled per step > 126 MB L2"},
            "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": ["sw_power_cap"], "samples": 17},
            "e2e": {"value": third, "unit": bench.UNIT, "ms_per_step": third, "h2d_bytes_per_step": 943718400, "d2h_bytes_per_step": 880803840, "steps": 10},
            "two_streams": {"ms_per_step": third, "value": third, "unit": bench.UNIT, "how": "x" * 300}, "gpu_launches": 1800, "layers": long,
            "cpu_baseline": {"value": third, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "seconds": third, "sample": "x" * 300},
            "roofline": {"bound": "hbm", "achieved": third, "peak": third, "unit": "GB/s", "frac": third, "traffic": 1.0 / 3.0, "kernel": "igemm_tf32", "peak_source": "x" * 99},
            "sweep_layers": long, "targets": long}
    short, tables = bench.headline(line)
    text = json.dumps(short)
    assert len(text) < 1500 and "\n" not in text, len(text)
    assert set(bench.HEADLINE_KEYS) | {"roofline", "cpu_baseline"} <= set(short) and abs(short["value"] / line["value"] - 1.0) < 1e-6
    assert tables["layers"] == long and tables["sweep_layers"] == long and "value" not in tables
    for missing in ("roofline", "cpu_baseline", "two_streams"):
        line.pop(missing)
    assert "roofline" not in bench.headline(line)[0]

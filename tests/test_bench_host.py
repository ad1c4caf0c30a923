"""Host-side logic of bench.py that needs no GPU: multi-rank aggregation under gloo (world size 2), and the
CPU reference arm's JSON contract."""
import json
import os
import subprocess
import sys

import torch.distributed as dist
import torch.multiprocessing as mp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def _worker(rank, world, port, out):
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port), RANK=str(rank), WORLD_SIZE=str(world))
    import bench
    dist.init_process_group("gloo", rank=rank, world_size=world)
    times = [1.0 + rank, 5.0 - rank, 2.5]                      # rank 0: 1, 5, 2.5 ; rank 1: 2, 4, 2.5
    got = bench.max_over_ranks(times, dist, "cpu")
    dist.barrier()
    if rank == 0:
        json.dump({"max": got, "value": bench.job_throughput(world, 1e9, got[0])}, open(out, "w"))
    dist.destroy_process_group()


def test_max_over_ranks_and_job_value_gloo(tmp_path):
    out = str(tmp_path / "r.json")
    mp.spawn(_worker, args=(2, 29000 + os.getpid() % 2000, out), nprocs=2, join=True)
    r = json.load(open(out))
    assert r["max"] == [2.0, 5.0, 2.5]                          # slowest rank per timer
    assert r["value"] == 2 * 1e9 / (2.0e-3) / 1e9               # all ranks' bytes over the slowest rank's time


def test_single_process_is_identity():
    import bench
    assert bench.max_over_ranks([3.0, 1.0]) == [3.0, 1.0]
    assert bench.job_throughput(1, 234881024, 0.04) == 234881024 / 0.04e-3 / 1e9


def test_reference_arm_prints_contract_line_and_other_ranks_stay_silent():
    env = dict(os.environ, RANK="0", WORLD_SIZE="1")
    p = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1", "--warmup", "3"],
                       capture_output=True, text=True, env=env, timeout=600)
    assert p.returncode == 0, p.stderr
    line = json.loads(p.stdout.strip().splitlines()[-1])
    assert line["impl"] == "reference" and line["metric"] == "hif8_encode_decode_throughput" and line["unit"] == "GB/s"
    assert line["cpu_baseline"]["kind"] == "oracle" and line["cpu_baseline"]["cores"] >= 1
    assert line["e2e"]["h2d_bytes_per_step"] == 0 and line["e2e"]["value"] == line["value"] > 0
    env1 = dict(os.environ, RANK="1", WORLD_SIZE="2")
    p = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1"],
                       capture_output=True, text=True, env=env1, timeout=600)
    assert p.returncode == 0 and p.stdout.strip() == ""


def test_headline_is_short_and_whole():
    """Standard output carries the contract's keys in a line that a bounded tail of a log holds; tables of any size stay out."""
    import bench
    table = {f"workload_{i}": {"ms": 1.0 / 3.0, "note": "x" * 200} for i in range(100)}
    text = "x" * 130
    line = {"metric": bench.METRIC, "value": 7000.0 / 3, "unit": "GB/s", "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": 0.1 / 3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u8", "data": "synthetic",
            "config": dict({k: text for k in bench.HEADLINE_CONFIG}, step_dram=table),
            "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965, "reasons": ["sw_power_cap"], "samples": 100},
            "e2e": {"value": 100.0 / 3, "unit": "GB/s", "ms_per_step": 1.7 / 3, "h2d_bytes_per_step": 1 << 26, "d2h_bytes_per_step": 5 << 24},
            "gpu_launches": 80, "roofline": dict({k: 1.0 / 3 for k in bench.HEADLINE_ROOFLINE}, by_config=table),
            "cpu_baseline": {"value": 0.07, "unit": "GB/s", "cores": 16, "kind": "oracle", "sample": text, "elements_per_s": 1e7 / 3, "legs": table},
            "kernels": table, "calls": table, "extra": table, "sharded": table}
    short = bench.headline(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype",
                "data", "clocks", "e2e", "gpu_launches"):
        assert short[key] == line[key]
    assert short["cpu_baseline"]["value"] == 0.07 and short["config"]["workload"] == text and len(json.dumps(short)) < 3800

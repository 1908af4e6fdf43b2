"""Host-side logic of bench.py: cost model, rank reduction (gloo, 2 processes), reference arm."""
import json
import os
import subprocess
import sys

import pytest
import torch
import torch.distributed as dist
import torch.multiprocessing as mp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402
from paper_2403_03507_b200 import workloads as wl  # noqa: E402


def test_algorithmic_cost_matches_hand_computation():
    # 4096 x 11008 bf16, r = 1024, 8-bit states: G + 2 W + 4 bytes per state element + absmax + P
    w = wl.WORKLOADS["llama_7b_q8"]
    by, fl = bench.algorithmic_cost(w, 4096, 11008)
    nel = 1024 * 11008
    assert by == 4096 * 11008 * 2 * 3 + 4 * nel + 16 * (nel // 2048) + 4096 * 1024 * 2
    assert fl == 4 * 4096 * 11008 * 1024
    # whole layer sets: parameters as listed for the workloads
    assert w.params == 6_476_005_376 and w.matrices == 224
    assert wl.WORKLOADS["llama_1b_q8"].params == 1_207_910_400
    assert wl.WORKLOADS["llama_130m"].params == 84_934_656
    total_flops = sum(bench.algorithmic_cost(w, m, n)[1] * c for m, n, c in w.shapes)
    assert abs(total_flops / 26.53e12 - 1) < 1e-3
    total_bytes = sum(bench.algorithmic_cost(w, m, n)[0] * c for m, n, c in w.shapes)
    assert abs(total_bytes / 47.22e9 - 1) < 5e-3


def _rank_main(rank, world, port, out):
    os.environ["MASTER_ADDR"] = "127.0.0.1"
    os.environ["MASTER_PORT"] = str(port)
    dist.init_process_group("gloo", rank=rank, world_size=world)
    try:
        got = bench.max_over_ranks(10.0 + 5.0 * rank, dist, torch.device("cpu"))
        out[rank] = got
    finally:
        dist.destroy_process_group()


def test_timing_is_the_maximum_over_ranks_gloo_world_size_2():
    mgr = mp.Manager()
    out = mgr.dict()
    mp.spawn(_rank_main, args=(2, 29533, out), nprocs=2, join=True)
    assert out[0] == 15.0 and out[1] == 15.0
    assert bench.max_over_ranks(3.5, None, None) == 3.5


def test_reference_arm_prints_one_json_line_and_other_ranks_stay_silent():
    cmd = [sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--workload", "single_60m_mlp",
           "--steps", "1", "--warmup", "0"]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0, r.stderr
    lines = [l for l in r.stdout.splitlines() if l.strip()]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["unit"] == "params/s" and d["value"] > 0
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] >= 1
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["d2h_bytes_per_step"] == 0
    env = dict(os.environ, RANK="1", WORLD_SIZE="2", LOCAL_RANK="1")
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=300, cwd=ROOT, env=env)
    assert r.returncode == 0 and r.stdout.strip() == ""


def test_clock_sampler_tolerates_a_missing_nvidia_smi():
    s = bench.ClockSampler(0)
    s.start()
    res = s.stop()
    assert set(res) >= {"sm_mhz", "sm_max_mhz", "reasons"}


def test_the_printed_line_keeps_the_figures_and_stays_short():
    """A line of every workload's full record was cut off by its readers."""
    phase = {"ms_per_step": 13.066239953041076, "launches_per_step": 1.0, "tflops": 1413.4410082145796, "gbs": 818.5579966722333,
             "roof_ms": 0.133789911422776, "frac_of_own_roof": 1.0239358216564616}
    refresh = [{"shape": [4096, 11008], "count": 64, "ms": 128.64598083496094, "iterations": 18, "residual": 6.749436290840305e-06}] * 3
    config = {"workload": "llama_7b_q8", "rank": 1024, "state_fmt": "q8", "l2": "inputs larger than L2 (whole layer set streamed each step)"}
    gaps = {str(t): 43726525071.28677 for t in (50, 200, 1000)}
    record = {"metric": bench.METRIC, "value": 226123456789.12345, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
              "ms_per_step": 28.612345678901234, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
              "data": "synthetic", "config": config, "clocks": {"sm_mhz": 1507.0, "sm_max_mhz": 1965.0, "reasons": ["sw_power_cap"], "samples": 6},
              "gpu_launches": 420, "roofline": {"bound": "tensor", "frac": 0.6904188076514539, "kernels": {k: phase for k in "abc"},
                                                "traffic": {k: 3645065883.062857 for k in "abc"}, "refresh_amortised": {"by_gap": gaps}},
              "refresh": refresh, "refresh_set": {"ms": 6000.0}, "refresh_amortised": {"by_gap": gaps},
              "e2e": {"value": 11544679720.197325, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2}, "device_status": 0}
    record["other_workloads"] = [{k: record[k] for k in ("value", "ms_per_step", "config", "roofline", "refresh", "clocks")} for _ in range(16)]
    line = json.dumps(bench.summary(record))
    assert len(line) < 5000 < len(json.dumps(record))
    got = json.loads(line)
    for key in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "clocks",
                "gpu_launches"):
        assert got[key] == record[key]
    assert abs(got["value"] / record["value"] - 1) < 1e-6 and abs(got["ms_per_step"] / record["ms_per_step"] - 1) < 1e-6
    assert got["e2e"]["h2d_bytes_per_step"] == 1 and len(got["other_workloads"]) == 16

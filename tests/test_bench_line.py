"""The line that bench.py prints is short enough for a log that keeps the last 3,000 characters, and
complete: every key of the headline, the end-to-end figure, clocks and roofline."""
import copy
import json
import os

import bench

RECORD = os.path.join(bench.ROOT, "results", "bench_cavity2048_fp32_with_ablation.json")


def test_line_of_the_recorded_run():
    rec = json.load(open(RECORD))
    rec["ttr_summary"]["oracle_extrap_s"] = 2824.0
    before = copy.deepcopy(rec)
    line = bench.bench_line(rec)
    assert rec == before
    assert len(json.dumps(line)) <= 2900
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
              "dtype", "data", "gpu_launches", "clocks", "last_residual", "ttr_summary"):
        assert line[k] == rec[k], k
    for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][k] == rec["e2e"][k]
    for k in ("workload", "nx", "ny", "velocities", "l2", "parallelism"):
        assert line["config"][k] == rec["config"][k]
    assert line["roofline"]["bound"] == "hbm" and line["cpu_baseline"]["kind"] == "oracle"
    assert len(line["configs_s"]) == len(rec["configs_time_to_residual"])


def test_line_of_a_run_without_extras():
    rec = json.load(open(RECORD))
    for k in ("e2e", "fp64", "second_order", "time_to_residual", "cpu_baseline", "configs_time_to_residual", "ttr_summary"):
        rec.pop(k)
    line = bench.bench_line(rec)
    assert line["value"] == rec["value"] and "e2e" not in line and "fp64" not in line

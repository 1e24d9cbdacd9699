"""The benchmark's result line stays short: details of a run (the other forms, rooflines, step times)
go to stderr, so that the line fits readers that keep the last 1500 characters of the output."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_result_line_is_short_and_complete():
    sys.path.insert(0, ROOT)
    import bench
    number = 1176.388619265555
    config = {"workload": "l32_batch_48t_6noise", "L": 32, "X": 32768, "n_ev": 128,
              "ndil": [32, 48, 64, 32, 32, 64], "n_t": 48, "n_noise": 6, "n_mom": 9, "n_spin": 4,
              "spin_pairs": 4, "form": "fp16x3", "jobs_per_step_per_gpu": 288,
              "blocks_per_step_per_gpu": 2592,
              "tiles": {"nc": 16, "chunk": 2, "source": "cost-model top 3 timed"},
              "timed_steps": "x" * 110, "l2": "x" * 70, "parallelism": "x" * 40}
    line = {"metric": bench.METRIC, "value": number, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": number, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "fp16", "data": "synthetic (seeded, workloads.py)", "config": config, "gpu_launches": 100,
            "e2e": {"value": number, "unit": bench.UNIT, "steps": 3, "h2d_bytes_per_step": 9984540672,
                    "d2h_bytes_per_step": 5067767808, "path": "x" * 150},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "power_w_median": 893.6, "samples": 58, "reasons": []},
            "speedup_vs_fp64_form": number, "roofline": {"x": ["y" * 700]}, "forms": {"x": ["y" * 6000]}}
    result, detail = bench.result_and_detail(line)
    assert len(json.dumps(result)) <= 1450
    assert set(line) - set(result) == {"roofline", "forms"} == set(detail["detail"])
    assert all(result[k] == line[k] for k in result)

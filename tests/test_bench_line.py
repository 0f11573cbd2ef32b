"""CPU: the bench's line on stdout carries the main workload's keys whole and stays short, however much the side legs
record."""
import json

import bench

REQUIRED = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "roofline", "cpu_baseline", "e2e", "gpu_launches", "clocks")


class Args:
    iters, precision, gpus = 10, "fp32", 1


def _record():
    x = 1234.567890123456789
    many = [{"n": 8192, "ms": x, "gbs_algorithmic": x, "note": "y" * 80} for _ in range(60)]
    return {"metric": bench.METRIC, "value": x, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": x,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": bench._config(Args()),
            "roofline": {"bound": "hbm", "achieved": x, "peak": x, "unit": "GB/s", "frac": x, "traffic": None,
                         "traffic_last_capture": {"bytes_per_launch": x, "workload": "w" * 60, "note": "n" * 200},
                         "kernel": "rows_pass2", "algorithmic_bytes_per_launch": 10 ** 9, "avg_launch_ms": x,
                         "peak_source": "measured copy bandwidth", "share_of_kernel_time": x},
            "cpu_baseline": {"value": x, "unit": bench.UNIT, "cores": 14, "kind": "oracle", "sample": "s" * 900},
            "e2e": {"value": x, "unit": bench.UNIT, "h2d_bytes_per_step": 2 ** 28, "d2h_bytes_per_step": 2 ** 28, "steps": 2},
            "gpu_launches": 4321, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 40},
            "fixed_iteration_note": "z" * 200, "iters_per_stage": [10, 10, 10], "final_residual": x,
            "hbm_frac_step_algorithmic": x, "ms_per_step_graph_mode": x,
            "fp32_vs_fp64": {"fp32_ms_per_step": x, "fp64_ms_per_step": x, "steps": 2, "speedup_fp32": x, "max_abs_diff": x,
                             "max_rel_diff_v": x},
            "ch2d8192_crop1024_err_vs_oracle": {"fp32": x, "fp64": x},
            "batched": {"ms_per_step": x, "schedule": many}, "sweep_microbench": many, "autotune": many, "kernels": many,
            "vector_ch": {"fp32": {"ms_per_step": x, "kernels": many}}, "split3d": {"error": "RuntimeError: " + "e" * 300},
            "fch1d": None, "fch2d": {"fp32": {"ms_per_step": x}}}


def test_line_is_short_and_whole():
    res = _record()
    text = bench.headline(res)
    assert "\n" not in text and len(text) <= bench.HEADLINE_BYTES < 3000
    line = json.loads(text)
    for key in REQUIRED:
        assert key in line, key
    assert line["value"] > 0 and abs(line["value"] / res["value"] - 1) < 1e-5
    assert line["e2e"]["h2d_bytes_per_step"] == 2 ** 28 and line["config"]["workload"] == bench.WORKLOAD["name"]
    assert line["cpu_baseline"]["value"] > 0 and line["roofline"]["kernel"] == "rows_pass2"
    # one figure of every leg that ran; a failed or skipped leg has none
    assert set(line["legs"]) == {"batched_ms", "vector_ch_ms", "fch2d_ms"}
    assert res == _record()


def test_line_without_side_legs():
    res = {k: v for k, v in _record().items() if k in REQUIRED}
    assert "legs" not in json.loads(bench.headline(res))

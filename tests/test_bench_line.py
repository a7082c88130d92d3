"""The benchmark's line on standard output: every field that its readers need,
and short enough for one that keeps the last 3 000 characters, however long the
record's curves and per-frame rows are."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def _record():
    x = 0.123456789012345678
    rows = [{"frame": i, **{k: x for k in "abcdefghij"}} for i in range(300)]
    stages = ("ntc_fwd", "project", "bin_sort", "raster_fwd", "loss", "raster_bwd", "project_bwd", "ntc_bwd", "adam")
    return {"metric": bench.METRIC, "value": x, "unit": "s/frame", "n_gpus": 1, "steps": 150, "warmup": 5,
            "ms_per_step": x, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
            "dtype": "mixed: f16 table, bf16 mlp, f32 raster", "data": "synthetic",
            "config": {"workload": "w" * 110, **{"key_%d" % i: 1352 for i in range(12)}, "l2": "l" * 40},
            "train_it_per_s": x, "full_frame_s": x, "raster_fwd_bwd_it_per_s": x, "raster_fwd_bwd_ms": x,
            "plain_fp32_direct_opt": {"ms_per_iter": x}, "speedup_vs_plain_per_iter": x,
            "equal_psnr": {"speedup_at_equal_psnr": x, "ntc": {"curve": rows}, "direct": {"curve": rows}},
            "graphs": True, "stages_ms": {k: 0.1234 for k in stages}, "bin_pairs_per_step": 10 ** 8,
            "composited_pairs": [10 ** 9] * 4, "warmup_loss": x, "warmup_s": x,
            "roofline": {"bound": "alu", "kernel": "raster_bwd", "achieved": x, "peak": x, "unit": "TFLOP/s", "frac": x,
                         "traffic": 10 ** 9, "algorithmic_flops": 10 ** 11, "pairs_evaluated": 10 ** 9,
                         "pairs_added": 10 ** 9, "ms": x, "sm_count": 152, "peak_source": "s" * 90},
            "raster_fwd_bwd_roofline": {"x": "y" * 300}, "mlp_roofline": {"x": "y" * 500},
            "render_only": {"fps": x, "autotune_ms": rows}, "bin_autotune": {"x": rows}, "bin_tiles": 4,
            "stage2": {"ms_per_iter": x, "workload": "w" * 100}, "stream": {"s_per_frame": x, "per_frame": rows},
            "large": {"ms_per_iter": x, "workload": "w" * 100}, "paper_context": {"note": "n" * 100},
            "cpu_baseline": {"value": x, "unit": "s/frame", "cores": 16, "kind": "oracle", "sample": "s" * 150,
                             "other_workloads": {"x": rows}},
            "e2e": {"value": x, "unit": "s/frame", "h2d_bytes_per_step": 10 ** 8, "d2h_bytes_per_step": 4},
            "gpu_launches": 3000, "tc_timeouts": 0,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 100}}


def test_line_is_whole_and_short():
    record = _record()
    line = bench.headline(record)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline"):
        assert line[k] == record[k]
    assert line["stream"] == {"s_per_frame": record["stream"]["s_per_frame"]}
    text = json.dumps(line)
    assert "\n" not in text and len(text) <= 2700


def test_line_without_the_side_workloads():
    record = _record()
    for k in ("equal_psnr", "render_only", "stage2", "stream", "large", "cpu_baseline", "speedup_vs_plain_per_iter"):
        record[k] = None
    line = bench.headline(record)
    assert line["stream"] is None and line["cpu_baseline"] is None and line["value"] == record["value"]

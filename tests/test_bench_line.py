"""bench.py's line on stdout: a summary that a log reader keeps whole, with the headline's numbers
untouched. CPU only, on a record of the size that a full run makes."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

KERNEL = {"kernel": "tma", "kp": 3, "warps": 8, "tile": [96, 48], "fp16": False, "form": "fp32", "loop": "block",
          "ctas_per_sm": 2, "tuned_us": 87.96800231933594}


def _record():
    stage = {"chosen": KERNEL, "candidates": [KERNEL] * 8}
    choice = {"tuned": True, "stages": [stage, stage], "batches": {"launched": 100, "max_in_flight": 1}, "graphs": 2}
    names = ["prep_compose_clear", "motion_mask", "motion_dilate", "motion_erode", "project_zbuf", "occlusion", "pool3",
             "jbf_stage1", "bp_rows", "jbf_stage2", "contour", "bp_count", "bp_write"]
    kernels = {k: {"total_us": 1234.5678901234567, "launches": 10, "avg_us": 123.456789012} for k in names}
    path = {"ideal_us_per_step": 123.45, "measured_us_per_step": 234.56, "frac": 0.526, "basis": "b" * 150,
            "kernels": {k: {"roof_us": 1.23, "measured_us": 2.34, "frac": 0.5} for k in names}}
    view = {"view": "1920x1080", "valid_mask_exact": True, "mask_differences_px": 0, "max_abs_m": 1.23456789e-6,
            "p99_abs_m": 1.2e-7, "max_rel": 4.96e-7, "pixels_over_bar": 0}
    cpu = {"value": 45.6789012345, "unit": "frames/s", "cores": 16, "kind": "oracle", "sample": "s" * 120}
    config = {"config": {"workload": "w" * 200}, "value": 12345.678901234, "unit": "frames/s", "ms_per_step": 0.27,
              "latency_ms_per_step": {"p50": 0.27, "max": 0.28}, "gpu_launches": 160, "kernels": kernels,
              "path_roofline": path, "filter_kernels": choice,
              "cpu_baseline": dict(cpu, error_vs_oracle=dict(view, all_masks_exact=True, per_view=[view] * 12))}
    run = {"offered_frames": 127829, "completed_frames": 127829, "frames_per_s": 49383.31863738978,
           "latency_ms": {q: 292.8694897361821 for q in ("p50", "p90", "p99", "max")}, "e_again_retries": 32975,
           "buffer_waits": 12, "batches": {"launched": 74572, "max_in_flight": 2}}
    return {
        "metric": bench.METRIC, "value": 29412.345678901234, "unit": "frames/s", "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 0.27199123456789, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic", "config": {"workload": "1080p_3scan_two_stage", "note": "c" * 350},
        "latency_ms_per_step": {"p50": 0.271, "p99": 0.28},
        "roofline": {"kernel": "jbf_stage2", "bound": "alu", "achieved": 2100.123456, "peak": 9157.1, "unit": "Gtap/s",
                     "frac": 0.229, "traffic": None, "traffic_unit": "t" * 60, "peak_basis": "p" * 200,
                     "peak_live": {"taps_per_s": 9.1e12, "binds": "issue", "bounds_taps_per_sm_clk": {"issue": 29.1}},
                     "taps_per_launch": 1, "avg_launch_us": 117.5},
        "kernels": kernels, "path_roofline": path, "kernels_how": "h" * 120, "filter_kernels": choice,
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 12}, "gpu_launches": 120,
        "e2e": {"value": 6612.3456789, "unit": "frames/s", "h2d_bytes_per_step": 85620012,
                "d2h_bytes_per_step": 198560112, "what": "w" * 90,
                "host_link": {"h2d_GBps": 200.1, "d2h_GBps": 193.2, "both_GBps": 250.0, "bound_frames_per_s": 7780.1,
                              "serial_frames_per_s": 5000.1, "duplex_frames_per_s": 7000.1, "note": "n" * 350}},
        "cpu_baseline": cpu, "fp16": dict(config, precision="p" * 100, jbf_stage2_avg_us=96.123456789),
        "configs": {f"workload_with_a_long_name_{i}": config for i in range(5)},
        "serving": dict({"viewpoints": "v" * 50, "paper_rate_seconds": 60.0, "note": "n" * 250},
                        **{f"mode{i}/load{j}_of_a_thousand": run for i in range(3) for j in range(3)}),
    }


def test_line_is_short_and_keeps_the_headline():
    out = _record()
    assert len(json.dumps(out)) > 20000
    text = json.dumps(bench.compact_line(out))
    assert len(text) < 8000 and "\n" not in text
    line = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "clocks", "gpu_launches"):
        assert line[k] == out[k], k
    for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][k] == (bench._sig(out["e2e"][k])), k
    assert line["cpu_baseline"]["kind"] == "oracle" and line["cpu_baseline"]["cores"] == 16
    assert line["serving"]["mode0/load0_of_a_thousand"]["e_again_retries"] == 32975
    assert line["configs"]["workload_with_a_long_name_0"]["error_vs_oracle"]["all_masks_exact"] is True
    assert set(line["kernels_us"]) == set(out["kernels"])


def test_parts_that_a_run_skips_stay_null():
    out = dict(_record(), e2e=None, cpu_baseline=None, fp16=None, configs=None, serving=None)
    line = json.loads(json.dumps(bench.compact_line(out)))
    assert all(line[k] is None for k in ("e2e", "cpu_baseline", "fp16", "configs", "serving"))

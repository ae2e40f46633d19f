"""bench.py's default line: the standard keys, short enough for a reader that
keeps the last 3,000 characters of a run's output."""
import json

import bench


def _full_line():
    kernels = {k: {"ms_per_launch": 1.234567890123, "launches": 20} for k in ("k_dual", "k_primal", "k_accumulate")}
    form = {"ms_per_step": 12.34567890123, "value": 1.23456789e10, "unit": bench.METRIC,
            "kernels": {f"kernel_{i}": 1.2345678901 for i in range(8)}}
    other = {"metric": bench.METRIC, "value": 34567890.123456, "unit": bench.METRIC, "ms_per_step": 1.9191919191,
             "e2e": {"value": 29123456.789}, "roofline": {"frac": 0.123456789, "achieved": 1.0},
             "variants": {"x" * 50: "y" * 5000}}
    return {
        "metric": bench.METRIC, "value": 12743210987.654321, "unit": bench.METRIC, "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 10.531234567, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "u32+f32 (dual step: u32 Philox and threshold compare; primal step: f32 with two-sum accumulation)",
        "data": "synthetic (seeded generators)",
        "config": {"workload": "potts3d", "description": bench._describe("potts3d"), "n_vars": 2097152, "n_edges": 6242304,
                   "n_labels": 8, "chains": 64, "mode": "plain", "dual_bits_per_edge": 49, "layout": "pivot",
                   "l2": "inputs larger than L2 (tables and theta are GBs); no flush needed",
                   "parallelism": "replicas x1 (independent chains per GPU)"},
        "roofline": {"bound": "alu", "achieved": 233.123456789, "peak": 647.123456789, "unit": "G Philox4x32-10 calls/s",
                     "frac": 0.36012345678, "traffic": 12345678901, "traffic_source": "t" * 200, "kernel": "k_dual",
                     "peak_source": "p" * 200, "hbm_view": dict.fromkeys(("achieved", "peak", "frac"), 1.0),
                     "philox_only_kernel": {"calls_per_s": 5.47e11, "frac": 0.43}},
        "kernels": kernels, "gpu_launches": 60,
        "variants": {"fused": form, "splash": form, "log_partition": {"note": "n" * 400}, "ess": {"table": "z" * 20000}},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 12},
        "e2e": {"value": 9.93e9, "unit": bench.METRIC, "h2d_bytes_per_step": 134217728, "d2h_bytes_per_step": 134217728,
                "steps": 20, "api": "a" * 100},
        "cpu_baseline": {"kind": "oracle/cpu_sweep.c", "cores": 16, "sample": "s" * 150, "value": 4350000.0,
                         "unit": bench.METRIC, "single_core_oracle": {"sample": "o" * 300}},
        "other_configs": {"dense4096": other, "er_batch_2000": other, "ba_learned_1e6": {"unavailable": "exit 1: " + "e" * 300}},
    }


def test_default_line_is_short_and_complete():
    full = _full_line()
    line = bench.compact_line(full)
    assert len(json.dumps(line)) <= 2900
    for key in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
                "config", "gpu_launches", "clocks"):
        assert line[key] == full[key]
    for key in ("value", "ms_per_step"):
        assert abs(line[key] - full[key]) <= 1e-5 * full[key]
    assert line["roofline"]["kernel"] == "k_dual" and line["e2e"]["h2d_bytes_per_step"] == 134217728
    assert line["variants_ms_per_step"] == {"fused": 12.3457, "splash": 12.3457}
    assert line["other_configs"]["er_batch_2000"]["value"] == 34567900.0
    assert line["other_configs"]["ba_learned_1e6"]["unavailable"].startswith("exit 1")


def test_line_without_optional_parts():
    full = _full_line()
    full.update(variants={}, e2e=None, cpu_baseline=None)
    del full["other_configs"]
    line = bench.compact_line(full)
    assert line["e2e"] is None and line["cpu_baseline"] is None and "other_configs" not in line

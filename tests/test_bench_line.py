"""bench.py's result line: the contract's keys, whole within the last 3,000 characters of the output however
long the reports beside it are."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def report():
    roof = {"kernel": "walk (predict4_kernel)", "bound": "alu", "achieved": 0.8317265819437161, "peak": 1.25856, "frac":
            0.6608557255543765, "unit": "T warp-inst/s", "smem_frac": 0.7832819231, "ms_per_launch": 4.031948280334473,
            "peak_source": "p" * 90, "timing": "t" * 90, "hbm_floor": {"traffic": [1.0] * 50}}
    return {"metric": bench.METRIC, "value": 17917352461.7, "unit": bench.ROWS_TREES_UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 7.4391235, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int64",
            "data": "synthetic",
            "config": {"workload": bench.WORKLOAD, "rows": 111000, "features": 32, "trees_per_gpu": 500, "queries": 1000000,
                       "select": "64x15", "seeds": {"data": 1, "forest": 2, "queries": 3}, "l2": "l" * 130, "parallelism": "1 GPU"},
            "e2e": {"value": 1.1e10, "unit": bench.ROWS_TREES_UNIT, "h2d_bytes_per_step": 143000000, "d2h_bytes_per_step": 8000000,
                    "ms_per_step": 9.1234567, "steps": 5, "note": "n" * 160},
            "gpu_launches": 700, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 31, "reasons": []},
            "cpu_baseline": {"value": 5.9e6, "unit": bench.ROWS_TREES_UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 90},
            "fit_ms": 3.0123, "predict": {"value": 2.3e8, "unit": "queries/s", "ms": 4.2912345, "trees": 500},
            "select": {"ms": 0.0912345, "kernels": 64, "devices": 15}, "parity": "bit-exact vs oracle (tests/test_gpu_parity.py)",
            "roofline": roof, "roofline_fit": dict(roof, kernel="tree"), "kernels": {"a": ["x" * 5000]},
            "serving": {"runs": ["y" * 9000]}, "surrogate": {"z": "z" * 4000}}


def test_the_line_is_short_and_has_the_contract():
    out = report()
    line = json.dumps(bench.headline(out))
    assert len(line) < 2800 and "\n" not in line
    got = json.loads(line)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
              "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "cpu_baseline"):
        assert got[k] == out[k]
    assert got["roofline"]["frac"] == out["roofline"]["frac"]
    assert not {"serving", "surrogate", "kernels"} & set(got)


def test_a_report_without_the_optional_parts_still_has_a_line():
    out = {k: v for k, v in report().items() if k not in ("e2e", "cpu_baseline", "serving", "surrogate")}
    got = bench.headline(out)
    assert got["value"] == out["value"] and "e2e" not in got

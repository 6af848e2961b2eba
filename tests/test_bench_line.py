"""The bench's printed record stays short whatever the variants hold."""
import json


def test_compact_line_keeps_the_headline_and_stays_short():
    import bench
    line = {"metric": bench.METRIC, "value": 1.0, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 1.0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64+f32",
            "data": "synthetic", "config": {"model": "m" * 400}, "roofline": {"frac": 0.5, "note": "n" * 2000},
            "e2e": {"value": 2.0, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2},
            "gpu_launches": 3, "clocks": {"sm_mhz": 2070.0}, "cpu_baseline": {"value": 0.1},
            "roofline_levels": {"x": "y" * 3000}, "vcycle": {"a": 1}, "solve": {"5": {"cycles": 18}},
            "variants": {"batched_64": {"value": 7.0, "rows": ["r" * 100] * 100}, "speedup": 1.5}}
    out = bench.compact_line(line, "details.json")
    assert len(json.dumps(out)) < 4000
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "cpu_baseline"):
        assert out[k] == line[k]
    assert out["roofline"] == {"frac": 0.5} and out["variants"] == {"batched_64": 7.0}
    assert out["details"] == "details.json"

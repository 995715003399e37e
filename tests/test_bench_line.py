"""The benchmark's printed line: what its readers need, short enough for the tail of a log."""
import json

import bench


def record(variants):
    note = "a note of some length, as the full record carries them " * 4
    return {"metric": bench.METRIC, "value": 75.699403300124, "unit": bench.UNIT, "n_gpus": 8,
            "steps": 200, "warmup": 5, "ms_per_step": 11.081471761067709, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": note[:120], "nx": 256, "ny": 256, "nz": 256, "sweeps_per_step": 50,
                       "parallelism": "replicas x8", "l2": note[:120]},
            "gpu_launches": 10600, "gpu_launches_note": note,
            "roofline": {"bound": "alu", "achieved": 535.5842457784481, "peak": 625.2051877649805,
                         "unit": "GFP64op/s", "frac": 0.8566535535207018, "traffic": 689409280,
                         "kernel": note[:80], "launch_ms": 0.2192755162715912, "peak_source": note},
            "roofline_hbm": {"bound": "hbm", "achieved": 1836.288842668965, "peak": 6770.5,
                             "unit": "GB/s", "frac": 0.27121908908780223, "peak_source": note},
            "cpu_baseline": {"value": 0.9501438311911874, "unit": bench.UNIT, "cores": 16,
                             "kind": "oracle", "sample": note},
            "e2e": {"value": 73.01715517649235, "unit": bench.UNIT, "h2d_bytes_per_step": 268435456,
                    "d2h_bytes_per_step": 134217728, "steps": 40, "timer": note},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 20,
                       "reasons": ["sw_power_cap", "hw_slowdown"]},
            "variants": variants}


def test_short_and_complete():
    good = {"value": 1.0, "err_vs_oracle": {"metric": "m", "value": 1e-13, "tolerance": 1e-12}}
    variants = [dict(good, name="v%d" % i, cpu_baseline={"sample": "s" * 200}) for i in range(60)]
    variants[3]["err_vs_oracle"] = {"value": 2e-12, "tolerance": 1e-12}
    variants[4]["err_vs_oracle"] = {"value": float("nan"), "tolerance": 1e-12}
    variants[5] = {"name": "v5", "error": "RuntimeError('x')"}
    variants.append({"workload": "adjoint", "results": [{"err_vs_oracle": {"gu": 1.0, "gb": 1e-12,
                                                                          "tolerance": 1e-11}}]})
    full = record(variants)
    text = json.dumps(bench.headline(full, "/somewhere/bench_details.json"))
    assert len(text) < 2500 and "\n" not in text
    line = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
              "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "gpu_launches",
              "clocks"):
        assert line[k] == full[k]
    assert line["e2e"].items() <= full["e2e"].items() and line["e2e"]["d2h_bytes_per_step"]
    assert line["variants"] == {"run": 61, "failed": ["v5"], "oracle_errors": 61,
                                "beyond_tolerance": ["adjoint", "v3", "v4"]}


def test_without_variants_or_cpu_leg():
    full = record([])
    full["cpu_baseline"] = None
    line = json.loads(json.dumps(bench.headline(full, "d")))
    assert line["cpu_baseline"] is None and line["variants"]["run"] == 0

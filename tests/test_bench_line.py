"""bench.py's result line is short and whole: the measurement's own keys as they
were, headline figures of the other legs, whatever the legs report."""

import json

import bench


def _line():
    return {
        "metric": bench.METRIC, "value": 1700.123456, "unit": bench.UNIT, "n_gpus": 1, "steps": 20,
        "warmup": 5, "ms_per_step": 0.63, "ms_per_step_median": 0.63, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic (seeded point + line absorbers, 3% noise; cfg2 recipe)",
        "config": bench.config_dict(type("A", (), dict(order=3, form="fp32", frames=32, gpus=1)),
                                    bench.workload()),
        "clocks": {"sm_mhz": 1995.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 40},
        "e2e": {"value": 1239.1234567, "unit": bench.UNIT, "h2d_bytes_per_step": 33554432,
                "d2h_bytes_per_step": 100663296, "call": "pa_beamform_host (pinned host buffers)",
                "steps": 20, "chunks": [8, 8, 8, 8]},
        "gpu_launches": 80,
        "roofline": {"bound": "alu", "achieved": 26.123456789, "peak": 40.27, "unit": "Top/s",
                     "frac": 0.65123456, "traffic": None, "kernel": "k" * 90, "kernel_ms_per_launch": 0.52,
                     "kernels_ms_per_launch": {"a": 1.0}, "post_filter": {"x": list(range(500))}},
        "graph_path": {"note": "n" * 3000},
    }


def _leg(n):
    spread = {"median": 0.123456789, "min": 0.1, "max": 0.2, "runs": list(range(n))}
    return {"offered": {"runs": list(range(n)), "latency_ms_p50": spread, "latency_ms_p99": spread},
            "saturation": {"served_frames_per_s": spread}}


def test_the_line_is_short_and_keeps_the_measurement():
    line = _line()
    extras = {"serving": {"workload": "w" * 500, "bf16_kahan": _leg(2000), "fp32": _leg(2000),
                          "paired": {"saturation": {"pairs": 3}, "offered": {"pairs": list(range(2000))}}},
              "precision_form": {"value": 1630.12345678, "more": "m" * 500},
              "nearest_form": {"value": 2116.1}, "off_lattice_form": {"value": 1286.4},
              "throughput_batch": {"frames_per_s": 24246.81234, "kernels": list(range(500))},
              "cpu_baseline": {"value": 0.27, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 99},
              "precision_report": {"x": list(range(3000))}}
    out = bench.result_line(line, extras)
    assert len(json.dumps(out)) < 2300
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
                "scaling", "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches"):
        assert out[key] == line[key], key
    assert out["other_legs"]["throughput_batch_frames_per_s"] == 24247.0
    assert out["serving"]["fp32"]["p99_ms"] == 0.1235 and set(out["serving"]) == {"bf16_kahan", "fp32"}
    assert "graph_path" in line and "post_filter" in line["roofline"]  # (not changed in place)


def test_without_the_other_legs():
    out = bench.result_line(_line(), {})
    assert "serving" not in out and "other_legs" not in out and out["value"] == 1700.123456

"""The benchmark's result line: one JSON object with every key of the
measurement contract, short enough to survive whole in the last few KB of a run's
output, whatever the other workloads have to report."""
import json

import bench

CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "clocks", "gpu_launches", "roofline", "cpu_baseline")


def _head():
    roof = {"kernel": "tc_gemm", "class": "gemm_tc", "bound": "tensor", "achieved": 109.58566537702129,
            "peak": 928.8888888888889, "unit": "TFLOP/s", "frac": 0.11797499861162579, "dtype": "tf32",
            "issue_efficiency": 0.589874993058129, "mmas_per_product": 5, "traffic": None, "peak_source": "s" * 90,
            "peak_note": "n" * 200, "launches": 200, "ms_per_launch": 18.25056218, "share": 0.5653435833107331,
            "class_share": 0.5, "breakdown_ms": {f"c{k}": 1.0 / 3 for k in range(8)},
            "breakdown_tflops": {f"c{k}": 1.0 / 3 for k in range(8)}, "serialised_step_ms": 6456.449748,
            "sites": [{"site": f"s{k}", "ms": 1.0 / 7, "launches": k} for k in range(16)]}
    return {"metric": bench.METRIC, "value": 0.32208578223242407, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 6209.52587890625, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "tf32x2/fp32-acc products, f64 stabilisation", "data": "synthetic " + "d" * 80,
            "config": {"workload": bench.workload_name(bench.LARGE), "global_batch": 1, "seq_len": 100, "lattice": "100x100",
                       "chains_per_gpu": 1, "precision": "3xtf32", "n_wrap": 10, "tile_n": 64, "parallelism": "replicas x1",
                       "l2": "w" * 63, "fit": {"lattice": "8x8", "J": [1.0 / 3] * 4}, "setup_s": 6.33},
            "ms_per_weight": 3104.762939453125, "ms_per_accept_step": 6209.52587890625, "accept_rate": 0.5,
            "fp64": {"value": 0.1099195998239569, "unit": bench.UNIT, "extrapolated": True, "note": "n" * 90},
            "precision": {"reference": "r" * 120, "logdet_rel_err": 4.554441940031966e-07, "max_abs_dG": 1.58e-07},
            "separable": {"value": 0.6157813206585011, "unit": bench.UNIT, "ms_per_step": 3247.90625, "roofline": dict(roof)},
            "decorrelated_samples_per_s": None, "decorrelation_note": "n" * 130, "roofline": roof,
            "cpu_baseline": {"value": 1.36e-4, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "extrapolated": True,
                             "sample": "s" * 220},
            "e2e": {"value": 0.3220510220745215, "unit": bench.UNIT, "steps": 4, "h2d_bytes_per_step": 1000008,
                    "d2h_bytes_per_step": 1000012},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 62}, "gpu_launches": 24252,
            "workloads": {f"w{k}": {"rows": [{"value": 1.0 / 3}] * 100} for k in range(8)}}


def test_result_line_is_short_and_whole():
    head = _head()
    text = bench.result_line(head)
    assert "\n" not in text and len(text) <= 3000
    line = json.loads(text)
    for k in CONTRACT:
        assert k in line
        if k not in ("config", "roofline"):
            assert line[k] == head[k]
    for k in ("workload", "global_batch", "seq_len", "parallelism", "l2"):
        assert line["config"][k] == head["config"][k]
    assert "workloads" in head and "workloads" not in line and len(head["roofline"]) > len(line["roofline"])


def test_result_line_of_a_partial_run():
    head = {"metric": bench.METRIC, "value": None, "unit": bench.UNIT, "n_gpus": 1, "steps": 2, "warmup": 3, "ms_per_step": None,
            "config": {"workload": "w"}, "partial": "headline workload not run", "workloads": {"local4": {"x": [1] * 5000}}}
    line = json.loads(bench.result_line(head))
    assert line["partial"] == head["partial"] and "workloads" not in line

"""bench.py's line on standard output: every field of the record that is compared from run to run, short enough to be read back from
the tail of a log."""
import json

import bench


def _record(name, tiles):
    roof = {"bound": "tensor", "achieved": 823.123456789012, "peak": 1649.9123456789, "unit": "TFLOP/s", "frac": 0.498765432109876,
            "traffic": 8852000000.0, "kernel": "moe_apk_pair_kernel", "traffic_source": "ncu " * 40, "peak_source": "measured",
            "peak_kind": "burst", "launch_ms_mean": 2.2345678901234, "launch_ms_min": 2.1, "algorithmic_flops_per_launch": 1.855e12,
            "algorithmic_bytes_per_launch": 7350000000.123, "tensor_frac_of_burst": 0.5, "tensor_frac_of_sustained": 0.6, "hbm_frac": 0.5}
    e2e = {"value": 815.123456789, "unit": "TFLOP/s", "h2d_bytes_per_step": 50855936, "d2h_bytes_per_step": 50331648, "how": "text " * 40}
    rec = {"value": 823.123456789012, "unit": "TFLOP/s", "steps": 20, "warmup": 5, "ms_per_step": 2.253456789012, "dtype": "bf16",
           "config": {"workload": name, "ops": [[1, 16384], [0, 256]], "layers": 8, "experts": 256, "top_k": 8, "hidden": 3072,
                      "inter": 1536, "l2": "inputs_exceed_l2 (weights >> 126 MB, no flush)", "buffers": "text " * 40, "replicas": 1,
                      "fused_combine": True, "paired_ops": True, "decode_budgets": [16, 32, 64]},
           "clocks": {"sm_mhz": 1342, "sm_max_mhz": 1965, "reasons": ["sw_power_cap"], "samples": 13}, "gpu_launches": 1234,
           "roofline": roof, "e2e": e2e, "e2e_serial": dict(e2e, steps=6, ms_per_step=4.123456789),
           "cpu_baseline": {"value": 0.0145123456789, "unit": "TFLOP/s", "cores": 16, "kind": "oracle",
                            "sample": "oracle plan on all 8192 tokens + FFN/combine on 256 seeded tokens of c3 (4.10 s)"}}
    if tiles:
        rec["tiles"] = {str(i): {"x": 1.0 / 3.0} for i in range(200)}
    return rec


def test_the_line_is_whole_and_short():
    full = {"metric": bench.METRIC, "n_gpus": 1, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "data": "synthetic"}
    full.update(_record("c3", False))
    full["sub_results"] = {n: _record(n, n == "c4") for n in ("c2", "c4", "c5")}
    text = json.dumps(bench.short_line(full))
    assert len(text) < 2700
    line = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
                "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "roofline", "cpu_baseline"):
        assert key in line, key
    assert abs(line["value"] / full["value"] - 1.0) < 1e-5
    assert line["e2e"]["h2d_bytes_per_step"] == 50855936 and line["e2e"]["d2h_bytes_per_step"] == 50331648
    assert line["gpu_launches"] == 1234 and line["clocks"] == full["clocks"]
    assert all(r["value"] > 0 and 0 < r["roofline"]["frac"] < 1 for r in line["sub_results"].values())
    full["tiles"] = full["sub_results"]["c4"]["tiles"]
    del full["sub_results"]
    assert len(json.dumps(bench.short_line(full))) < 2700

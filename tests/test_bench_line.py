"""bench.py prints one line short enough for a reader that keeps the end of the output, with the contract's fields in it."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

CONTRACT = {"metric": "hbmm_effective_binary_tops", "value": 264.34215821988977, "unit": "TOPS", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.4478288173675537, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": {"workload": "w", "l2": "x" * 900}, "gpu_launches": 1600,
            "e2e": {"value": 30.046388547849, "unit": "TOPS", "ms_per_step": 3.9, "h2d_bytes_per_step": 144506880, "d2h_bytes_per_step": 192675840},
            "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": []}}


def _record():
    row = {"name": "alexnet_fc6_b256", "M": 256, "N": 4096, "K": 9216, "beta": 64, "scale_dtype": "f32", "kernel": "k" * 30,
           "hbmm_gemm_ms": 0.05123456789, "tops": 377.123456789123, "frac_of_popcount_hbm_roofline": 1.0312345678912, "timing": "t" * 60,
           "cublas": {"fp32_ms": 0.1234567891234, "bf16_ms": 0.0123456789}, "oracle": {"rows": 64, "seconds": 1.23456789, "note": "n" * 200}}
    kernel = {"layer": "conv2_x", "ms": 0.05, "bound": "tensor", "achieved": 960.4163676767721, "frac": 0.14660607, "timing": "t" * 80}
    return dict(CONTRACT, configs=[dict(row) for _ in range(40)], kernels=dict({k: [dict(kernel) for _ in range(4)] for k in "abcd"}, buffer_sets_per_layer=[3, 5, 9, 12]),
                other_rows=[dict(row) for _ in range(60)], context={"paper": "p" * 300}, roofline=dict(kernel),
                measured_alu_rates={"popc": {"ops_per_s": 4.6e12, "sm_mhz": 1965}, "planning_figures": {"a": 1}})


def test_printed_line_is_short_and_keeps_the_contract():
    import bench
    text = bench.printed_line(_record(), "rows.json")
    assert len(text) <= bench.LINE_BYTES and "\n" not in text
    line = json.loads(text)
    assert {k: line[k] for k in CONTRACT} == CONTRACT
    assert len(line["configs"]) == 40 and line["configs"][0]["hbmm_gemm_ms"] == 0.0512346
    assert line["kernels"]["a"][0] == {"layer": "conv2_x", "ms": 0.05, "frac": 0.146606}


def test_rows_go_before_the_contract_does():
    import bench
    r = _record()
    r["configs"] = r["configs"] * 10
    text = bench.printed_line(r)
    assert len(text) <= bench.LINE_BYTES
    assert {k: json.loads(text)[k] for k in CONTRACT} == CONTRACT

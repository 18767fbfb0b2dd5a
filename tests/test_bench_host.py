"""Host-side arithmetic of bench.py (no GPU): op and byte counts per layer, the traffic table's keys, and the
shape of the reference arm's JSON line."""
import json
import os
import subprocess
import sys

import bench
from paper_2507_14811_b200 import workloads as WL

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_op_and_byte_counts():
    adaln, fc2 = WL.WORKLOADS["dit_xl2"]
    executed, useful = bench.layer_ops(adaln)
    assert useful == 2 * 2048 * 6912 * 1152 and executed == 2 * useful          # dual: two GEMMs
    fc1 = WL.WORKLOADS["sd3_mmdit"][1]
    assert bench.layer_ops(fc1) == (2.0 * 8858 * 6144 * 1536, 2.0 * 8858 * 6144 * 1536)
    # GEMM: both code matrices + weight codes + bf16 output; quantize: bf16 in + one byte per code matrix
    assert bench.gemm_bytes(fc2) == 2048 * 4608 * 2 + 1152 * 4608 + 2 * 2048 * 1152
    assert bench.quant_bytes(fc2) == 2048 * 4608 * (2 + 2)
    assert bench.quant_bytes(fc1) == 8858 * 1536 * (2 + 1)
    assert bench.layer_ops(fc2, M=100)[1] == 2.0 * 100 * 1152 * 4608


def test_traffic_table_names_workloads_and_goes_stale_with_the_kernel_source():
    assert set(bench.GEMM_DRAM_TRAFFIC) <= set(WL.WORKLOADS)
    for e in bench.GEMM_DRAM_TRAFFIC.values():
        assert isinstance(e["bytes"], int) and e["bytes"] > 0 and len(e["source_tag"]) == 16 and e["from"]
    assert bench.gemm_dram_traffic("no_such_workload")[0] is None
    saved = dict(bench.GEMM_DRAM_TRAFFIC)
    try:
        bench.GEMM_DRAM_TRAFFIC["tiny_qkv"] = {"bytes": 123, "source_tag": "0" * 16, "from": "test"}
        assert bench.gemm_dram_traffic("tiny_qkv")[0] is None                      # another kernel source: stale
        bench.GEMM_DRAM_TRAFFIC["tiny_qkv"]["source_tag"] = bench.gemm_source_tag()
        assert bench.gemm_dram_traffic("tiny_qkv") == (123, "test")
    finally:
        bench.GEMM_DRAM_TRAFFIC.clear()
        bench.GEMM_DRAM_TRAFFIC.update(saved)


def test_fractions_against_the_three_peaks():
    p8 = bench.eight_bit_peaks({"bf16_tflops": 1600.0, "bf16_tflops_sustained": 1400.0})
    assert p8 == {"burst": 3200.0, "sustained": 2800.0, "nominal": 4500.0}
    f = bench.fractions(1600.0, p8)
    assert f == {"of_measured_burst": 0.5, "of_measured_sustained": round(1600 / 2800, 4), "of_nominal_4500": round(1600 / 4500, 4)}


def test_measured_peaks_have_the_fields_the_roofline_uses():
    p = bench.measured_peaks()
    assert p["hbm_gbs"] > 1000 and p["bf16_tflops"] > 100 and p["source"] in ("measured", "fallback")


def test_reference_arm_prints_one_json_line_on_the_tiny_workload():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--workload", "tiny_qkv",
                          "--steps", "1", "--warmup", "0"], capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert out.returncode == 0, out.stderr[-2000:]
    lines = [l for l in out.stdout.splitlines() if l.strip()]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["unit"] == "TOPS" and d["value"] > 0 and d["higher_is_better"] is True
    assert d["cpu_baseline"]["kind"] == "oracle" and d["e2e"]["h2d_bytes_per_step"] == 0
    assert d["config"]["workload"] == "tiny_qkv"


def test_report_line_is_short_and_keeps_the_measurement():
    """The line on standard output: every figure of the measurement, no tables, and short enough for a log that keeps the last
    few thousand characters, for every workload and eight GPUs."""
    note = "x" * 400
    for name, specs in WL.WORKLOADS.items():
        out = {"metric": bench.METRIC, "value": 12345.67, "unit": "TOPS", "n_gpus": 8, "steps": 20, "warmup": 5, "ms_per_step": 0.12345,
               "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int8", "data": "synthetic",
               "config": bench.report_config(name, specs, 8, 20, 81, 0.5123, "CUDA graph", 4, 123 << 20),
               "timed_region_s": 0.5123, "graph_replays": 81, "useful_tops": 1234.56,
               "whole_step": dict(bench.fractions(1600.0, bench.eight_bit_peaks({"bf16_tflops": 1600.0, "bf16_tflops_sustained": 1400.0})), note=note),
               "ms_per_step_kernels_timed_alone": 0.12345, "ms_per_step_planned_calls_from_host": 0.12345, "planned_calls_note": note,
               "frac_of_nominal_4500_tops": 0.4567,
               "e2e": {"value": 136.78, "unit": "TOPS", "h2d_bytes_per_step": 190000000, "d2h_bytes_per_step": 218000000, "ms_per_step": 5.4321, "call": note},
               "gpu_launches": 12345,
               "roofline": {"bound": "tensor+hbm (per layer, see per_layer.gemm_bound)", "achieved": 2765.4, "peak": 3166.6, "unit": "TFLOP/s",
                            "frac": 0.8765, "frac_of_sustained_peak": 1.0123, "traffic": None, "kernel": "segquant_gemm_kernel",
                            "launches_per_step": 3, "note": note},
               "quantize_roofline": {"bound": "hbm", "achieved": 5432.1, "peak": 6549.8, "unit": "GB/s", "frac": 0.8294, "kernel": "quantize_kernel"},
               "cpu_baseline": {"value": 0.08112, "unit": "TOPS", "cores": 16, "kind": "oracle", "sample": note},
               "clocks": {"sm_mhz": 1447.0, "sm_max_mhz": 1965.0, "reasons": ["sw_power_cap"], "samples": 12},
               "per_layer": [{"note": note}] * 20,
               "workloads": {w: {"ms_per_step": 0.12345, "per_layer": [note] * 9} for w in WL.WORKLOADS if w != name}}
        line = bench.report_line(out)
        assert len(json.dumps(line)) <= bench.LINE_MAX_CHARS, (name, len(json.dumps(line)))
        for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype",
                    "data", "config", "gpu_launches", "clocks"):
            assert line[key] == out[key]
        assert set(line["e2e"]) >= {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
        assert line["roofline"]["frac"] == 0.8765 and line["clocks"]["reasons"] == ["sw_power_cap"]
        assert "per_layer" not in line and "workloads" not in line
        assert line["ms_per_step_of_workloads"] == {w: 0.12345 for w in WL.WORKLOADS if w != name}

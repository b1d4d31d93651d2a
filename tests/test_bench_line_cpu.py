"""The line that bench.py prints stays short enough to be read back whole."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def full_line():
    """A line with everything in it, with the lengths that the four matrices' sections have."""
    names = ["stencil27_128^3", "fem3x3_n3M", "rmat_s22", "uniform_n1M"]
    roof = {"kernel": "k_spmv_g1_segs+k_spmv_fixup", "achieved": 3333.3, "peak": 6778.7, "frac": 0.4919, "unit": "GB/s",
            "why": "w" * 300, "traffic": {"bytes": 1650000000, "source": "profiles/traffic.json"}}
    sweep = {f"{r}x{c}": {str(v): 123.4 for v in range(12)} for r in (1, 2, 4, 8) for c in (4, 8, 16)}
    per = [{"matrix": n, "n": 3000000, "nnz": 161981010, "shape": "1x8", "variant": 22, "convert_ms": 1.744,
            "convert_over_spmv": 3.52, "avg_nnz_per_block": 2.7, "segments": 0, "ms": 0.4941, "gflops": 655.6, "gbs": 3333.3,
            "hbm_frac": 0.4919, "sweep_gflops": sweep, "roofline": roof} for n in names]
    csr = {"value": 435.1, "unit": "GFLOP/s", "speedup_beta_over_csr": 1.21,
           "per_matrix": {n: {"group": 8, "long_rows_split": True, "gflops": 435.1, "gbs": 5000.1, "plain_gflops": 400.1,
                              "beta_over_csr": 1.234} for n in names}}
    cg = {"workload": "w" * 120, "format": "f" * 60,
          **{k: {"ms": 10.123, "iterations": 406, "outer": 8, "rel_residual": 9.9e-11, "converged": True}
             for k in ("fp64_cg", "mixed_f32", "mixed_bf16", "reliable_f32", "reliable_bf16")}, "speedup_mixed_f32": 1.7}
    low = {"value": 757.1, "unit": "GFLOP/s", "hbm_gbs": 3333.3, "per_matrix": per, "roofline": roof, "hbm_frac": 0.49,
           "csr": csr, "error_vs_float64": {n: {"max_rel_to_max": 1e-7, "rel_l2": 1e-7} for n in names}}
    spmm = {n: {f"k{k}": {"ms": 0.6099, "gflops": 1711.6, "shape": "1x8", "ktile": 8, "gbs": 1483.5, "hbm_frac": 0.2188}
                for k in (1, 2, 4, 8, 16, 32)} for n in names[:2]}
    return {"metric": bench.METRIC, "value": 552.1, "unit": "GFLOP/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 1.1, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": "w" * 90, "formats": {n: "beta(1,8) variant 22" for n in names},
                                            "selection": "s" * 80, "l2": "l" * 70, "parallelism": "single GPU"},
            "hbm_gbs": 3000.1, "hbm_peak": {"measured_gbs": 6778.7, "measured_source": "MEASURED_PEAKS.json",
                                            "nominal_gbs": 7672.3, "nominal_source": "n" * 50},
            "roofline": {**roof, "alu_fp64": {"achieved": 655.6, "peak": 1250.0, "unit": "GFLOP/s", "frac": 0.52,
                                              "peak_measured": 1240.1, "frac_of_measured": 0.53, "why": "w" * 200,
                                              "peak_source": "p" * 200}},
            "cpu_baseline": {"value": 17.1, "unit": "GFLOP/s", "note": "n" * 300},
            "e2e": {"value": 530.1, "unit": "GFLOP/s", "h2d_bytes_per_step": 79000000, "d2h_bytes_per_step": 79000000},
            "gpu_launches": 200, "clocks": {"sm_mhz": 1900, "sm_max_mhz": 2070, "reasons": ["sw_power_cap"]},
            "wall_s_timed": 1.0, "csr": csr, "per_matrix": per, "f32": low, "bf16": low, "cg": {**cg, "shifted": cg},
            "spmm_f32": spmm, "selector": {"model": "m" * 60, "held_out": {k: {"mean": 0.0171, "median": 0.0025, "p90": 0.046}
                                                                        for k in ("regret_mlp", "regret_poly")}},
            "batch_f32": {"workload": "w" * 90, "nnz_total": 99489071, "shapes": {}, "graph_ms": 0.37, "gflops_graph": 533.5,
                          "direct_ms": 0.38, "speedup_vs_per_matrix": 6.1}}


def test_printed_line_is_short_and_keeps_the_figures():
    line = full_line()
    short = bench.short_line(line)
    text = json.dumps(short)
    assert len(json.dumps(line)) > 20000 and len(text) <= bench.LINE_MAX
    sections = {"roofline", "per_matrix", "csr", "f32", "bf16", "cg", "spmm_f32", "batch_f32", "selector"}
    assert all(short[k] == line[k] for k in line if k not in sections)
    assert set(line) <= set(short)
    assert short["per_matrix"]["rmat_s22"]["gflops"] == 655.6 and short["f32"]["value"] == 757.1
    assert short["cg"]["ms_and_iterations"]["reliable_f32"] == (10.123, 406) and "shifted" in short["cg"]
    assert short["selector"] == {"regret_mlp": 0.0171, "regret_poly": 0.0171}
    assert short["roofline"]["frac"] == 0.4919 and "why" not in short["roofline"]["alu_fp64"]

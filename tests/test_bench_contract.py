"""Host logic of ``bench.py`` on the CPU: the algorithmic work each kernel's
roofline divides by, the roofline arithmetic, the source-hash gating of the
DRAM traffic figures and the workload description of the JSON line."""
import hashlib
import os
import shutil

import pytest

import bench


class _Shape:
    """The fields of a layer that the bench's models read."""

    def __init__(self, name, din, dout, g, bits, K):
        self.name, self.din, self.dout, self.g, self.bits, self.K = name, din, dout, g, bits, K


Q_PROJ = _Shape(bench.WORKLOAD, 4096, 4096, 128, 3, 10)


def test_kernel_work_closed_forms():
    p, d, g = 4096, 4096, 128
    G = d // g
    # sweep product: one (p x d) x (d x 256) product of useful work, four digit planes issued
    m = bench.kernel_model("sweep_product", Q_PROJ)
    assert m["bound"] == "tensor" and m["work"] == 2.0 * p * 256 * d == 8589934592.0
    assert m["issued"] == 4 * m["work"]
    # Gram: the G (G + 1) / 2 blocks h <= i of c_h^T H_hi c_i, 2 p g^2 each
    m = bench.kernel_model("gram", Q_PROJ)
    assert m["work"] == 2.0 * p * g * g * G * (G + 1) / 2 == 70866960384.0
    # target projection P = W H and its 18 digit pairs
    m = bench.kernel_model("proj", Q_PROJ)
    assert m["work"] == 2.0 * p * d * d and m["issued"] == 18 * m["work"]
    # Babai: the dense triangular back substitution, g^2 flops per (row, group), two groups a launch
    assert bench.kernel_model("sweep_babai", Q_PROJ) == {"bound": "alu", "work": 2.0 * g * g * p}
    # the scale solve moves each row's float64 Gram matrix once
    m = bench.kernel_model("scale_solve", Q_PROJ)
    assert m["bound"] == "hbm" and m["work"] >= 8.0 * p * G * G
    assert bench.kernel_model("no_such_kernel", Q_PROJ) is None


def test_roofline_arithmetic():
    pk = {"hbm_gbs": 6789.0, "bf16_tflops": 1942.2, "bf16_tflops_sustained": 1736.3}
    # 10 launches of 35 us each
    e = bench.roofline_entry("sweep_product", {"launches": 10, "total_ms": 0.35}, Q_PROJ, pk, "measured")
    achieved = 2.0 * 4096 * 256 * 4096 / 35e-6 / 1e12
    assert e["bound"] == "tensor" and e["unit"] == "TFLOP/s"
    assert e["achieved"] == pytest.approx(achieved) and e["peak"] == 1736.3
    assert e["frac"] == pytest.approx(achieved / 1736.3)
    assert e["issued_frac"] == pytest.approx(4 * e["frac"])
    assert e["avg_us"] == pytest.approx(35.0)
    # an HBM-bound kernel against the copy bandwidth
    e = bench.roofline_entry("rhs", {"launches": 2, "total_ms": 0.08}, Q_PROJ, pk, "measured")
    assert e["unit"] == "GB/s" and e["peak"] == 6789.0
    assert e["frac"] == pytest.approx(e["achieved"] / 6789.0)
    # Babai against the float32 FMA rate of 152 SMs at 2070 MHz
    e = bench.roofline_entry("sweep_babai", {"launches": 1, "total_ms": 0.0186}, Q_PROJ, pk, "measured")
    assert e["bound"] == "alu"
    assert e["peak"] == pytest.approx(152 * 128 * 2 * 2070e6 / 1e12)
    # no launches, no entry
    assert bench.roofline_entry("sweep_product", {"launches": 0, "total_ms": 0.0}, Q_PROJ, pk, "x") is None


def test_traffic_is_reported_only_for_an_unchanged_source(tmp_path, monkeypatch):
    # with the committed sources, a figure is either the committed one (hash
    # matches) or absent; never a different number
    for k, (fname, sha, val) in bench.TRAFFIC.items():
        path = os.path.join(bench.ROOT, "paper_2609_38599_gb300", "csrc", fname)
        cur = hashlib.sha1(open(path, "rb").read()).hexdigest()[:12]
        assert bench.traffic_for(k) == (val if cur == sha else None)
    # a changed source file withdraws its figure
    csrc = tmp_path / "paper_2609_38599_gb300" / "csrc"
    csrc.mkdir(parents=True)
    fname = bench.TRAFFIC["sweep_product"][0]
    shutil.copy(os.path.join(bench.ROOT, "paper_2609_38599_gb300", "csrc", fname), csrc / fname)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    unchanged = bench.traffic_for("sweep_product")
    with open(csrc / fname, "a") as fh:
        fh.write("\n// changed\n")
    assert bench.traffic_for("sweep_product") is None
    assert unchanged in (None, bench.TRAFFIC["sweep_product"][2])
    assert bench.traffic_for("not_in_table") is None


def test_roofline_traffic_only_for_the_main_workload():
    pk = {"hbm_gbs": 6789.0, "bf16_tflops": 1942.2, "bf16_tflops_sustained": 1736.3}
    other = _Shape("llama2_7b_down_proj_4096x11008_g128_w4", 11008, 4096, 128, 4, 10)
    e = bench.roofline_entry("sweep_product", {"launches": 1, "total_ms": 0.07}, other, pk, "measured")
    assert e["traffic"] is None


def test_config_names_the_workload_and_its_l2_note():
    c = bench.config_dict(Q_PROJ)
    assert c["workload"] == bench.WORKLOAD
    assert (c["din"], c["dout"], c["group_size"], c["bits"], c["K"]) == (4096, 4096, 128, 3, 10)
    assert c["early_stop"] is False and c["host"] == "RTN"
    # W 64 MB, P and the folded P 128 MB each, digit planes 448 MB: all larger than L2
    assert "W 64 MB" in c["l2"] and "128 MB" in c["l2"] and "448 MB" in c["l2"]
    assert bench.config_dict(Q_PROJ, note="x")["note"] == "x"


def test_printed_line_is_short_and_keeps_the_contract():
    """A record as long as a full run's, printed in fewer than 2600 characters
    with every key of the contract unrounded."""
    import json
    x = 1.0 / 3
    kernels = {k: {"launches": 7160, "total_ms": 1e3 * x, "avg_us": 1e4 * x, "share": x}
               for k in ("validate", "residual", "init_rows", "gram", "scale_solve", "slice_rows", "proj", "whw",
                         "rhs", "ptilde", "sweep_product", "sweep_babai")}
    roof = bench.roofline_entry("sweep_product", {"launches": 10, "total_ms": x}, Q_PROJ,
                                {"bf16_tflops_sustained": 1736.3}, "measured")
    cfg = {"din": 4096, "dout": 14336, "s_per_layer": x, "weights_per_s": 1e9 * x, "launches_per_step": 358.0,
           "roofline": roof, "roofline_all": {k: roof for k in kernels}, "kernels": kernels}
    full = {"metric": bench.METRIC, "value": 1e9 * x, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 40 * x, "s_per_layer": x, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": bench.DTYPE, "data": "synthetic (seeded Llama-2-7B-shaped layer, RTN host)",
            "config": bench.config_dict(Q_PROJ), "roofline": roof, "roofline_all": {k: roof for k in kernels},
            "gpu_launches": 7160, "kernel_timing": "x" * 130, "launches_per_step": 358.0,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 12, "reasons": ["sw_power_cap"]},
            "kernels": kernels,
            "postpass": {k: {"ms": x, "bytes": 51380224, "GB_s": 1e3 * x, "hbm_frac": x, "note": "y" * 50}
                         for k in ("dequantize_f16", "pack_codes", "canonicalize")},
            "configs": {k: cfg for k in ("tiny_256x256_g64_w3", "llama2_7b_down_proj_4096x11008_g128_w4",
                                         "llama3_8b_gate_proj_14336x4096_g128_w3", "llama2_7b_block")},
            "hessian": {"kernel_ms": 10 * x, "tokens_per_s": 1e8 * x, "roofline": roof, "cpu_baseline": {}},
            "early_stop": {"s_per_layer": x, "iters_mean": 28 * x, "rows_solved_at_k": [x] * 10},
            "mu_target": {"ms_per_layer_mu_0.5": 50 * x, "ms_per_layer_mu_1.0": 40 * x, "workload": "z"},
            "ablations": {k: 100 * x for k in ("gap_independent_pct_median", "gap_coordinate_pct_median",
                                               "probe_ms_per_group", "babai_after_single_code_pct",
                                               "joint_over_fixed_heldout_pct_median", "rows_improved_by_joint")},
            "e2e": {"value": 1e9 * x, "unit": bench.UNIT, "h2d_bytes_per_step": 84934656,
                    "d2h_bytes_per_step": 17301504, "ms_per_step": 40 * x},
            "cpu_baseline": {"value": 1e5 * x, "unit": bench.UNIT, "cores": 16, "kind": "oracle",
                             "sample": "94 of 4096 rows, K=10, full din, 15.5 s"}}
    short = bench.short_line(full)
    text = json.dumps(short)
    assert len(text) < 2600 and "\n" not in text, len(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "roofline", "gpu_launches", "clocks", "e2e",
                "cpu_baseline"):
        assert short[key] == full[key], key
    assert short["configs_s"]["llama2_7b_block"] == 0.33333 and short["kernels"]["gram"] == [7160, 3333.3]

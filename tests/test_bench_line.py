"""The benchmark's printed line holds what a reader of it needs and stays short:
sweeps and per-system lists, which made it 40 kB long, go to the details file."""
import json

import bench


def _line():
    sweep = [{"requests": 1, "p50_ms": 1.23456789, "p99_ms": 2.0, "atom_steps_per_s": 3.0e7} for _ in range(4)]
    one = {"p50_ms": 1.0, "p99_ms": 2.0, "atom_steps_per_s": 3.0e7, "calls": 7}
    errors = {"max_dE_rel": 1e-9, "max_dF_over_rms": 1e-5, "per_system": {"n": list(range(512)), "dE_rel": [1e-9] * 512}}
    ev = {"atom_evals_per_s": 1.0e8, "ms_per_eval": 7.0, "kernel_ms": {"k_desc": 1.0}}
    return {"metric": bench.METRIC, "value": 231408434.23490256, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 3,
            "ms_per_step": 4.531278228759765, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": {"workload": "large"}, "forms": {"fp32": {"value": 1.0, "ms_per_step": 4.5}},
            "roofline": {"kernel": "k_force", "frac": 0.48}, "kernels": {f"k_{i}": {"launches": 20, "ms_per_launch": 1.0 / (i + 1),
                                                                                  "share": 0.1} for i in range(15)},
            "cpu_baseline": {"value": 1.0, "split": {"atoms": 1}}, "e2e": {"value": 2.0e8}, "gpu_launches": 176,
            "clocks": {"sm_mhz": 2070.0}, "batch": {"workload": "x" * 200, **{k: {"atom_evals_per_s": 1.0e8, "errors": errors}
                                                                             for k in ("fp32", "bf16")}},
            "radial_table": {"direct": one}, "paper_models": {"workload": "y" * 200, "k32": {"fp32": ev, "bf16": ev}},
            "graphs": {"eager": one}, "serving": {"batched_fp32": {"sweep": sweep}, "at_2000_per_s": {
                k: one for k in ("batched_fp32", "batched_bf16", "per_request_fp32")}}}


def test_printed_line_is_whole_and_short():
    line = _line()
    out = json.loads(json.dumps(bench.compact(line)))
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert k in out, k
    assert abs(out["value"] / line["value"] - 1) <= 5e-6
    assert out["serving_2000_per_s"]["batched_fp32"] == {"p50_ms": 1.0, "p99_ms": 2.0, "atom_steps_per_s": 3.0e7}
    assert out["batch"]["fp32"]["max_dF_over_rms"] == 1e-5 and out["paper_models_ms"]["k32"]["bf16"] == 7.0
    assert len(json.dumps(out)) < 4000
    assert "per_system" in line["batch"]["fp32"]["errors"]        # the argument is left as it was


def test_short_lines_pass_through():
    line = {k: v for k, v in _line().items() if k not in ("batch", "radial_table", "paper_models", "graphs", "serving")}
    out = bench.compact(line)
    assert out["metric"] == bench.METRIC and "batch" not in out

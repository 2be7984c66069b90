"""The benchmark's printed line is short and whole: every key of the contract, no side
measurement however long."""
import json


def test_headline_keeps_the_contract_keys_and_stays_short():
    import bench
    form = {"value": 3.5e8, "ms_per_step": 0.28, "final_rmse": 0.41, "phases_ms": {"omp": 0.2},
            "per_iteration": [[0.123456789] * 2] * 500}
    line = {"metric": bench.METRIC, "value": 3.5e8, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.28, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": {"workload": "w" * 200}, "roofline": {"kernel": "omp", "frac": 0.2},
            "phases_ms": {"omp": 0.2}, "phase_roofline": {}, "forms": {f: dict(form) for f in ("fp32", "bf16", "fp8")},
            "atom_update_variants": {"x" * 3000: 1}, "batched": {"y" * 3000: 1}, "table1": {"z" * 3000: 1},
            "learned": None, "c1": None, "fp32_peak": {}, "cpu_baseline": None,
            "e2e": {"value": 2.5e8, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
            "gpu_launches": 200, "clocks": {"sm_mhz": 1900, "sm_max_mhz": 2070, "reasons": []}}
    text = json.dumps(bench.headline(line, "/somewhere/bench_details.json"))
    assert len(text) < 4000 and "\n" not in text
    out = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "forms"):
        assert k in out, k
    assert out["details"] == "bench_details.json"
    assert set(out["forms"]["bf16"]) == {"value", "ms_per_step", "final_rmse"}

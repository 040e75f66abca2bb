"""The benchmark's JSON line (no GPU): the required fields as they were measured, and short enough for
a reader that keeps the last 3 KB of the output."""
import json


def _full():
    wide = {"workload": "w" * 200, "profiled_run": {"x%d" % i: 1.0 / 3.0 for i in range(200)}}
    return {
        "metric": "CLR multiply TFLOP/s and ms per Newton-Schulz S^-1/2 iteration at stated error",
        "value": 514.3168157949493, "unit": "TFLOP/s", "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 17.102479934692383, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "bf16x3", "data": "synthetic",
        "config": {"workload": "w" * 90, "n": 16384, "clusters": 96, "precision": "bf16x3",
                   "l2": "l" * 120, "parallelism": "replicas"},
        "accuracy": {"rel_frob_sampled": 4.761541273497395e-06, "tiles_sampled": 4,
                     "frob_over_normA_normB_sampled": 3.731639651836636e-08},
        "phases_ms_per_step": {"ms_%d" % i: 0.09548799693584442 for i in range(6)},
        "algorithmic_flops_per_step": 8796093022208.0,
        "roofline": {"bound": "tensor", "achieved": 576.7960149871348, "peak_basis": "p" * 150,
                     "kernel": "split_gemm_kernel<2, 1>"},
        "cpu_baseline": {"value": 0.1597858715409343, "unit": "TFLOP/s", "cores": 16,
                         "kind": "oracle", "sample": "s" * 150},
        "e2e": {"value": 90.04388786663608, "unit": "TFLOP/s", "h2d_bytes_per_step": 4294967296,
                "d2h_bytes_per_step": 2147483648, "ms_each": [62.3, 197.11, 33.6]},
        "fp64_dense": dict(wide, tflops=0.98), "fp64_accurate_tensor": dict(wide, tflops=34.2),
        "chain_product": {"fp64": {"us_per_product": 411.07}}, "ns": dict(wide, ms_per_iteration=3.2),
        "ns_lattice": dict(wide, ms_per_iteration=451.7), "ns_lattice_split": None,
        "ns_lattice_ozaki": dict(wide, ms_per_iteration=108.6), "ns_coulomb": wide,
        "ns_lattice_large": {"ozaki": dict(wide, ms_per_iteration=484.0)},
        "batch": {"autotuned": dict(wide, ms_per_batch=33.5)}, "gpu_launches": 28,
        "clocks": {"sm_mhz": 1900.0, "sm_max_mhz": 2070.0, "reasons": []}}


def test_the_line_is_short_and_keeps_the_required_fields(repo_root, monkeypatch):
    monkeypatch.syspath_prepend(repo_root)
    import bench
    full = _full()
    text = json.dumps(bench.headline(full))
    assert len(text) < 2800
    line = json.loads(text)
    for k in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "gpu_launches", "clocks"):
        assert line[k] == full[k], k
    assert abs(line["value"] / full["value"] - 1) < 1e-5
    assert abs(line["ms_per_step"] / full["ms_per_step"] - 1) < 1e-5
    assert line["e2e"]["h2d_bytes_per_step"] == 4294967296
    assert line["config"]["workload"] == full["config"]["workload"]
    assert line["also"]["ns_lattice_4096_ms_per_iteration"]["ozaki"] == 108.6
    assert line["also"]["ns_lattice_8192_ms_per_iteration"]["fp64"] is None

"""The line that bench.py prints is short and keeps the keys that a reader of the line looks up (CPU)."""
import json

import bench

CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "clocks", "gpu_launches")


def _record(fat):
    """A record of the kind run_gpu makes, its texts and lists `fat` times as long as usual."""
    text = "operator and vectors in shared memory, grid sums on the arrivals, and so on; " * fat
    roof = {"kernel": "k_pcg_stream (newmark system, FP32 inner PCG, learned preconditioner, FP64 residual)",
            "bound": "hbm", "achieved": 4521.399841518282, "peak": 6803.8, "peak_kind": "measured", "unit": "GB/s",
            "frac": 0.6650877940511138, "algorithmic_bytes_per_launch": 2475361536, "avg_launch_ms": 11.247681640625,
            "iterations_per_launch": 40, "traffic": None, "note": text, "model_rule": text}
    config = {"workload": "cube96_jit_e50M_i50M", "mesh": "cube 96^3 x 6 tets, +-10% jitter", "n_tets": 5308416,
              "n_edges": 6289056, "particles": 100000000, "alive_in_timed_steps": 99995540.0, "counted": text, "species": 2,
              "dt_s": 3.572386752878211e-11, "B0_T": [0.0, 0.0, 0.2], "sort_every": 10,
              "precision": "fp32 particle path, fp64 walk test", "deposits": text,
              "l2": "flushed between timed steps: 256 MB written, then another 256 MB read (outside the step events)",
              "parallelism": "single GPU",
              "step": "sort (periodic) + push/gather/walk/deposit + implicit field step (Newmark + Gauss-law projection "
                      "+ Faraday, Jacobi-CG to 1e-10 relative residual in FP64) + fp64 residuals"}
    series = [9.711836545062922e-09] * 20 * fat
    return {"metric": bench.METRIC, "value": 4591342719.0961635, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 21.790221977233887, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic", "config": config, "roofline": dict(roof), "roofline_push": dict(roof),
            "field_solve": {"ms_per_step": 16.61, "precond": {"newmark": "learned preconditioner", "gauss": "learned"},
                            "newmark_iters": [40] * 20 * fat, "newmark_iters_mean": 40, "gauss_iters_mean": 9,
                            "max_rel_res": 7.6e-11, "learned_vs_plain": {
                                "protocol": {"text": text}, "newmark": {"learned_vs_plain_ms": 0.63, "plain": series},
                                "gauss": {"learned_vs_plain_ms": 0.71, "plain": series}}},
            "residuals": {"per_step": {"continuity_interior_rel_max": 9.7e-09, "divB_rel_max": 1.4e-15, "divB_rel": series}},
            "status": 0, "gpu_launches": 207, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [],
                                                         "samples": 33, "samples_busy": 22},
            "e2e": {"value": 1114950505.2781713, "unit": bench.UNIT, "h2d_bytes_per_step": 2964112388,
                    "d2h_bytes_per_step": 2859008004, "ms_per_step": 25.793801599740982, "overlap": text},
            "cpu_baseline": {"value": 5523943.530470847, "unit": bench.UNIT, "cores": 16, "kind": "oracle",
                             "sample": "8000000 of 50000000 particles of species 0, 4 step(s), FP64 oracle, 5.8 s",
                             "field_step": {"skipped": text}},
            "adams": {"particle_steps_per_s": 1.2e10, "ms_per_call": 0.2, "roofline": roof},
            "fp64_mode": {"particle_steps_per_s": 3.0e9, "ms_per_call": 0.7, "bound": text},
            "workloads": {"cube32_jit_e2M": {"value": 2.1e9, "unit": bench.UNIT, "ms_per_step": 0.93, "roofline": roof}}}


def test_line_is_short_and_complete():
    for fat in (1, 100):
        out = _record(fat)
        line = json.dumps(bench.headline(out))
        assert len(line) <= bench.LINE_BYTES < 3000 and "\n" not in line
        d = json.loads(line)
        for k in CONTRACT:
            assert k in d, k
        assert abs(d["value"] - out["value"]) <= 1e-6 * out["value"] and d["gpu_launches"] == 207
        assert d["e2e"]["h2d_bytes_per_step"] == 2964112388 and d["e2e"]["d2h_bytes_per_step"] == 2859008004
        assert d["clocks"]["sm_mhz"] == 2070.0 and d["clocks"]["reasons"] == []
        assert d["cpu_baseline"]["value"] > 0 and d["field_solve"]["learned_vs_plain_ms"] == {"newmark": 0.63, "gauss": 0.71}
        assert d["roofline"]["frac"] > 0 and d["workloads"]["cube32_jit_e2M"]["ms_per_step"] == 0.93


def test_line_without_the_optional_measurements():
    out = _record(1)
    for k in ("e2e", "field_solve", "adams", "fp64_mode"):
        out[k] = None
    del out["workloads"], out["cpu_baseline"]
    d = json.loads(json.dumps(bench.headline(out)))
    assert d["e2e"] is None and "field_solve" not in d and "adams" not in d and d["value"] > 0


def test_mixed_kernel_names_the_solver_that_runs():
    """Rows and entries of the cube meshes' systems (nnz about 15.5 per edge row and 13 per node row with
    PEC walls): what the sizes measured with the library showed."""
    edges = lambda n: 7 * n ** 3 + 9 * n ** 2 + 3 * n
    nodes = lambda n: (n + 1) ** 3
    for n, kern in ((4, "k_pcg_resident"), (32, "k_pcg_resident"), (36, "k_pcg_stream"), (64, "k_pcg_stream"),
                    (96, "k_pcg_stream")):
        for deg in (1, 3):
            assert bench.mixed_kernel(edges(n), int(15.5 * edges(n)), deg) == kern, (n, deg)
    for n, kern in ((32, "k_pcg_resident"), (60, "k_pcg_resident"), (72, "k_pcg_stream"), (96, "k_pcg_stream")):
        assert bench.mixed_kernel(nodes(n), 13 * nodes(n)) == kern, n

"""The line bench.py prints for its consumers, and the capture its DRAM traffic comes from (no GPU)."""
import json

import bench


def test_final_line_is_short_and_complete():
    # a full record the size a run makes, its extras far larger
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 226, "power_w_max": 1093.13, "reasons": []}
    roof = {"kernel": "k" * 80, "bound": "hbm", "achieved": 5012.3, "peak": 6680.5, "unit": "GB/s", "frac": 0.7503,
            "traffic": 1.0e9, "peak_kind": "measured", "bytes_per_site": 496, "sites_per_launch": 2 ** 21, "launch_ms": 0.2}
    rec = {"metric": bench.METRIC, "value": 6.2, "unit": "solves/s", "n_gpus": 1, "steps": 20, "warmup": 5,
           "ms_per_step": 160.0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
           "data": "synthetic", "config": {k: "v" * 40 for k in "abcdefghijk"},
           "time_to_solution_s": {"mixed": 0.16, "fp64": 0.9, "speedup": 5.6, "other_inner_formats": {"x": "y" * 3000}},
           "iterations": {"mixed": 330, "reliable_updates": 7, "fp64": 312}, "true_rel_resid": {"mixed": 9e-11, "fp64": 9e-11},
           "roofline": roof, "fp64_roofline": dict(roof), "fma_peaks": {"x": "y" * 3000}, "cg_kernels": {"x": "y" * 3000},
           "dslash": {n: {"ms": 0.15, "GB/s": 5000.1, "frac_hbm": 0.75, "GFLOP/s": 20000.1} for n in bench.GAUGE_B},
           "e2e": {"value": 2.0, "unit": "solves/s", "h2d_bytes_per_step": 2 ** 31, "d2h_bytes_per_step": 2 ** 28,
                   "clocks": clocks, "pinned_copy_gbs": {"x": "y" * 3000}}, "gpu_launches": 21000, "clocks": clocks,
           "cpu_baseline": {"value": 0.0026, "unit": "solves/s", "cores": 16, "kind": "oracle", "sample": "s" * 300,
                            "single_core": {"x": "y" * 3000}}, "extras": {"x": "y" * 20000}}
    line = json.dumps(bench.final_line(rec))
    assert len(line) < 4000
    got = json.loads(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert key in got, key
    assert set(got["e2e"]) >= {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert set(got["clocks"]) >= {"sm_mhz", "sm_max_mhz", "reasons"}


def test_traffic_is_of_the_kernel_as_it_is():
    """The bytes per site were captured from these sources; a change of the code asks for another capture."""
    assert all(t["src"] == bench.kernel_source_hash() for t in bench.NCU_TRAFFIC.values())

"""The line that the benchmark prints stays short, whatever else it measured."""
import json

import bench


def test_headline_is_short_and_whole():
    rates = {str(r): 2.7e12 / r for r in range(1, 17)}
    line = {"metric": bench.METRIC, "value": 2734567890123.456, "unit": "cell-updates/s", "n_gpus": 1, "steps": 20,
            "warmup": 5, "ms_per_step": 1.5705123456789, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "e4m3", "data": "synthetic", "gpu_launches": 320,
            "config": {"workload": "radius_sweep_16384x16384_r1-16_bernoulli0.5", "grid": [16384, 16384],
                       "radii": list(range(1, 17)), "rule": "R_r C2 M1 S0.34n..0.58n B0.34n..0.45n NM", "boundary": "zero",
                       "kernel": "tcgen05/fp8", "l2": "inputs (256 MiB per grid) larger than L2",
                       "parallelism": "replicas x1"},
            "roofline": {"bound": "hbm", "achieved": 5412.3456789, "peak": 6770.5, "unit": "GB/s", "frac": 0.7994,
                         "kernel": "ltl_tc_kernel<FP8, r >= 8>", "launch_time_source": "x" * 200, "traffic": rates},
            "e2e": {"value": 1.6e11, "unit": "cell-updates/s", "h2d_bytes_per_step": 4294967296,
                    "d2h_bytes_per_step": 4294967296, "runs_cell_updates_per_s": [1.6e11] * 3, "host_link": rates},
            "cpu_baseline": {"value": 174479508.68837774, "unit": "cell-updates/s", "cores": 16, "kind": "oracle",
                             "sample": "first 8192 rows x 16384 columns of the grid, one step per r in 1..16 (12.3 s)"},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 6},
            "per_r_cell_updates_per_s": rates, "batched": {"roofline": {k: rates for k in rates}}}
    out = bench.headline(line)
    assert len(json.dumps(line)) > 5000 and len(json.dumps(out)) < 1490
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks"):
        assert out[key] == line[key]
    assert set(out["e2e"]) == {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}

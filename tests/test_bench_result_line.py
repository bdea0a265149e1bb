"""The benchmark's result line is short, the last line and the only JSON object; the
details before it hold what it cuts."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def _full():
    """The shape of a default run: long descriptions and thousands of numbers."""
    many = {f"stage_{i}": {"bound": "hbm", "achieved": 1.0 / (i + 3), "note": "x" * 80} for i in range(60)}
    workload = "long_dna: " + "n=20000 strings over ACGT, 2000 clusters, " * 9
    roof = bench.verify_roofline(1.0e9, 0.4, 1, None, "verify_pq_kernel, " + "the merged launch of a batch " * 4,
                                 "the eager pass " * 6, 13691904)
    return {"metric": bench.METRIC, "value": 23.1e6 / 7, "unit": "pairs/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.9 / 7, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u64",
            "data": "synthetic",
            "config": {"workload": workload, "n": 20000, "Ks": [50, 150, 250], "l2": "flushed (256 MiB write)",
                       "parallelism": "single GPU", "autotune": True, "headline": "y" * 300},
            "band_cells_per_s": 1.5e15, "stage_roofline": many, "workloads": {"protein": many, "text": many},
            "roofline": roof, "recall": None, "gpu_launches": 440,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 115, "source": "z" * 200},
            "e2e": {"value": 21.7e6 / 7, "unit": "pairs/s", "ms_per_step": 1.0 / 7, "h2d_bytes_per_step": 100160008,
                    "d2h_bytes_per_step": 104328, "note": "w" * 400},
            "cpu_baseline": {"value": 140.0 / 7, "unit": "pairs/s", "cores": 1, "kind": "oracle", "all_cores": many}}


def test_result_line_is_short_last_and_alone(capsys):
    full = _full()
    bench.print_result(full)
    out = capsys.readouterr().out.splitlines()
    assert [ln for ln in out if ln.startswith("{")] == [out[-1]]
    assert len(out[-1]) < 2500
    d = json.loads(out[-1])
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "clocks", "gpu_launches", "e2e"):
        assert key in d, key
        if not isinstance(full[key], dict):
            assert d[key] == full[key]
    assert d["clocks"]["sm_mhz"] == 2070.0 and d["clocks"]["reasons"] == []
    assert d["e2e"]["value"] == full["e2e"]["value"] and d["e2e"]["d2h_bytes_per_step"] == 104328
    detail = {ln.split(" ", 2)[1]: json.loads(ln.split(" ", 2)[2]) for ln in out[:-1]}
    for k, v in full.items():
        assert (d[k] if k in d and k not in detail else detail[k]) == v, k

"""The benchmark's JSON line stays short: long curves are left out of it (they
are in the full record on stderr), the contract's figures are kept whole."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_line_leaves_out_curves_and_keeps_figures():
    if ROOT not in sys.path:
        sys.path.insert(0, ROOT)
    import bench
    record = {"metric": bench.METRIC, "value": 17715783975.928158, "unit": bench.UNIT, "n_gpus": 1, "ms_per_step":
              0.059188795, "higher_is_better": True, "vs_baseline": None, "gpu_launches": 40,
              "config": {"workload": "tracking", "G": 64}, "e2e": {"value": 18235343220.464577, "h2d_bytes_per_step": 1048576},
              "clocks": {"sm_mhz": 2070.0, "reasons": []}, "arna_n_ex": list(range(12)),
              "sharing": {"patch": {m: {"final_error_px": 0.1 + i, "n_ex": list(range(40)),
                                        "pe_eff_over_G": [0.5] * 40} for i, m in enumerate("abcdefgh")}},
              "pe_eff_recovery": {"G%d" % g: {"arna": {"at_20": 0.9, "curve": [0.123456789] * 30}} for g in range(12)}}
    line = bench.short_line(record)
    for key in ("metric", "value", "unit", "n_gpus", "ms_per_step", "higher_is_better", "vs_baseline", "gpu_launches",
                "config", "clocks", "arna_n_ex"):
        assert line[key] == record[key], key
    assert abs(line["e2e"]["value"] / record["e2e"]["value"] - 1) < 1e-5
    assert line["sharing"]["patch"]["a"] == {"final_error_px": 0.1}
    assert line["pe_eff_recovery"]["G0"]["arna"] == {"at_20": 0.9}
    assert len(json.dumps(line)) < 2000 < 8000 < len(json.dumps(record))

"""bench.py's line on stdout (no GPU): the headline whole, the other forms and workloads by their rates,
times and errors, short enough for a reader that keeps a few KB of output."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

ROOF = {"kernel": "collide_stream", "bound": "hbm", "achieved": 4094.123456789, "peak": 6779.0, "unit": "GB/s",
        "frac": 0.60417224426575061, "traffic": None, "algorithmic_per_launch": 3407872.0, "launch_ms": 0.0083206399,
        "peak_source": "measured", "executed_per_launch": 3801088.0, "executed_frac": 0.0673884647579526,
        "other_kernel_ms": {"fractional_operator": 0.010097759971395136, "collide_stream": 0.008320639915764332}}
ACC = {"rel_l2_vs_fp64_oracle": 9.7e-07, "max_node_err_rel_to_max": 2.3e-06, "lattice_steps": 200}
FORM = {"dtype": "f32+bf16x6", "value": 8108.416322509101, "unit": "MLUPS", "us_per_lattice_step": 8.08246609366504,
        "roofline": ROOF, "roofline_other": ROOF, "launch_config": "operator per-tile bn=64 ks=4, collide chunk=0",
        "accuracy": ACC, "status": "ok"}
ENTRY = dict(FORM, desc=bench.WORKLOADS["batch64"]["desc"], e2e={"value": 23809.3, "unit": "MLUPS"},
             accuracy=dict(ACC, members=[ACC] * 64), forms={"fp32": FORM, "tf32split": FORM})


def test_the_line_is_short_and_keeps_the_headline():
    walk = {"desc": "killed walk", "unit": "Mpath-steps/s", "fp32": {"value": 5.9e4}, "fp64": {"value": 945.0}}
    line = {"metric": bench.METRIC, "value": 1.0, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 1.0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32+bf16x6",
            "data": "synthetic", "config": {"workload": "mrt_aniso_512", "desc": bench.WORKLOADS["mrt_aniso_512"]["desc"]},
            "roofline": ROOF, "roofline_other": ROOF, "cpu_baseline": {"value": 70.0, "unit": "MLUPS"},
            "accuracy": dict(ACC, by_horizon={str(k): ACC for k in range(9)}),
            "forms": {k: FORM for k in bench.HEADLINE_FORMS},
            "workloads": dict({k: ENTRY for k in bench.EXTRA_WORKLOADS}, levy_walk=walk, broken={"error": "E: x"}),
            "e2e": {"value": 2.0, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
            "gpu_launches": 200000, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}, "status": "ok"}
    full, out = json.dumps(line), bench.result_line(line)
    assert len(json.dumps(out)) < 6000 < len(full)
    for k in line:
        if k not in ("forms", "workloads", "accuracy"):
            assert out[k] == line[k], k
    assert out["accuracy"] == ACC
    assert set(out["forms"]) == set(line["forms"]) and set(out["workloads"]) == set(line["workloads"])
    assert out["workloads"]["batch64"]["value"] == ENTRY["value"]
    assert out["workloads"]["batch64"]["e2e"] == 23809.3
    assert out["workloads"]["levy_walk"]["fp64"]["value"] == 945.0
    assert out["workloads"]["broken"] == {"error": "E: x"}
    assert json.loads(full) == line  # (the record itself is not changed)

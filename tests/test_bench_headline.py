"""The benchmark's line on standard output stays short whatever the legs
report (a reader of the end of a log still gets all of it), and keeps every
field that says what was measured and how.  No GPU is touched."""
import json

import bench


def test_line_keeps_the_contract_and_drops_the_sweeps():
    sweep = [{"n": i, "ms": i * 0.1, "offload": bool(i % 2)} for i in range(400)]
    report = {
        "metric": bench.METRIC, "value": 803.9, "unit": "Gkeys/s", "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 0.33, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int64",
        "data": "synthetic", "gpu_launches": 120,
        "config": {"workload": "topk", "n": 1 << 28, "k": 1000, "l2": "inputs larger than L2"},
        "roofline": {"bound": "hbm", "achieved": 6900.0, "frac": 1.0, "kernel_ms": 0.3, "last_launch": sweep},
        "e2e": {"value": 26.0, "unit": "Gkeys/s", "h2d_bytes_per_step": 1 << 31, "d2h_bytes_per_step": 12004,
                "keys_only": {"value": 1}},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
        "join": {"value": 90.0, "unit": "Gprobes/s", "ms_per_step": 3.0, "cells": sweep},
        "gate": {"unit": "relative error", "cells": sweep}, "serving": {"value": 2.0, "unit": "ms", "gated": sweep},
        "cpu_baseline": {"value": 0.01, "unit": "Gkeys/s", "cores": 1, "kind": "oracle", "host": sweep},
    }
    line = bench.headline(report)
    assert len(json.dumps(line)) < 2500
    for key, v in report.items():
        if not isinstance(v, dict):
            assert line[key] == v
    assert line["config"] == report["config"] and line["clocks"] == report["clocks"]
    assert {k: line["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")} == \
        {k: report["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")}
    assert line["join"] == {"value": 90.0, "unit": "Gprobes/s", "ms_per_step": 3.0}
    assert "gate" not in line and "last_launch" not in line["roofline"]

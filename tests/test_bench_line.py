"""The default benchmark run prints one short line: the keys that its readers need,
and a value for every nested workload; the rest goes to stderr."""
from __future__ import annotations

import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_printed_line_is_short():
    import bench

    bulky = [{"beta": b, "note": "x" * 400} for b in range(20)]
    line = {k: {"value": 1.25} for k in bench.CONTRACT}
    line.update(metric="LDD GTEPS", value=229.05030377446545, unit="GTEPS", per_beta=bulky,
                parity={"text": "y" * 4000})
    nested = {name: dict(line, value=1.0 / 3, ms_per_step=2.0 / 3, per_beta=bulky)
              for name, _, _ in bench.EXTRAS}
    out = bench.short(line, nested)
    assert len(json.dumps(out)) < 3000
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
              "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "clocks",
              "e2e", "gpu_launches"):
        assert out[k] == line[k]
    assert set(out["workloads"]) == set(nested)
    assert all(x["value"] == 1.0 / 3 for x in out["workloads"].values())

"""The bench's line on standard output holds the headline's fields and stays short, however much is measured beside it."""
import json

import bench


def test_headline():
    line = {k: 1 for k in bench.HEADLINE}
    line["config"] = {"workload": "w" * 60, "mach": "m" * 60, "motion": "p" * 60, "l2": "l" * 110, "nodes": 4056108, "parallelism": "single GPU"}
    line["precision"], line["metric"] = "f" * 90, "u" * 90
    line["clocks"] = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 100}
    line["roofline"] = {"bound": "hbm", "kernel": "k_stream_fast", "achieved": 2280.69313400667, "peak": 6748.3, "unit": "GB/s", "frac": 0.33,
                        "peak_source": "measured", "traffic": 962600000.0, "note": "n" * 300}
    line["step_roofline"] = None
    line["e2e"] = {"value": 1438.85, "unit": "M node-updates/s", "h2d_bytes_per_step": 292039776, "d2h_bytes_per_step": 292039776,
                   "steps": 10, "note": "n" * 300}
    line["cpu_baseline"] = {"value": 1.0, "unit": "u", "cores": 16, "kind": "oracle", "cpu_model": "Neoverse-V2", "sample": "s" * 400}
    line["precision_study"] = {"rows": list(range(2000))}
    out = json.loads(json.dumps(bench.headline(line)))
    assert len(json.dumps(out)) < 2000
    assert all(out[k] == line[k] for k in bench.HEADLINE)
    assert out["e2e"] == {k: v for k, v in line["e2e"].items() if k != "note"} and out["step_roofline"] is None
    assert out["roofline"]["frac"] == 0.33 and out["cpu_baseline"]["cores"] == 16

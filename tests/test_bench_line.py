"""The line that bench.py prints stays short whatever its tables hold, and keeps the figures."""
import json

import bench


def test_the_printed_line_is_short_and_keeps_the_figures():
    x = 1234.5678901234567
    job = {k: x for k in bench.JOB_KEYS} | {"field": "zero_slabs", "variants": [0.25 / 3] * 4, "bytes": 10 ** 9,
                                            "eb": 1e-3 / 3, "step": x, "nrmse": x, "bit_rate": x}
    rows = [{f"{a}_{b}": x for a in ("cr", "compress_gbs", "decompress_gbs") for b in range(6)}] * 6
    record = {"metric": bench.METRIC, "value": 3246.361512345, "unit": "GB/s", "steps": 100,
              "e2e": {"value": 243.31912345, "h2d_bytes_per_step": 1583802972}, "gpu_launches": 3000,
              "clocks": {"sm_mhz": 2070.0, "reasons": []}, "jobs": [job] * 6,
              "ablation": {"cr": rows, "single_vs_multipass": rows, "single_pass_speedup_geomean": x},
              "tiles": {"rows": rows, "vs_32x8": {"64x8": {"win": 3}}},
              "batched": {"compress": {"batched_gbs": x}, "tuning_ms": {str(k) * 40: x for k in range(48)}},
              "serving": None}
    text = json.dumps(bench.printed_line(record))
    line = json.loads(text)
    assert len(text) < 4096 and "\n" not in text
    assert line["value"] == 3246.36 and line["e2e"]["h2d_bytes_per_step"] == 1583802972
    assert line["clocks"] == {"sm_mhz": 2070.0, "reasons": []} and line["gpu_launches"] == 3000
    assert [j["cr"] for j in line["jobs"]] == [1234.57] * 6
    assert line["batched"] == {"compress": {"batched_gbs": 1234.57}} and line["serving"] is None
    assert line["tiles"] == {"vs_32x8": {"64x8": {"win": 3}}}
    assert record["tiles"]["rows"] == rows and record["value"] == 3246.361512345   # the record is whole

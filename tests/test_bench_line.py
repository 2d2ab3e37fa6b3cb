"""The benchmark's printed line: short enough to be read back from the end of a
program's output, with every key that its readers use."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def _line():
    point = {"mech": "ldg", "cta": 256, "grid": 608, "status": 0, "resident_per_sm": 8, "gbs_median": 4402.7,
             "steps_gbs_median": 7005.7, "k": 1, "cop": 0, "order": 0, "frac_of_datasheet": 0.5503,
             "frac_of_measured_copy": 0.6593, "checksum_ok": True}
    curves = [{**point, "mech": m, "k": k, "gbs_median": 4000.0 + 100 * k} for m in ("ldg", "cpasync", "tma", "ldg32")
              for k in range(1, 35)] + [{"mech": "tma", "status": 4, "gbs_median": None}]
    prec = {"parity": True, "value": 7538.0, "per_payload": [
        {"payload": d, "best": point, "points": [dict(point) for _ in range(34)]} for d in ("f32", "bf16", "fp8", "x")]}
    return {"metric": bench.METRIC, "value": 7673.1, "unit": "GB/s", "n_gpus": 1, "steps": 50, "e2e": {"value": 211.0},
            "clocks": {"sm_mhz": 2070}, "gpu_launches": 50, "curves": curves, "precision": prec, "batched": {"a": 1}}


def test_printed_line_is_short_and_complete():
    line = _line()
    full = json.dumps(line)
    out = bench.printed(line)
    text = json.dumps(out, separators=(",", ":"))
    assert len(full) > 60000 > 16384 > len(text) and "\n" not in text
    assert set(out) == set(line)
    for key in set(line) - {"curves", "precision"}:
        assert out[key] == line[key]
    assert out["curves"]["ldg"]["k"] == 34 and out["curves"]["ldg"]["points"] == 34
    assert out["curves"]["tma"]["points"] == 35 and out["curves"]["tma"]["gbs_median"] == 7400.0
    assert out["precision"]["per_payload"][1]["points"] == 34 and out["precision"]["parity"]
    assert json.dumps(line) == full  # what goes to the file keeps every point

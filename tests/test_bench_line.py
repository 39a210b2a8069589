"""The printed line of bench.py (no GPU): valid JSON with the values to six digits, the headline's rooflines whole and the
nested ones without what they repeat."""
import json

import bench


def test_line_keeps_values_and_drops_repetitions():
    pk = {"hbm_gbs": 6781.1, "source": "measured (MEASURED_PEAKS.json)"}
    roof = bench.roofline("k", 6.78e9, 3.0, 3, pk, alg_flops=2.0e12)
    line = {"metric": "m", "value": 995.3896638079177, "vs_baseline": None, "steps": 20, "higher_is_better": True,
            "rel_err": {"df32": 3.050759670657366e-14}, "roofline": roof, "bytes": 1663008768,
            "cfg": {"cells": 32768, "df32": {"ms_per_step": 0.04396960008889437, "roofline": roof}}, "list": [1.23456789, "a"]}
    text = bench.line_text(line)
    assert "\n" not in text and len(text) < len(json.dumps(line))
    got = json.loads(text)
    assert got["value"] == 995.39 and got["vs_baseline"] is None and got["steps"] == 20 and got["higher_is_better"] is True
    assert got["rel_err"]["df32"] == 3.05076e-14 and got["bytes"] == 1663008768 and got["list"] == [1.23457, "a"]
    assert set(got["roofline"]) == set(roof) and got["roofline"]["peak"] == 6781.1
    nested = got["cfg"]["df32"]["roofline"]
    assert nested["frac"] == float(f"{roof['frac']:.6g}") and nested["kernel"] == "k" and "peak" not in nested
    assert got["cfg"]["df32"]["ms_per_step"] == 0.0439696

"""The benchmark prints its record as JSON: a strict parser reads it back whatever the record holds."""
import json
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench


def strict(text):
    def refuse(word):
        raise ValueError(word)
    return json.loads(text, parse_constant=refuse)


def test_line_is_json_with_values_that_are_not_numbers():
    record = {"value": 1.5, "final_marg_err": float("nan"), "vs_baseline": None, "dtype": "f64", "n": 3, "ok": True,
              "workloads": [{"final_marg_err": np.float64("nan"), "x": (float("inf"), -2.0)}]}
    line = bench.json_line(record)
    assert "\n" not in line
    back = strict(line)
    assert back["value"] == 1.5 and back["final_marg_err"] is None and back["n"] == 3 and back["ok"] is True
    assert back["workloads"] == [{"final_marg_err": None, "x": [None, -2.0]}]


def test_every_record_is_printed_through_it():
    src = open(bench.__file__).read()
    prints = [ln.strip() for ln in src.splitlines() if "print(" in ln and "json" in ln]
    assert prints and all("json_line(" in ln or "dumps({" in ln for ln in prints), prints

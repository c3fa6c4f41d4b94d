"""The bench's JSON line stays short enough to be read whole: rows in short on the line, in full
on stderr; the contract's keys untouched."""

import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench  # noqa: E402

CONTRACT = {"metric": "m" * 90, "value": 69970737783.85143, "unit": "cells/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.022478882598876954, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic", "config": {"workload": "w" * 600},
            "e2e": {"value": 5129254099.935753, "unit": "cells/s", "h2d_bytes_per_step": 58021148,
                    "d2h_bytes_per_step": 25165824}, "gpu_launches": 20,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}, "roofline": {"kernel": "k" * 2500}}
ROWS = {f"row_of_a_path_with_a_long_name_{i}": {"ms_per_launch": 0.159761234, "hbm_frac_of_measured": 0.12445470766,
        "rel_maxnorm_err_vs_oracle": 3.0667725924530164e-16, "timing": "x" * 600, "cells": 1572864} for i in range(25)}
ROWS["pcg"] = {"ms_per_solve": 30.70660800000269, "iterations": 259, "rel_residual": 9.4e-9}
ROWS["serving"] = {"requests": 500, "poisson": {"p50_ms": 0.40032679413570804, "p99_ms": 1.539765821789274,
                                                "req_per_s": 19359.363055272996}, "rate_sweep": [1] * 500}
ROWS["sweep"] = {str(1 << e): {"cells_per_s": 1.9e10, "ms": 0.003419123} for e in range(16, 24)}
ROWS["failed"] = {"error": "RuntimeError('" + "y" * 250 + "')"}


def test_line_is_short_and_whole(capsys):
    bench.print_line(dict(CONTRACT, rows=ROWS))
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) <= bench.LINE_LIMIT
    line = json.loads(out)
    for k, v in CONTRACT.items():
        assert line[k] == v, k
    r = line["rows"]
    assert set(r) == set(ROWS)
    assert r["row_of_a_path_with_a_long_name_3"] == {"ms": 0.1598, "frac": 0.1245, "err": 3.067e-16}
    assert r["pcg"] == {"ms": 30.71, "iters": 259}
    assert r["serving"] == {"p50_ms": 0.4003, "p99_ms": 1.54, "req_per_s": 19360.0}
    assert r["sweep"]["65536"] == 0.003419 and len(r["failed"]["error"]) == 80
    full = {ln.split(" ", 3)[2]: json.loads(ln.split(" ", 3)[3]) for ln in err.strip().split("\n")}
    assert full == ROWS


def test_no_number_of_rows_makes_it_long(capsys):
    bench.print_line(dict(CONTRACT, rows={f"{k}_{i}": v for k, v in ROWS.items() for i in range(20)}))
    out = capsys.readouterr().out
    assert len(out) <= bench.LINE_LIMIT and json.loads(out)["value"] == CONTRACT["value"]

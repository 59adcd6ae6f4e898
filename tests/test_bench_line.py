"""The benchmark's printed line stays short however long its whole result is: it carries the contract's
keys and names the file with the rest."""
import json

import bench


def _result():
    long = {"candidates": [{"shape": i, "ms": 1.0 / (i + 1), "note": "x" * 200} for i in range(200)]}
    variants = {v: {"value": 1e8, "kernel_ms": 8.0, "meets_stated_error": True, "stated_error_T": 1e-5,
                    "error_vs_fp64_gpu": {"max_rel_T": 1e-9, "max_abs_Y": 1e-9}, "roofline_frac": 0.5, "table": long}
                for v in ("fp64", "mixed", "hybrid")}
    result = {k: 1.0 for k in bench.HEADLINE_KEYS if k != "impl"}
    result |= {"config": {"workload": bench.WORKLOAD, "variant": "hybrid"}, "roofline": {"frac": 0.5, "note": "y" * 250},
               "e2e": {"value": 1.0, "unit": "cells/s", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
               "variants": variants, "surrogate": long, "shock_bubble": long, "reactors_4096": {"ms": 1.5},
               "amr_batch": {"fp64": {"persistent_ms": 179.0, "autotuned": long}, "mixed": None}}
    return result


def test_line_is_short_and_complete(tmp_path):
    result = _result()
    path = str(tmp_path / "detail.json")
    text = json.dumps(bench.headline(result, bench.write_detail(result, path)))
    assert len(json.dumps(result)) > 100000 and len(text) < 3000
    line = json.loads(text)
    for k in bench.HEADLINE_KEYS:
        assert k == "impl" or line[k] == result[k], k
    assert line["legs"] == {"reactors_4096_fp64_ms": 1.5, "amr_256_boxes_fp64_ms": 179.0}
    assert line["detail"] == path and json.load(open(path)) == result


def test_unwritable_detail_is_no_failure(tmp_path):
    assert bench.write_detail(_result(), str(tmp_path / "no" / "such" / "folder.json")) is None

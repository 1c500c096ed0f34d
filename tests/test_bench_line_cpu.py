"""The bench's sections on its one line: a few figures each, so that the line fits
readers that keep the last 3000 characters."""
import json

import bench


def test_sections_in_short():
    long = 1234.567890123456789
    rates = {f"{r:g}": {f"field {i}": long for i in range(12)} for r in (1e4, 1e5, 1e6, 2e6, 4e6, 8e6)}
    serving = {"rates": rates, "saturation": {"max_sustained_gbps": long, "saturated_at_rate": 2e6, "rule": "x" * 200}}
    row = {"hbm_frac": 0.912345678, "l2_resident": False, "config": "x" * 100}
    sections = {
        "batched": {"workload": "x" * 300, "persistent_graph": {"gbps": long, "hbm_frac": 0.67123456, "variant": 9,
                                                              "ms": long}},
        "serving": serving, "serving_host": serving,
        "shortened": {"hbm_frac_min": 0.41234567, "hbm_frac_mean": 0.5, "hbm_frac_max": 0.7, "grid": [row] * 45},
        "secded": {"codes": {str(n): {"secded_hbm_frac": 0.87654321, "plain_us": long} for n in (15, 31, 63, 127, 255)}},
        "per_code": {"rows": [dict(row, hbm_frac=f) for f in (0.95, 0.71234567)] + [dict(row, l2_resident=True)]},
        "adt": {"codes": {str(n): {"speedup": 1.57015107} for n in (15, 31, 63)}},
    }
    got = bench.section_summary(sections)
    assert set(got) == set(sections)
    assert got["batched"] == {"gbps": 1235.0, "hbm_frac": 0.6712, "variant": 9}
    assert got["serving"] == {"max_sustained_gbps": 1235.0, "saturated_at_rate": 2e6}
    assert got["secded"]["255"] == 0.8765 and got["adt"]["15"] == 1.57
    assert got["per_code"] == {"hbm_frac_min": 0.7123, "hbm_frac_max": 0.95}
    assert len(json.dumps(got)) < 800


def test_sections_that_did_not_run():
    assert bench.section_summary({"batched": None, "serving": None, "secded": None, "adt": None}) == {}

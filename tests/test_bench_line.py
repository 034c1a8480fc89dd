"""The benchmark's printed line stays short: descriptions and tables go to the
record on stderr, the headline's figures stay as they are."""
import json

import bench


def test_line_is_short_and_exact(capsys):
    leg = {"workload": "w" * 300, "ms_per_step": 1.0 / 3.0, "unit": "words/s",
           "accuracy": {"max_dz_rel": 1.23456789e-15, "reading": "r" * 200}}
    line = {"metric": bench.METRIC, "value": 1.0e12 / 3.0, "unit": "words/s", "n_gpus": 1,
            "ms_per_step": 10.0 / 3.0, "config": {"workload": "c" * 120}, "lod": dict(
                leg, valid_settings=[{"margin": -0.4, "ms": 1.5}] * 100, per_group=[leg] * 16)}
    line.update({f"leg{k}": leg for k in range(12)}, paper_scan=leg, multiseed=leg)
    bench.print_line(line)
    out, err = capsys.readouterr()
    assert json.loads(err) == line
    assert out.count("\n") == 1 and len(out) < 4000
    got = json.loads(out)
    for k in ("metric", "value", "unit", "n_gpus", "ms_per_step", "config"):
        assert got[k] == line[k]
    assert got["leg0"] == {"ms_per_step": 0.333333, "unit": "words/s",
                           "accuracy": {"max_dz_rel": 1.23457e-15}}
    assert "paper_scan" not in got and "valid_settings" not in got["lod"]

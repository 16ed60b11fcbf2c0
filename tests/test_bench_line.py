"""bench.py's result stays one short JSON line on stdout: the extras (tables of
many thousand characters) go to stderr, and floats carry seven digits."""
import json

import pytest

pytest.importorskip("torch")


def test_extras_do_not_lengthen_the_line(capsys):
    import bench
    line = {"metric": "m", "value": 2.0 / 3.0, "clocks": {"sm_mhz": 2070.0, "reasons": []}, "n": 3, "none": None,
            "list": [1.0 / 3.0, True]}
    extras = {"rows": [{"x": k / 7.0} for k in range(2000)]}
    bench.report(line, extras)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) < 300
    got = json.loads(out)
    assert got["value"] == pytest.approx(2.0 / 3.0, rel=1e-6) and got["list"][1] is True and got["n"] == 3
    assert json.loads(err)["extras"]["rows"][1999]["x"] == pytest.approx(1999 / 7.0, rel=1e-6)


def test_full_line_fits(capsys):
    import bench
    from paper_2603_12550_gb300 import inputs
    n = 1.0 / 3.0
    roof = {k: n for k in ("achieved", "peak", "frac", "launch_ms", "traffic")}
    line = {"config": bench._config(inputs.WORKLOADS[bench.WORKLOAD], n), "metric": bench.METRIC,
            "roofline": [roof, roof], "cpu_baseline": "x" * 300, "text": "y" * 700}
    bench.report(line)
    assert len(capsys.readouterr().out) < 2800

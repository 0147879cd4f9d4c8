"""bench.py's result lines say what was run (no GPU)."""
import argparse
import json

import bench


def test_the_oracle_arm_names_its_own_arithmetic(monkeypatch, capsys):
    """The oracle computes in plain FP64 on the host: its line must not carry the description of the
    GPU's pairs."""
    monkeypatch.setattr(bench, "cpu_oracle_rate", lambda steps=1, threads=1: (1.0e7, 1.0e-3, 4))
    bench.run_reference(argparse.Namespace(gpus=1, steps=1, warmup=0))
    line = json.loads(capsys.readouterr().out)
    assert line["impl"] == "reference" and line["dtype"] == "f64"
    assert line["arithmetic"].startswith("FP64") and "pairs" not in line["arithmetic"]

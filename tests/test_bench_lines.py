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


def test_captured_counters_are_only_given_for_the_captured_kernel(monkeypatch, tmp_path):
    """Instruction and traffic figures of an ncu capture hold for that kernel and that source."""
    src = tmp_path / "head.cuh"
    src.write_text("kernel")
    import hashlib
    sha = hashlib.sha256(b"kernel").hexdigest()[:16]
    monkeypatch.setattr(bench, "HEAD_SOURCE", str(src))
    monkeypatch.setattr(bench, "HEAD_CAPTURE", dict(bench.HEAD_CAPTURE, kernel="k<double>", source_sha16=sha))
    assert bench.head_capture("k<double>") is bench.HEAD_CAPTURE
    assert bench.head_capture("k<float>") is None and bench.head_capture(None) is None
    src.write_text("another kernel")
    assert bench.head_capture("k<double>") is None


def test_no_kernel_name_without_a_profile():
    def fails():
        raise RuntimeError
    assert bench.dominant_kernel(fails) is None

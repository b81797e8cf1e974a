"""bench.py's traffic record belongs to one form: the forms' kernels share their timer
names, and a form without a capture reports none."""
import hashlib
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_records_are_by_form(tmp_path, monkeypatch):
    import bench
    src = tmp_path / "k.cu"
    src.write_text("kernel")
    rec = {"bytes_per_launch": 30e6, "sources": ["k.cu"], "source_sha": hashlib.sha256(b"kernel").hexdigest()[:16]}
    os.mkdir(tmp_path / "profiles")
    json.dump({"fp16x3": {"fwd_tc": rec}}, open(tmp_path / "profiles" / "traffic.json", "w"))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    units = 999600 * 256 * 256
    kprof = {"fwd_tc": (4.81, 10), "adj_tc": (4.45, 10)}
    assert bench.roofline(kprof, units, 2, 1.5, "fp16x3")["traffic"] == 30e6
    assert bench.roofline(kprof, units, 2, 3.0, "bf16x3")["traffic"] is None
    assert bench._traffic("adj_tc", "fp16x3") is None
    src.write_text("another kernel")
    assert bench._traffic("fwd_tc", "fp16x3") is None


def test_committed_records():
    rec = json.load(open(os.path.join(ROOT, "profiles", "traffic.json")))
    for form, kernels in rec.items():
        if form == "_about":
            continue
        for k in kernels.values():
            assert form in k["capture"] and os.path.exists(os.path.join(ROOT, k["capture"]))

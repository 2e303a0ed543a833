"""Figures that bench.py takes from a committed profiler capture hold only for the kernel sources it was taken from."""
import hashlib
import json

import bench


def write(tmp_path, **doc):
    (tmp_path / "profiles").mkdir(exist_ok=True)
    (tmp_path / "k.cuh").write_bytes(b"kernel")
    doc.update(sources=["k.cuh"], sources_sha256=hashlib.sha256(b"kernel").hexdigest())
    for name in ("fp64_alu.json", "roofline_traffic.json"):
        (tmp_path / "profiles" / name).write_text(json.dumps(doc))


def test_counts_of_other_sources_are_not_used(tmp_path, monkeypatch):
    write(tmp_path, kernel="k", fp64_flops_per_lup=2, fp64_instructions_per_lup=1, dram_bytes_per_step=7)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.fp64_alu_counts() == (2.0, 1.0)
    assert bench.captured_traffic("k") == 7 and bench.captured_traffic("other") is None
    (tmp_path / "k.cuh").write_bytes(b"another kernel")
    assert bench.fp64_alu_counts() is None and bench.captured_traffic("k") is None

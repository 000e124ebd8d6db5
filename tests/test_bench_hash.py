"""The stamp that ties the committed traffic profile to the kernel's sources."""
import importlib.util
import os
import shutil

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_hash_covers_every_source_of_the_screen(tmp_path, monkeypatch):
    spec = importlib.util.spec_from_file_location("bench_hash", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    src = os.path.join(ROOT, "paper_1302_0435_gb300", "csrc")
    dst = tmp_path / "paper_1302_0435_gb300" / "csrc"
    shutil.copytree(src, dst)
    here = bench.kernel_source_hash()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_source_hash() == here
    units = [f for f in os.listdir(dst) if f.startswith("d2_lane")]
    assert "d2_lane_a8.cu" in units
    for f in units + ["d2_solve.cuh", "d2_solver.cuh", "d2_internal.h"]:
        text = (dst / f).read_bytes()
        (dst / f).write_bytes(text + b"\n")
        assert bench.kernel_source_hash() != here, f
        (dst / f).write_bytes(text)

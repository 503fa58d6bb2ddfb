"""The committed counters are keyed by a hash of the sources that decide which
kernel a plan launches: the size rule of variant 0 is among them."""
import importlib.util
import os
import shutil

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join("paper_2603_25282_gb300", "csrc")


def test_size_rule_is_hashed(tmp_path, monkeypatch):
    spec = importlib.util.spec_from_file_location("bench_counters_mod", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    shutil.copytree(os.path.join(ROOT, CSRC), tmp_path / CSRC)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench.csrc_hash()
    # the file that says up to how many points a 2D grid takes the split passes
    rule = [f for f in (tmp_path / CSRC).iterdir() if "dim == 2 ? 3LL << 16" in f.read_text()]
    assert len(rule) == 1
    rule[0].write_text(rule[0].read_text().replace("3LL << 16", "3LL << 15"))
    assert bench.csrc_hash() != before

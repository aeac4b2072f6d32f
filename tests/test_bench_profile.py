"""Where bench.py applies the committed ncu record of the target-walk kernel.  CPU only."""
import argparse
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


@pytest.fixture
def bench(monkeypatch, tmp_path):
    import bench as b
    rec = {"kernel_sources_sha256": b.kernel_source_sha256(), "dram_bytes_per_launch": 20,
           "target_steps_of_launch": 10, "l2_sectors_from_l1_of_launch": 5}
    path = tmp_path / "record.json"
    path.write_text(json.dumps(rec))
    monkeypatch.setattr(b, "PROFILE", str(path))
    return b


@pytest.mark.parametrize("layout,literal,warmup,applies", [
    ("narrow", False, False, True), ("wide", False, False, False), ("csr", False, False, False),
    ("narrow", True, False, False), ("narrow", False, True, False)])
def test_record_is_of_the_default_run(bench, layout, literal, warmup, applies):
    args = argparse.Namespace(literal_shuffle=literal, warmup_rule=warmup)
    assert bench.recorded_l2_sectors(args, layout) == (0.5 if applies else None)
    assert bench.recorded_traffic(args, layout) == (2.0 if applies else None)
    assert bench.kernel_name(args) == ("k_target_walks" if literal else "k_lockstep")


def test_record_follows_all_sources_of_the_reads(bench, monkeypatch, tmp_path):
    args = argparse.Namespace(literal_shuffle=False, warmup_rule=False)
    csrc = os.path.join(ROOT, "paper_2304_04015_gb300", "csrc")
    fake = tmp_path / "paper_2304_04015_gb300" / "csrc"
    fake.mkdir(parents=True)
    names = ("srk_lockstep.cu", "srk_device.cuh", "srk_internal.h", "srk_source.cu", "srk_graph.cu")
    for name in names:
        (fake / name).write_text(open(os.path.join(csrc, name)).read())
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    for name in names:
        text = (fake / name).read_text()
        (fake / name).write_text("// a comment\n" + text)
        assert bench.recorded_l2_sectors(args, "narrow") == 0.5, name
        (fake / name).write_text("int changed;\n" + text)
        assert bench.recorded_l2_sectors(args, "narrow") is None, name
        (fake / name).write_text(text)

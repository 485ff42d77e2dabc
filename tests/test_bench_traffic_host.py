"""The benchmark's traffic figure belongs to the kernel its roofline names: it comes from that kernel's
capture, and a change of any of the kernel's sources withdraws it."""
import hashlib
import os
import re
import shutil

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = ("pair_tc.cu", "tc_device.cuh", "sis_device.cuh")


@pytest.fixture()
def tree(tmp_path, monkeypatch):
    import bench
    kernel = re.search(r'"bound": "tensor", "kernel": "(\w+)"', open(os.path.join(ROOT, "bench.py")).read()).group(1)
    csrc = tmp_path / "paper_2410_01752_gb300" / "csrc"
    csrc.mkdir(parents=True)
    (tmp_path / "profiles").mkdir()
    for f in os.listdir(os.path.join(ROOT, "paper_2410_01752_gb300", "csrc")):
        shutil.copy(os.path.join(ROOT, "paper_2410_01752_gb300", "csrc", f), csrc / f)
    sha = hashlib.sha256(b"".join((csrc / f).read_bytes() for f in SOURCES)).hexdigest()
    (tmp_path / "profiles" / f"{kernel}_rung3_N1000_d10_traffic.md").write_text(
        f"traffic_bytes_per_launch: 12345\nsource_sha256 (at capture): {sha}\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    return bench, csrc


def test_traffic_of_the_named_kernel(tree):
    bench, _ = tree
    assert bench.captured_traffic() == 12345


@pytest.mark.parametrize("source", SOURCES)
def test_a_changed_source_withdraws_it(tree, source):
    bench, csrc = tree
    with open(csrc / source, "a") as f:
        f.write("// changed\n")
    assert bench.captured_traffic() is None

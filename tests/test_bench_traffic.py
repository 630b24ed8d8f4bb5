"""The bench's DRAM traffic record counts only for the sources it was captured
on: the (re, im) passes' file, and for the fused form every source of the wide
pass (body, launches, op-loop generator)."""
import hashlib
import json
import os
import shutil

import pytest

import bench

SOURCES = ["qs_fused.cu", "qs_wide_device.cuh", "qs_wide.cu", "gen_op_loop.py"]


@pytest.fixture
def tree(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_1608_00263_gb300" / "csrc"
    csrc.mkdir(parents=True)
    (tmp_path / "profiles").mkdir()
    for name in SOURCES:
        shutil.copy(os.path.join(bench.ROOT, "paper_1608_00263_gb300", "csrc", name), str(csrc))
    sha = lambda names: hashlib.sha1(b"".join((csrc / n).read_bytes() for n in names)).hexdigest()
    rec = {"qubits": 28, "bytes_per_launch": 2.0 ** 32, "launch": "a pass", "source_sha1": sha(SOURCES[:1])}
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps(
        {"fused": dict(rec, wide_sha1=sha(SOURCES[1:])), "tc": rec}))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    return csrc


def test_current_sources(tree):
    assert bench.load_traffic("fused", 30) == (2.0 ** 34, "a pass")
    assert bench.load_traffic("tc", 28) == (2.0 ** 32, "a pass")


@pytest.mark.parametrize("name", SOURCES)
def test_a_changed_source_voids_the_record(tree, name):
    with open(tree / name, "a") as f:
        f.write("\n")
    assert bench.load_traffic("fused", 30) is None
    assert (bench.load_traffic("tc", 30) is None) == (name == "qs_fused.cu")

"""The recorded DRAM and issue figures of the sweep kernel hold only for the
sources, the workload and the launch shape that they were taken with."""
import hashlib
import os
import re
import sys
from types import SimpleNamespace

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_1704_01888_gb300", "csrc")


def _included(name, seen):
    if name not in seen and os.path.exists(os.path.join(CSRC, name)):
        seen.add(name)
        for inner in re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, name)).read()):
            _included(inner, seen)
    return seen


def test_the_record_covers_every_source_of_the_kernel():
    joined = bench._sweep_sources()
    for name in _included("pa_sweep.cu", set()):
        assert open(os.path.join(CSRC, name), "rb").read() in joined, name


def test_the_record_holds_for_its_case_and_launch_alone(tmp_path, monkeypatch):
    os.makedirs(tmp_path / "profiles")
    sources = bench._sweep_sources()
    text = "case: q10-L64\nlaunch: 48,512,304  (replicas, threads, blocks)\ndram_bytes_per_replica: 3191.5\n"
    (tmp_path / "profiles" / "sweep_traffic.txt").write_text(
        text + f"source_sha256: {hashlib.sha256(sources).hexdigest()}\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setattr(bench, "_sweep_sources", lambda: sources)
    w = SimpleNamespace(q=10, L=64)
    assert bench._sweep_record(w, (48, 512, 304)) == {"dram_bytes_per_replica": 3191.5}
    assert bench._sweep_record(w, (44, 512, 304)) is None
    assert bench._sweep_record(SimpleNamespace(q=10, L=32), (48, 512, 304)) is None
    monkeypatch.setattr(bench, "_sweep_sources", lambda: sources + b" ")
    assert bench._sweep_record(w, (48, 512, 304)) is None

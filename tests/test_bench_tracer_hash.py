"""The recorded tracer counters of the bench hold for the sources they were measured with: the hash changes
with the tracer, the grid's construction and every constant and rule of the default cells, and not with
the rest of the API."""
import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

CSRC = os.path.join("paper_2501_05828_gb300", "csrc")


def sha(monkeypatch, tmp_path, edits):
    """tracer_sha of a copy of the sources with the (file, old, new) edits."""
    dst = tmp_path / str(len(list(tmp_path.iterdir())))
    shutil.copytree(os.path.join(ROOT, CSRC), dst / CSRC)
    for name, old, new in edits:
        p = dst / CSRC / name
        text = p.read_text()
        assert text.count(old) >= 1, old
        p.write_text(text.replace(old, new, 1))
    monkeypatch.setattr(bench, "ROOT", str(dst))
    return bench.tracer_sha()


@pytest.mark.parametrize("name,old,new", [
    ("ur_api.cu", "kCellSlab = {{9.f", "kCellSlab = {{8.f"),
    ("ur_api.cu", "kCellRough = {{4.f", "kCellRough = {{5.f"),
    ("ur_api.cu", "kCellIso = {{14.f", "kCellIso = {{13.f"),
    ("ur_api.cu", "kCellFine[3] = {0.5f", "kCellFine[3] = {0.6f"),
    ("ur_api.cu", "kCoarseCell = 16.f", "kCoarseCell = 17.f"),
    ("ur_api.cu", "std::pow(rule.density / density, rule.power)", "std::pow(rule.density / density, 0.4f)"),
    ("ur_api.cu", "sd.density = (float)((double)n / box)", "sd.density = (float)((double)n / box / 2)"),
    ("ur_trace.cuh", "kIdleMin = 18", "kIdleMin = 17"),
    ("ur_grid.cu", "kScanPer = 4", "kScanPer = 8"),
])
def test_hash_follows_what_sets_the_counters(monkeypatch, tmp_path, name, old, new):
    same = sha(monkeypatch, tmp_path, [])
    assert sha(monkeypatch, tmp_path, [(name, old, new)]) != same


def test_hash_leaves_the_rest_of_the_api_out(monkeypatch, tmp_path):
    same = sha(monkeypatch, tmp_path, [])
    assert sha(monkeypatch, tmp_path, [("ur_api.cu", "bad device index", "no such device")]) == same

"""bench.py's kernel source hash covers the kernel that runs, and a capture of
one precision's kernel is not quoted for the other's (no GPU)."""
import os
import shutil
import sys
import types

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("name,changes", [("rtgd_fp64.cu", {"fp64"}), ("rtgd_kernels.cu", {"mixed"}),
                                          ("rtgd_fp64.cuh", {"fp64", "mixed"}), ("rtgd_api.cu", set())])
def test_hash_follows_the_kernel(tmp_path, monkeypatch, name, changes):
    csrc = "paper_2506_18579_gb300/csrc"
    shutil.copytree(os.path.join(ROOT, csrc), tmp_path / csrc)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = {p: bench.kernel_source_hash(p) for p in ("mixed", "fp64")}
    with open(tmp_path / csrc / name, "a", encoding="utf-8") as fh:
        fh.write("// a comment\n")
    assert before == {p: bench.kernel_source_hash(p) for p in before}
    with open(tmp_path / csrc / name, "a", encoding="utf-8") as fh:
        fh.write("int more;\n")
    assert {p for p in before if bench.kernel_source_hash(p) != before[p]} == changes


def test_traffic_is_of_the_precision(monkeypatch):
    cfg = types.SimpleNamespace(kernel=1, stencil=2, lanes_per_ray=1)
    monkeypatch.setattr(bench, "TRAFFIC", {("c4", "mixed", 1, 2, 1): {"bytes_per_launch": 7,
                                                                   "source_sha256": bench.kernel_source_hash("mixed")}})
    assert bench.captured_traffic("c4", cfg, "mixed") == 7
    assert bench.captured_traffic("c4", cfg, "fp64") is None

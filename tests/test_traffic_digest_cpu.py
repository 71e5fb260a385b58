"""The digest under which bench.py reuses the committed DRAM counters covers every file that decides them, and no comments."""
import importlib.util
import os
import re
import shutil

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture()
def bench(tmp_path, monkeypatch):
    spec = importlib.util.spec_from_file_location("bench_digest", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    shutil.copytree(os.path.join(ROOT, "paper_1004_5058_gb300", "csrc"), tmp_path / "paper_1004_5058_gb300" / "csrc")
    monkeypatch.setattr(m, "ROOT", str(tmp_path))
    return m


# the segment height (halo rows read again), the kernel form and the promotion size are chosen in lb_tiled.cu
@pytest.mark.parametrize("name,old,new", [
    ("lb_tiled.cu", "(ty + 5.5)", "(ty + 6.5)"), ("lb_tiled.cu", "256LL << 20", "512LL << 20"),
    ("lb_tiled.cu", "L2_PROMOTION_L2_256B", "L2_PROMOTION_L2_64B"), ("lb_tiled.cuh", "constexpr int RING = 6", "constexpr int RING = 7")])
def test_digest_follows_the_code(bench, name, old, new):
    before = bench.source_digest()
    path = os.path.join(bench.ROOT, "paper_1004_5058_gb300", "csrc", name)
    src = open(path).read()
    assert old in re.sub(r"//[^\n]*", "", src)
    open(path, "w").write("// a comment\n" + src)
    assert bench.source_digest() == before
    open(path, "w").write(src.replace(old, new))
    assert bench.source_digest() != before

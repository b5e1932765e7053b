"""The bench's DRAM figure of the dominant kernel stands only as long as every
file the kernel is made of is what it was when the counters were read."""
import os
import re
import shutil
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_sources_cover_the_kernels_headers():
    csrc = os.path.dirname(bench.ROOFLINE_SOURCES[0])
    seen, todo = set(), [os.path.basename(bench.ROOFLINE_SOURCES[0])]
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        todo += re.findall(r'#include "(\w+\.cuh)"', open(os.path.join(csrc, name)).read())
    assert seen == {os.path.basename(p) for p in bench.ROOFLINE_SOURCES}


def test_a_change_in_any_source_drops_the_figure(tmp_path, monkeypatch):
    copies = [shutil.copy(p, tmp_path) for p in bench.ROOFLINE_SOURCES]
    monkeypatch.setattr(bench, "ROOFLINE_SOURCES", copies)
    traffic = tmp_path / "traffic.txt"
    traffic.write_text(f"source_sha256_16={bench._source_hash()}\ndram_bytes_per_record=7.5\n")
    monkeypatch.setattr(bench, "TRAFFIC_FILE", str(traffic))
    assert bench._traffic_per_record() == 7.5
    for path in copies:
        before = open(path).read()
        with open(path, "a") as f:
            f.write("// changed\n")
        assert bench._traffic_per_record() is None
        with open(path, "w") as f:
            f.write(before)
        assert bench._traffic_per_record() == 7.5

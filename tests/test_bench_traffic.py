"""The committed DRAM-traffic record of the scan is used only while all of the scan's
code is the one it was captured on."""
import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_1807_01409_gb300", "csrc")


@pytest.mark.parametrize("name, at, counts", [
    ("select.cuh", "sel_walk(const SelScratch &sc", True), ("select.cuh", "void sel_finish(", True),
    ("select.cuh", "inline unsigned sel_index_grid(", True), ("compact.cu", "sc->ranges = (unsigned)", True),
    ("compact.cu", "int compact_filter(", False)])
def test_traffic_record_follows_all_of_the_scan(tmp_path, name, at, counts):
    csrc = tmp_path / "csrc"
    csrc.mkdir()
    for f in ("match.cu", "select.cuh", "compact.cu"):
        shutil.copy(os.path.join(CSRC, f), csrc / f)
    match = os.path.join(CSRC, "match.cu")
    assert bench._kernel_region_sha1(match, str(csrc)) == bench._kernel_region_sha1(match)
    text = (csrc / name).read_text()
    i = text.index(at)
    (csrc / name).write_text(text[:i] + "/* changed */ " + text[i:])
    assert (bench._kernel_region_sha1(match, str(csrc)) != bench._kernel_region_sha1(match)) == counts
    if counts:
        assert bench._traffic_record(match, str(csrc)) is None

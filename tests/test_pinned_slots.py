"""The learned path's read-back slots: the guard on the number of its groups holds
for the layout of the plan's page-locked words as it is, and refuses a number whose
boundaries would reach the bins' slots."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_14558_gb300", "csrc")


def compiles(groups, tmp_path):
    internal = open(os.path.join(CSRC, "spg_internal.cuh")).read()
    learned = open(os.path.join(CSRC, "learned.cu")).read()
    slots = re.search(r"constexpr int kPinnedHist[^;]*;", internal).group(0)
    guard = re.search(r"static_assert\([^;]*kLearnedGroups[^;]*;", learned, re.S).group(0)
    src = tmp_path / f"guard{groups}.cpp"
    src.write_text(f"#include <cstdint>\n{slots}\nconstexpr int64_t kLearnedGroups = {groups};\n{guard}\n")
    return subprocess.run(["g++", "-std=c++17", "-fsyntax-only", str(src)], capture_output=True).returncode == 0


@pytest.mark.skipif(not shutil.which("g++"), reason="needs g++")
def test_the_guard_knows_where_the_bins_slots_begin(tmp_path):
    internal = open(os.path.join(CSRC, "spg_internal.cuh")).read()
    learned = open(os.path.join(CSRC, "learned.cu")).read()
    slot = {n: int(v) for n, v in re.findall(r"(kPinned\w+) = (\d+)", internal)}
    groups = int(re.search(r"kLearnedGroups = (\d+)", learned).group(1))
    most = (slot["kPinnedBins"] - slot["kPinnedHist"]) // 2 - 1
    assert groups <= most and compiles(groups, tmp_path) and compiles(most, tmp_path)
    assert not compiles(most + 1, tmp_path)
    # every other slot that the learned path names lies among the counters'
    assert all(int(n) < slot["kPinnedHist"] for n in re.findall(r"h_pinned(?: \+ |\[)(\d+)", learned))

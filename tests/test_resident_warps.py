"""The rule that picks the warps per CTA of the batch's kernels, compiled here with
occupancies as registers and shared memory give them."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_14558_gb300", "csrc")

SOURCE = r"""
#include <algorithm>
#include <cassert>
#include <cstdio>
#include "resident_warps.cuh"
using spg::most_resident_warps;
// CTAs of w warps on an SM: four partitions of 16,384 registers, 228 KB with 1 KB kept per CTA
static int sm(int w, int regs, long table) {
    const long smem = table * w;
    if (smem > 227 * 1024) return 0;
    return (int)std::min<long>(4 * (16384 / ((regs + 7) / 8 * 8 * 32)) / w, 228 * 1024 / (smem + 1024));
}
int main() {
    auto pick = [](int least, int most, int regs, long table) {
        return most_resident_warps(least, most, [&](int w) { return sm(w, regs, table); });
    };
    // shared memory alone would keep 32 warps either way: registers decide
    assert(sm(8, 72, 6656) == 3 && sm(4, 72, 6656) == 7 && pick(4, 8, 72, 6656) == 7);
    assert(sm(8, 80, 6656) == 3 && sm(4, 80, 6656) == 6 && pick(4, 8, 80, 6656) == 8);
    assert(pick(2, 4, 72, 6656) == 4);
    // few registers: shared memory decides, and of equal numbers the largest CTA
    assert(pick(4, 8, 32, 6656) == 8 && pick(4, 8, 32, 25088) == 8 && pick(2, 4, 32, 25088) == 3);
    // more asked than fits, and nothing fits
    assert(pick(4, 8, 32, 40000) == 5 && pick(4, 8, 32, 60000) == 0);
    for (int regs = 32; regs <= 128; regs++)
        for (long table : {6656l, 12800l, 25088l})
            for (int most : {4, 8}) {
                const int w = pick(most / 2, most, regs, table);
                for (int o = most / 2; o <= most; o++) assert(o * sm(o, regs, table) <= w * sm(w, regs, table));
            }
    puts("warps ok");
}
"""


@pytest.mark.skipif(not shutil.which("g++"), reason="needs g++")
def test_most_resident_warps(tmp_path):
    src, exe = tmp_path / "warps.cpp", tmp_path / "warps"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True, timeout=120)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and "warps ok" in r.stdout, r.stdout + r.stderr

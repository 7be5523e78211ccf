"""The rule that picks the ICP kernels' blocks per pose (host code): only
clusters that the device holds all at once, and only for poses with the pixels
to pay for their barriers."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "icp_shape.h"
int main() {
    const rl::IcpResident devices[] = {{}, {51, 148}, {0, 148}, {57, 152}};
    const int sizes[][2] = {{96, 64}, {160, 120}, {240, 180}, {320, 240}, {400, 300}, {500, 375}, {640, 480}, {1024, 768}};
    for (const rl::IcpResident &r : devices)
        for (const auto &s : sizes)
            for (int poses = 1; poses <= 200; ++poses)
                std::printf("%d %d %d %d %d\n", r.of8, r.of4, s[0], poses,
                            rl::icp_blocks(r, 152, poses, s[0] * s[1] * (6 / 16.0 + 3 / 4.0 + 2) / 11));
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_clusters_only_where_resident_and_worth_it(tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1810_12163_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [tuple(map(int, ln.split())) for ln in out.splitlines()]
    assert len(rows) == 4 * 8 * 200
    # fewest pixels (as image widths of the default levels) at which a cluster of c blocks pays, by blocks on an SM
    least = {8: {1: 240, 2: 240, 3: 320}, 4: {1: 400, 2: 400, 3: 500, 4: 640}}
    for of8, of4, width, poses, blocks in rows:
        held = {8: of8, 4: of4}
        pays = [c for c in (8, 4) if poses <= held[c] and width >= least[c].get(-(-poses * c // 152), 1 << 30)]
        assert blocks == max(pays, default=1), (of8, of4, width, poses)

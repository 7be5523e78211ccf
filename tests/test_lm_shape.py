"""The rule that picks the LM kernel's clusters (host code): never one that
the device cannot hold, whatever the number of frames."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "lm_shape.h"
int main() {
    const rl::LmResident devices[] = {{}, {0, 16, 0}, {8, 16, 8}, {3, 9, 0}};
    for (const rl::LmResident &r : devices)
        for (int first = 0; first < 2; ++first)
            for (int sparse = 0; sparse < 2; ++sparse)
                for (int frames = 1; frames <= 70; ++frames)
                    std::printf("%d %d %d %d %d %d %d\n", r.first4, r.first2, r.later2, first, sparse, frames,
                                rl::lm_sets(r, first != 0, frames, sparse != 0));
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_sets_follow_what_the_device_holds(tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1810_12163_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [tuple(map(int, ln.split())) for ln in out.splitlines()]
    assert len(rows) == 4 * 2 * 2 * 70
    for first4, first2, later2, first, sparse, frames, sets in rows:
        held = {4: first4, 2: first2} if first else {2: later2}
        # at most one waits; where most frames are empty, clusters of 16 (4 x 4, 8 x 2) two deep and of 8 three
        deep = {s: 1 if not sparse else 2 if s * (4 if first else 8) == 16 else 3 for s in held}
        fits = [s for s, n in held.items() if n > 0 and frames <= deep[s] * (n + 1)]
        assert sets == max(fits, default=1), (first4, first2, later2, first, sparse, frames)

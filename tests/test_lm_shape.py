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
        for (int kind = 0; kind < 8; ++kind)
            for (int frames = 1; frames <= 70; ++frames)
                std::printf("%d %d %d %d %d %d %d %d\n", r.first4, r.first2, r.later2, kind & 1, kind >> 1 & 1, kind >> 2,
                            frames, rl::lm_sets(r, kind & 1, frames, kind >> 1 & 1, kind >> 2));
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
    assert len(rows) == 4 * 8 * 70
    for first4, first2, later2, first, sparse, heavy, frames, sets in rows:
        held = {4: first4, 2: first2} if first else {2: later2}
        # none waits; of heavy ones one; where most frames are empty, clusters of 16 (4 x 4, 8 x 2) two deep, of 8 three
        deep = {s: 1 if not sparse else 2 if s * (4 if first else 8) == 16 else 3 for s in held}
        fits = [s for s, n in held.items() if n > 0 and frames <= (deep[s] * (n + 1) if heavy else n)]
        assert sets == max(fits, default=1), (first4, first2, later2, first, sparse, heavy, frames)

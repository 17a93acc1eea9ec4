"""Checkpoint memory of plans (host rule, compiled here by itself): the slots asked for, and the share
of the free memory that a plan without persistence leaves to its program."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_09417_gb300", "csrc")
GB = 1 << 30

# (items, tiles, pairs, tile_px, seg_len, recompute), persistent, free bytes -> slots
CASES = [
    ((100000, 1024, 24 * 100000, 256, 64, 0), 0, 200 * GB, 3125),           # two pairs an item, ample memory
    ((100000, 1024, 24 * 100000, 256, 64, 1), 0, 200 * GB, 3125 + 1024),    # and a final state a tile
    ((100000, 1024, 6400, 256, 64, 0), 0, 200 * GB, 100),                   # no more than the pairs can use
    ((50000000, 8192, 2 ** 31 - 1, 256, 64, 0), 0, 200 * GB, GB // 4096),   # a GiB
    ((50000000, 8192, 2 ** 31 - 1, 256, 64, 0), 0, 2 * GB, GB // 8 // 4096),   # a 16th of the free memory
    ((50000000, 8192, 2 ** 31 - 1, 256, 64, 0), 1, 2 * GB, GB // 4096),     # asked for: a GiB
    ((50000000, 8192, 2 ** 31 - 1, 256, 64, 0), 0, 0, 1),
    ((0, 1, 1, 32, 32, 0), 0, 200 * GB, 1),
]


def test_checkpoint_slots(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    lines = ["#include <cstdio>", '#include "checkpoints.h"', "int main() {"]
    for args, persistent, free, _ in CASES:
        lines.append('printf("%%lld\\n", (long long)vbm::checkpoint_slots(%s, vbm::checkpoint_bytes(%d, %dll)));'
                     % (", ".join("%dll" % a if i < 4 else str(a) for i, a in enumerate(args)), persistent, free))
    lines.append("}")
    src, exe = tmp_path / "slots.cpp", tmp_path / "slots"
    src.write_text("\n".join(lines))
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    got = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert [int(x) for x in got] == [c[3] for c in CASES]

"""Which batches become chains of passes and which persistent launches, compiled on the host from the rule's
header: lists on which chains measured slower than the persistent launches must not take them, and a class must
not keep more blocks resident than its grids can use."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_05983_gb300", "csrc")

# (grids, classes, passes, chains)
LISTS = [(40, 1, 1000, False), (47, 1, 470, False), (32, 1, 1600, False), (16, 1, 800, False), (8, 1, 400, False),
         (32, 7, 3000, False), (47, 8, 3000, False), (3, 1, 30, False), (96, 16, 6000, False),
         (24, 16, 1400, True), (2, 1, 20, True), (8, 4, 700, True), (8, 4, 20001, False), (1, 1, 20000, True)]

# tiles, tiles of one pass of every grid, resident slots, blocks
BLOCKS = [(6400, 32, 304, 64), (6400, 400, 304, 304), (40, 32, 304, 40), (1, 1, 304, 1), (10, 1, 1, 1)]


def test_rule(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "rule.cpp"
    calls = "\n".join(f'  std::printf("%d\\n", (int)stn::batch_as_chains({n}, {c}, {p}));' for n, c, p, _ in LISTS)
    blocks = "\n".join(f'  std::printf("%d\\n", (int)stn::batch_blocks({t}, {p}, {m}));' for t, p, m, _ in BLOCKS)
    src.write_text(f'#include <cstdio>\n#include "{CSRC}/batch_rule.h"\nint main() {{\n{calls}\n{blocks}\n}}\n')
    exe = tmp_path / "rule"
    subprocess.run([cxx, "-std=c++17", str(src), "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert [bool(int(g)) for g in got[:len(LISTS)]] == [w for *_, w in LISTS]
    assert [int(g) for g in got[len(LISTS):]] == [w for *_, w in BLOCKS]

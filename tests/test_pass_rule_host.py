"""Which 3D streaming passes are launched as dependents of the pass before, compiled on the host: not the ones
whose blocks leave slots free (an explicit segment on a small grid), where early blocks crowd a few SMs."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_05983_gb300", "csrc")

# (whole waves, blocks, slots, dependent)
PASSES = [(1, 96, 608, True), (0, 96, 608, False), (0, 608, 608, False), (0, 759, 608, False), (0, 760, 608, True), (0, 5000, 608, True)]


def test_dependent_passes(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    calls = "\n".join(f'  std::printf("%d\\n", (int)stn::dependent_pass({w}, {b}, {s}));' for w, b, s, _ in PASSES)
    src = tmp_path / "rule.cpp"
    src.write_text(f'#include <cstdio>\n#include "{CSRC}/pass_rule.h"\nint main() {{\n{calls}\n}}\n')
    exe = tmp_path / "rule"
    subprocess.run([cxx, "-std=c++17", str(src), "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert [bool(int(g)) for g in got] == [w for *_, w in PASSES]
    with open(os.path.join(CSRC, "stencil_api.cu")) as fh:
        api = fh.read()
    assert "st, ps.dependent && like)" in api and "st, h->dim == 3)" not in api   # the streaming launch uses the rule
    # and not beside another kind of pass
    assert "const bool like = j > 0 ? j < L - 1 || t_last == t : rag != nullptr;" in api

"""The adjoint's walk over the components of a shell with one value along an axis (axis_component of
csrc/eri_bwd_table.h, the code the kernel calls), built by the host compiler, against the definition: every
component with that value once, at its place in output order."""
import os
import shutil
import subprocess

import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                      "paper_2303_13632_gb300", "csrc", "eri_bwd_table.h")


def test_components_of_a_value_along_an_axis(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "dump.cpp", tmp_path / "dump"
    src.write_text(f'#include <cstdio>\n#include "{HEADER}"\n'
                   "int main() { for (int L = 0; L < 4; ++L) for (int x = 0; x < 3; ++x) for (int v = 0; v <= L; ++v)\n"
                   "for (int n = 0; n <= L - v; ++n)\n"
                   'std::printf("%d %d %d %d\\n", L, x, v, eri::axis_component(L, x, v, n)); }\n')
    subprocess.run([cxx, "-std=c++17", "-O1", str(src), "-o", str(exe)], check=True)
    got = {}
    for line in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines():
        L, x, v, i = map(int, line.split())
        got.setdefault((L, x, v), []).append(i)
    for L in range(4):
        comps = [(lx, ly, L - lx - ly) for lx in range(L, -1, -1) for ly in range(L - lx, -1, -1)]
        for x in range(3):
            for v in range(L + 1):
                assert sorted(got.pop((L, x, v))) == [i for i, c in enumerate(comps) if c[x] == v]
    assert not got

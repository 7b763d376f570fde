"""Decisions the host takes before a launch (csrc/imb_host.h), compiled with the host compiler and
checked over their whole range, without a GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1809_07008_gb300", "csrc")


def run_cpp(tmp_path, body):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "imb_host.h"\n#include <cstdio>\n#include <cstdlib>\nusing namespace imb;\n'
                   '#define CHECK(c) do { if (!(c)) { std::printf("failed: %s\\n", #c); std::exit(1); } } while (0)\n' + body)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_adjoint_blocks_hold_the_edge_columns_together(tmp_path):
    # every width a lattice can have (3 rows at least): each column in one block, 0 beside 1, nx - 2 beside
    # nx - 1 (also where every multiple of 32 up to 256 leaves one column: nx = 1 modulo 26880)
    run_cpp(tmp_path, """
int main() {
    for (int nx = 3; nx <= (1 << 27) / 3; ++nx)
        for (int inlet = 0; inlet < 2; ++inlet) {
            const AdjointGrid g = adjoint_grid(nx, inlet);
            auto block = [&](int x) { return (x + g.shift) / ADJ_BLOCK; };
            CHECK(g.shift >= 0 && g.shift < ADJ_BLOCK);
            CHECK(g.blocks > 0 && block(nx - 1) == g.blocks - 1 && block(0) == 0);
            if (inlet) CHECK(block(1) == 0 && block(nx - 2) == g.blocks - 1);
        }
}
""")

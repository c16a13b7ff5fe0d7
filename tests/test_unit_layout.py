"""The units the decision kernels work on (tree_layout.h unit_node): every inner node below a
tree's top nodes is the node of exactly one (unit, lane), a unit's lanes hold its upper nodes
in heap order and then, per bottom subtree, left child, right child and root, and the top
nodes are one fewer than the units."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2511_09376_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "tree_layout.h"
int main() {
    for (int D = 2; D <= 8; ++D) {
        std::printf("%d %d %d", D, wdf::units_per_tree(D), wdf::unit_subtrees(D));
        for (int u = 0; u < wdf::units_per_tree(D); ++u)
            for (int i = 0; i < (1 << wdf::unit_height(D)) - 1; ++i) std::printf(" %d", wdf::unit_node(D, u, i));
        std::printf("\n");
    }
    return 0;
}
"""


def test_units_cover_every_node(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "unit.cpp", tmp_path / "unit"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    for line in filter(None, subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")):
        D, U, S, *nodes = map(int, line.split())
        per = len(nodes) // U
        assert U * S == 1 << (D - 2)
        assert sorted(nodes + list(range(U - 1))) == list(range((1 << D) - 1)), D
        for u in range(U):
            mine = nodes[u * per:(u + 1) * per]
            assert mine[:S - 1] == sorted(mine[:S - 1])
            for s in range(S):
                r = (1 << (D - 2)) - 1 + u * S + s
                assert mine[S - 1 + 3 * s:S + 2 + 3 * s] == [2 * r + 1, 2 * r + 2, r], (D, u, s)

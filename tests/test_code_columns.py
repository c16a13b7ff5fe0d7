"""Code columns of wide ensembles (pack.cpp, tree_layout.h): every unit node names a column of
its own feature and, with all its quads, stays inside a row block, on both sides of 2^16
columns and past 2^17 (host); the counts of such rows equal a direct comparison (GPU)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2511_09376_gb300 import synth

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2511_09376_gb300", "csrc")

# stumps, feature i with threshold i / 2: tree i of the depth-2 layout has its root in lane 2
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "wdf_internal.h"
int main(int, char **v) {
    const int n = std::atoi(v[1]);
    std::vector<int64_t> off;
    std::vector<int32_t> f, l, r;
    std::vector<float> t, w;
    for (int i = 0; i <= n; ++i) off.push_back(3 * (int64_t)i);
    for (int i = 0; i < n; ++i)
        for (int k = 0; k < 3; ++k) {
            f.push_back(k ? -1 : i); l.push_back(k ? -1 : 1); r.push_back(k ? -1 : 2);
            t.push_back(0.5f * (float)i); w.push_back((float)k);
        }
    wdf::Packed p;
    std::string err;
    if (wdf::pack_ensemble(n, n, off.data(), f.data(), t.data(), l.data(), r.data(), w.data(), &p, &err)) return 1;
    int bad = 0;
    for (int i = 0; i < n; ++i) {
        const uint32_t at = p.unit[(size_t)i * 32 + 2].at;
        const int c = wdf::unit_column(at), q = wdf::unit_quads(at);
        bad += c >= (int)p.scol.size() || p.scol[c].feature != i || q != 1 || p.qbase[q - 1] + c >= p.quads ||
               wdf::unit_start(at) != 1u;
    }
    std::printf("%d\n", bad);
    return 0;
}
"""


@pytest.mark.parametrize("columns", [65_535, 65_536, 65_537, 70_000, 140_000])
def test_columns_of_stumps(tmp_path, columns):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "cols.cpp", tmp_path / "cols"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), os.path.join(CSRC, "pack.cpp"), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe), str(columns)], capture_output=True, text=True, check=True).stdout
    assert int(out) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("columns", [70_000, 140_000])
def test_counts_of_stumps(columns):
    import torch

    import paper_2511_09376_gb300 as wdf
    n, m = columns, 131
    rng = np.random.default_rng(columns)
    node = np.tile(np.array([0, -1, -1], np.int32), n)
    ens = synth.Ensemble(n, 3 * np.arange(n + 1, dtype=np.int64),
                         np.where(node == 0, np.repeat(np.arange(n, dtype=np.int32), 3), -1).astype(np.int32),
                         np.repeat(rng.standard_normal(n).astype(np.float32), 3),
                         np.where(node == 0, 1, -1).astype(np.int32), np.where(node == 0, 2, -1).astype(np.int32),
                         np.tile(np.array([0.0, 1.0, 2.0], np.float32), n))
    B = rng.standard_normal((m, n)).astype(np.float32)
    ctx = wdf.ctx_create(0)
    e = wdf.load_ensemble(ctx, ens)
    wdf.set_background(e, torch.from_numpy(B).cuda())
    got = wdf.debug_leaf_hist(e)  # leaves 0 (left) and 2 (right); the children send every row left
    left = (B < ens.threshold[::3]).sum(axis=0)
    np.testing.assert_array_equal(got[:, 0, 3], left)
    np.testing.assert_array_equal(got[:, 0, 1], m - left)
    np.testing.assert_array_equal(got[:, 2, 3], m - left)
    np.testing.assert_array_equal(got[:, 2, 1], left)
    base = wdf.expected_value(e)
    want = float((left * 1.0 + (m - left) * 2.0).sum()) / m
    assert abs(base - want) <= 1e-9 * want
    e.close()
    ctx.close()

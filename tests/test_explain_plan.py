"""The plan of a consumer call (explain_plan.h): its scratch stays within 320 MB whatever the
estimate prefers (split tiles then run in slices of the rows), calls of few rows still get
theirs, and a call whose scratch cannot be allocated runs with whole tiles (a host allocator
that refuses stands in for the GPU's); sliced calls give the bits of a batch (GPU)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2511_09376_gb300", "csrc")
LIMIT = 320 << 20

PROGRAM = r"""
#include <cstdio>
#include "explain_plan.h"
int main() {
    long long D, n, T, F, tile, per_sm, room;
    while (std::scanf("%lld %lld %lld %lld %lld %lld %lld", &D, &n, &T, &F, &tile, &per_sm, &room) == 7) {
        wdf::ExplainPlan p = wdf::explain_plan((int)D, n, (int)T, (int)F, (int)tile, 152, per_sm);
        std::printf("%d %zu %lld", p.splits, p.scratch_floats, (long long)p.rows);
        size_t got = 0;  // an allocator that has `room` bytes
        const int e = wdf::take_scratch(&p, n, 1000, 2, [&](size_t bytes) { got = bytes; return bytes > (size_t)room ? 2 : 0; });
        std::printf(" %d %d %zu %zu\n", e, p.splits, p.scratch_floats, got);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(d / "plan.cpp"), "-o", str(d / "plan")], check=True)

    def run(calls):
        text = "\n".join(" ".join(map(str, c)) for c in calls)
        out = subprocess.run([str(d / "plan")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.strip().split("\n")]

    return run


# (depth, rows, trees, features, blocks per SM): node values, split at once, split in slices
@pytest.mark.parametrize("call,route", [((6, 1, 100, 127, 8), "values"), ((7, 777, 500, 112, 8), "values"),
                                        ((8, 20_011, 1000, 134, 6), "split"), ((8, 293_300, 1000, 134, 6), "slices"),
                                        ((8, 100_000, 400, 500, 2), "slices"), ((6, 200_000, 1000, 127, 8), "slices")])
def test_choice(plan, call, route):
    D, n, T, F, per_sm = call
    (splits, _, rows, *_), = plan([(D, n, T, F, 32, per_sm, 1 << 40)])
    assert route == ("values" if splits == 0 else "whole" if splits == 1 else "split" if rows == n else "slices")


def test_scratch_is_bounded(plan):
    calls = [(D, n, T, F, 32, max(1, min(8, 1600 // F)), 1 << 40)
             for D in range(2, 9) for T in (1, 10, 100, 300, 1000, 5000) for F in (1, 20, 127, 500, 1700)
             for n in (1, 33, 1000, 8000, 20_000, 77_777, 293_300, 778_113, 1 << 20)]
    for c, (splits, floats, rows, *_) in zip(calls, plan(calls)):
        assert 4 * floats <= LIMIT, c
        assert (floats == 0) == (splits == 1), c
        assert rows == c[1] or (splits > 1 and 0 < rows < c[1] and rows % 128 == 0), c  # tiles do not cross slices


def test_refused_scratch(plan):
    # room for the codes alone, for everything, for nothing
    for call in [(8, 20_011, 1000, 134, 32, 6), (8, 293_300, 1000, 134, 32, 6), (6, 300, 100, 127, 32, 8)]:
        (s, f, *_), = plan([call + (1 << 40,)])
        assert f > 0
        assert plan([call + (2000,)])[0][3:] == (0, 1, 0, 1024)
        assert plan([call + (1024 + 4 * f,)])[0][3:] == (0, s, f, 1024 + 4 * f)
        assert plan([call + (10,)])[0][3] == 2


@pytest.mark.gpu
def test_slices_match_a_batch():
    import numpy as np
    import torch

    import paper_2511_09376_gb300 as wdf
    from paper_2511_09376_gb300 import synth
    n, T, D, F = 30_007, 200, 8, 500  # eight parts: slices of 15,104 rows
    ens, _, B = synth.make(synth.Workload("s", 9, 1, 500, F, 400, T, D, 0.1, 0.1, False))
    ctx = wdf.ctx_create(0)
    e = wdf.load_ensemble(ctx, ens)
    wdf.set_background(e, torch.from_numpy(B).cuda())
    C = torch.randn((n, F), generator=torch.Generator("cuda").manual_seed(3), device="cuda")
    out = torch.full((n, F + 5), 7.0, device="cuda")
    wdf.explain(e, C, out=out[:, :F])
    batch = wdf.batch_create(ctx, [e])
    want = wdf.batch_explain(batch, [(0, C)])[0]
    np.testing.assert_array_equal(out[:, :F].cpu().numpy(), want.cpu().numpy())
    assert (out[:, F:] == 7.0).all()
    batch.close()
    e.close()
    ctx.close()

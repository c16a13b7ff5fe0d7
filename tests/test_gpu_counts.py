"""The counting kernel's pattern counts are exact (integers equal to a direct walk of every
background row) at the edges of its row tiles (32-row blocks, 128-row tiles, the 512-row
runs of long chunks), at every depth, with columns of more than 255 and more than 4,095
thresholds, with NaN and infinite values, and with rows too wide for its shared-memory
tiles."""
import numpy as np
import pytest

from paper_2511_09376_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2511_09376_gb300 as wdf
    return wdf.ctx_create(0)


def _counts_equal(ctx, ens, B):
    """Every live leaf's pattern counts against a walk of its path for every row."""
    import torch

    import paper_2511_09376_gb300 as wdf
    e = wdf.load_ensemble(ctx, ens)
    wdf.set_background(e, torch.from_numpy(B).cuda())
    got = wdf.debug_leaf_hist(e).astype(np.int64)
    D = wdf.ensemble_info(e)["depth"]
    T, NL = ens.n_trees, 1 << D
    for t in range(T):
        o = int(ens.tree_offset[t])
        for q in range(NL):
            # walk the complete layout: an early leaf sends every row left
            v, path, live = 0, [], True
            for k in range(D):
                turn = (q >> (D - 1 - k)) & 1
                if ens.feature[o + v] < 0:
                    path.append((None, turn))
                    live = live and turn == 0
                else:
                    path.append((v, turn))
                    v = int((ens.right if turn else ens.left)[o + v])
            live = live and ens.value[o + v] != 0.0
            p = np.zeros(B.shape[0], np.int64)
            for node, turn in path:
                if node is None:
                    bit = np.full(B.shape[0], turn == 0)
                else:
                    left = B[:, ens.feature[o + node]] < ens.threshold[o + node]
                    bit = ~left if turn else left
                p = 2 * p + bit
            if live:
                np.testing.assert_array_equal(got[t, q], np.bincount(p, minlength=NL), f"tree {t} leaf {q}")
    e.close()


@pytest.mark.parametrize("depth", range(2, 9))
@pytest.mark.parametrize("m", [1, 31, 33, 127, 128, 129, 1000])
def test_tile_edges(ctx, depth, m):
    w = synth.Workload("c", 900 + depth, 1, m, 9, 6, 3, depth, 0.5, 0.15, False)
    ens, _, B = synth.make(w)
    _counts_equal(ctx, ens, B)


@pytest.mark.parametrize("depth", [3, 6, 7])
@pytest.mark.parametrize("m", [16383, 16384, 16897])
def test_long_chunks(ctx, depth, m):
    ens, _, B = synth.make(synth.Workload("c", 950 + depth, 1, m, 7, 5, 2, depth, 0.5, 0.1, False))
    B[::7, 0], B[1::11, 1], B[2::13, 2] = np.nan, np.inf, -np.inf
    _counts_equal(ctx, ens, B)


@pytest.mark.parametrize("trees,features", [(30, 2), (330, 2)])  # columns of 9 and of 12 bits, the latter cut in two
def test_wide_columns(ctx, trees, features):
    ens, _, B = synth.make(synth.Workload("c", 970, 1, 300, features, features, trees, 6, 0.5, 0.1, False))
    if trees > 100:
        assert max(np.unique(ens.threshold[ens.feature == f]).size for f in range(features)) > 4095
    _counts_equal(ctx, ens, B)


def test_wide_rows(ctx):
    ens, _, B = synth.make(synth.Workload("c", 980, 1, 260, 3000, 2500, 60, 6, 0.5, 0.0, True))
    assert np.unique(ens.feature).size > 1400
    _counts_equal(ctx, ens, B)


@pytest.mark.parametrize("depth", [7, 8])
@pytest.mark.parametrize("features", [1000, 3000])  # fewer units per block; codes read from global memory
def test_wide_rows_of_deep_trees(ctx, depth, features):
    ens, _, B = synth.make(synth.Workload("c", 990 + depth, 1, 200, features, features, 40, depth, 0.5, 0.1, False))
    _counts_equal(ctx, ens, B)

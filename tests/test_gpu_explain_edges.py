"""The consumer kernel at the edges of its tiles and parts, against the FP64 oracle (the
FP32-mode bar of conftest.py): row counts around 32, 64 and 128; one tree, odd numbers of
trees (its two warps take trees in turn) and tree counts around the limits of the parts that
a row's sum is made of; so few features that the flush batches repeat them, singly and more
than once; a feature nothing splits on."""
import numpy as np
import pytest

import oracle
from conftest import assert_phi_close
from paper_2511_09376_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2511_09376_gb300 as wdf
    return wdf.ctx_create(0)


def _check(ctx, D, T, F, n, seed, early=0.12):
    import torch

    import paper_2511_09376_gb300 as wdf
    ens, C, B = synth.make(synth.Workload("x", seed, n, 400, F, max(1, F - 2), T, D, 0.3, early, False))
    e = wdf.load_ensemble(ctx, ens)
    wdf.set_background(e, torch.from_numpy(B).cuda())
    got = wdf.explain(e, torch.from_numpy(C).cuda()).cpu().numpy()
    want = oracle.values_hist(ens, oracle.bg_hist(ens, B), B.shape[0], C)
    assert_phi_close(got, want, f"D={D} T={T} F={F} n={n}")
    batch = wdf.batch_create(ctx, [e])
    tile = wdf.batch_explain(batch, [(0, torch.from_numpy(C).cuda())])[0]
    np.testing.assert_array_equal(got, tile.cpu().numpy())
    batch.close()
    e.close()


@pytest.mark.parametrize("depth", range(2, 9))
@pytest.mark.parametrize("n", [1, 31, 33, 64, 129])
def test_rows(ctx, depth, n):
    _check(ctx, depth, 7, 20, n, 1000 + depth)


@pytest.mark.parametrize("depth", range(2, 9))
@pytest.mark.parametrize("features", [1, 2, 5])
def test_repeated_features(ctx, depth, features):
    _check(ctx, depth, 6, features, 70, 1100 + depth, early=0.0)


# parts hold about 3200 / 2^depth trees: one, two and three parts, even and odd
@pytest.mark.parametrize("depth,trees", [(6, 1), (6, 2), (6, 74), (6, 75), (6, 126), (8, 18), (8, 19), (8, 100), (5, 151),
                                         (7, 39), (3, 601)])
def test_parts(ctx, depth, trees):
    _check(ctx, depth, trees, 30, 65, 1200 + depth)


# more rows, with fewer tiles than the GPU holds blocks: the tile kernel, parts on several blocks
@pytest.mark.parametrize("depth,trees,rows", [(8, 101, 5000), (7, 260, 4033), (6, 230, 6001), (5, 640, 5000)])
def test_parts_on_several_blocks(ctx, depth, trees, rows):
    _check(ctx, depth, trees, 40, rows, 1300 + depth)

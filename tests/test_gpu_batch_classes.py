"""A batch whose ensembles of one depth are in several classes: wdf_batch_tile_rows reports the
smallest of their tile sizes, whatever their order, and results stay those of single calls."""
import numpy as np
import pytest

from paper_2511_09376_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [(0, 1, 2), (2, 1, 0), (1, 2, 0)])
def test_smallest_tile_of_a_depth(order, tmp_path):
    import torch

    import paper_2511_09376_gb300 as wdf
    ctx = wdf.ctx_create(0)
    ens, reqs = [], []
    rng = np.random.default_rng(8)
    for k, F in enumerate([20, 20, 500]):  # the second one of another depth
        e_np, _, B = synth.make(synth.Workload("c", 80 + k, 1, 300, F, F, 30, 5 if k == 1 else 6, 0.3, 0.1, False))
        ens.append(wdf.load_ensemble(ctx, e_np))
        wdf.set_background(ens[-1], torch.from_numpy(B).cuda())
    for i, k in enumerate(order):
        F = wdf.ensemble_info(ens[k])["n_features"]
        reqs.append((i, torch.from_numpy(rng.standard_normal((300, F)).astype(np.float32)).cuda()))
    cache = tmp_path / "tiles.txt"
    batch = wdf.batch_create(ctx, [ens[k] for k in order])
    wdf.batch_autotune(batch, reqs, reps=1, cache_path=str(cache))
    batch.close()
    lines = [line.split() for line in cache.read_text().splitlines()]
    assert sorted((r[0], r[1]) for r in lines) == [("5", "32"), ("6", "32"), ("6", "512")]
    tile = {("5", "32"): "64", ("6", "32"): "128", ("6", "512"): "32"}
    cache.write_text("".join(" ".join(r[:3] + [tile[r[0], r[1]]] + r[4:]) + "\n" for r in lines))
    batch = wdf.batch_create(ctx, [ens[k] for k in order])
    wdf.batch_autotune(batch, reqs, reps=1, cache_path=str(cache))
    assert (wdf.batch_tile_rows(batch, 5), wdf.batch_tile_rows(batch, 6), wdf.batch_tile_rows(batch, 7)) == (64, 32, -1)
    for (i, C), got in zip(reqs, wdf.batch_explain(batch, reqs)):
        np.testing.assert_array_equal(got.cpu().numpy(), wdf.explain(ens[order[i]], C).cpu().numpy())
    batch.close()
    ctx.close()

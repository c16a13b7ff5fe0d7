"""Batches whose tiles are split into groups of parts, and the same tiles unsplit (a batch of
many rows): bit-identical to per-ensemble calls, call after call and after autotuning, with
rows of odd counts and a phi wider than the features."""
import numpy as np
import pytest

from paper_2511_09376_gb300 import synth

pytestmark = pytest.mark.gpu


# (trees, depth): one part (never split), two, five, eight; small batches split, large ones do not
@pytest.mark.parametrize("sizes", [(1, 33, 70, 129), (1, 3000, 300_001, 40)])
def test_groups(sizes):
    import torch

    import paper_2511_09376_gb300 as wdf
    ctx = wdf.ctx_create(0)
    ens, reqs, outs = [], [], []
    rng = np.random.default_rng(3)
    for k, (T, D, F) in enumerate([(20, 5, 9), (100, 6, 40), (250, 6, 21), (130, 8, 30)]):
        e_np, _, B = synth.make(synth.Workload(f"g{k}", 60 + k, 1, 500, F, F, T, D, 0.2, 0.1, False))
        e = wdf.load_ensemble(ctx, e_np)
        wdf.set_background(e, torch.from_numpy(B).cuda())
        ens.append(e)
    for k, n in enumerate(sizes):
        for i in {k, 3 - k}:
            F = wdf.ensemble_info(ens[i])["n_features"]
            reqs.append((i, torch.from_numpy(rng.standard_normal((n, F)).astype(np.float32)).cuda()))
            outs.append(torch.full((n, F + 3), 7.0, device="cuda"))
    batch = wdf.batch_create(ctx, ens)
    want = [wdf.explain(ens[i], C).cpu().numpy() for i, C in reqs]

    def check():
        views = [o[:, :w.shape[1]] for o, w in zip(outs, want)]
        for v in views:
            v.fill_(np.nan)
        wdf.batch_explain(batch, reqs, views)
        for o, v, w in zip(outs, views, want):
            np.testing.assert_array_equal(v.cpu().numpy(), w)
            assert (o[:, w.shape[1]:] == 7.0).all()

    check()
    check()
    wdf.batch_autotune(batch, reqs, [o[:, :w.shape[1]] for o, w in zip(outs, want)], reps=2)
    check()
    batch.close()
    ctx.close()

"""Explain calls on host rows in one, two and more chunks (by bytes), with padded row strides:
bit-identical to the same rows on the device."""
import numpy as np
import pytest

from paper_2511_09376_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,features,pad", [(700, 30, 0), (33_333, 30, 0), (33_334, 30, 5), (300_007, 31, 0),
                                              (9_001, 512, 3)])
def test_chunks(rows, features, pad):
    import torch

    import paper_2511_09376_gb300 as wdf
    ctx = wdf.ctx_create(0)
    ens, _, B = synth.make(synth.Workload("h", 70, 1, 400, features, features, 12, 4, 0.3, 0.1, False))
    e = wdf.load_ensemble(ctx, ens)
    wdf.set_background(e, torch.from_numpy(B).cuda())
    full = np.random.default_rng(rows).standard_normal((rows, features + pad)).astype(np.float32)
    C = full[:, :features]
    for _ in range(2):
        got = wdf.explain(e, C)
        want = wdf.explain(e, torch.from_numpy(np.ascontiguousarray(C)).cuda()).cpu().numpy()
        np.testing.assert_array_equal(np.asarray(got), want)
    e.close()
    ctx.close()

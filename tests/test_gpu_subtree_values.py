"""Values and pair values from the joint counts by subset sums, against the FP64
oracle (the FP32-mode bar of conftest.py): every depth and both metrics, paths whose
positions all ask the same feature, or two, or repeat some; early leaves and dead subtrees;
counts near the 2^32 - 1 rows that a background may have."""
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


def _setup(depth, features, early=0.15, m=300):
    return synth.make(synth.Workload("v", 1500 + depth, 40, m, features, features, 3, depth, 0.3, early, False))


@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("depth", range(2, 9))
@pytest.mark.parametrize("features", [1, 2, 4, 30])
def test_values(ctx, depth, features, metric):
    import torch

    import paper_2511_09376_gb300 as wdf
    ens, C, B = _setup(depth, features)
    e = wdf.load_ensemble(ctx, ens)
    wdf.set_metric(e, ["shapley", "banzhaf"][metric])
    wdf.set_background(e, torch.from_numpy(B).cuda())
    got = wdf.explain(e, torch.from_numpy(C).cuda()).cpu().numpy()
    want = oracle.values_hist(ens, oracle.bg_hist(ens, B), B.shape[0], C, metric)
    assert_phi_close(got, want)
    assert abs(wdf.expected_value(e) - oracle.predict(ens, B).mean()) <= 1e-9 * max(1.0, np.abs(ens.value).max())
    e.close()


@pytest.mark.parametrize("depth", [2, 6, 8])
def test_large_counts(ctx, depth):
    """Counts times 2^23 for 500 rows: 4,194,304,000 rows with the same frequencies."""
    import torch

    import paper_2511_09376_gb300 as wdf
    ens, C, B = _setup(depth, 12, m=500)
    e = wdf.load_ensemble(ctx, ens)
    counts = wdf.background_counts(e, torch.from_numpy(B).cuda())
    Cd = torch.from_numpy(C).cuda()
    wdf.set_background_counts(e, counts, 500)
    want = wdf.explain(e, Cd).cpu().numpy()
    big = (counts.to(torch.int64) * (1 << 23)).to(torch.uint32 if counts.dtype == torch.uint32 else torch.int32)
    wdf.set_background_counts(e, big, 500 << 23)
    # every count, and so every product and sum, is the same number times a power of two
    np.testing.assert_array_equal(wdf.explain(e, Cd).cpu().numpy(), want)
    e.close()


@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("depth", range(2, 9))
@pytest.mark.parametrize("features", [2, 4, 30])
def test_pairs(ctx, depth, features, metric):
    import torch

    import paper_2511_09376_gb300 as wdf
    ens, C, B = _setup(depth, features)
    e = wdf.load_ensemble(ctx, ens)
    wdf.set_metric(e, ["shapley", "banzhaf"][metric])
    wdf.set_background(e, torch.from_numpy(B).cuda())
    got = wdf.explain_interactions(e, torch.from_numpy(C[:12]).cuda()).cpu().numpy()
    want = oracle.iv_hist(ens, oracle.bg_hist(ens, B), B.shape[0], C[:12], metric)
    assert_phi_close(got, want)
    e.close()

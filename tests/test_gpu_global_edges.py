"""Global attribution of packed rows against FP64 sums, at the edges of its runs, threads
and blocks, and for magnitudes that its FP32 parts cannot hold.  Tolerance: a run's sum is
within 2^-42 of its largest element times its length, so both means are within 1e-12 of the
mean magnitude."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _check(x):
    import torch

    import paper_2511_09376_gb300 as wdf
    ctx = wdf.ctx_create(0)
    ma, mn = wdf.global_attribution(ctx, torch.from_numpy(x).cuda())
    ma, mn = ma.cpu().numpy(), mn.cpu().numpy()
    with np.errstate(invalid="ignore"):
        d = x.astype(np.float64)
        want_abs, want = np.abs(d).mean(axis=0), d.mean(axis=0)
    fin = np.isfinite(want_abs)
    assert (np.abs(ma - want_abs)[fin] <= 1e-12 * want_abs[fin]).all()
    assert (np.abs(mn - want)[fin] <= 1e-12 * want_abs[fin]).all()
    np.testing.assert_array_equal(ma[~fin], want_abs[~fin])
    np.testing.assert_array_equal(mn[~fin], want[~fin])
    ctx.close()


@pytest.mark.parametrize("F", [1, 3, 20, 127, 128, 257, 500, 512])
@pytest.mark.parametrize("n", [1, 3, 31, 32, 33, 511, 9727, 9729, 40_003])
def test_sizes(F, n):
    rng = np.random.default_rng(F * 100_003 + n)
    scale = 10.0 ** rng.uniform(-6, 3, (1, F)) * 10.0 ** rng.uniform(-4, 0, (n, 1))
    _check((rng.standard_normal((n, F)) * scale).astype(np.float32))


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3e38, -2e37, 1e37, 1e-45, -1e-38])
def test_extremes(value):
    rng = np.random.default_rng(5)
    x = rng.standard_normal((5001, 40)).astype(np.float32)
    x[::7, 3] = value
    x[:, 5] = value
    x[17, 11] = value
    if value == np.inf:
        x[18, 11] = -np.inf
    _check(x)

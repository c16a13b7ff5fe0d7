"""Global attribution of packed rows: columns whose elements lie many binades apart lose nothing
that FP64 sums keep.

Tolerance.  Everything up to a thread's sum of three FP32 is exact to 2^-57 of a run's largest
element per run of sixteen (k_reduce.cu), so what remains are FP64 roundings, each at most
2^-53 of the sum of magnitudes: two in a thread's sum, one for each of the four threads of a
feature at F = 512, one for each of at most ceil(304 / 32) = 10 blocks that one thread of the second pass
adds and five levels of its tree, two in the division by n: 23 * 2^-53, and 2^-57 for the runs."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

F, TOL = 512, 23 * 2.0 ** -53 + 2.0 ** -57


def _rows(kind, n):
    rng = np.random.default_rng(n)
    row = np.arange(n)
    if kind == "one_large":  # a run's sixteen elements lie four rows apart: one large, fifteen below 2^-20 of it
        x = np.nextafter(np.float32(2.0 ** -20), np.float32(0)) * (1 - rng.integers(0, 1 << 10, (n, F)) * 2.0 ** -23)
        large = row // 4 % 16 == 0
        x[large] = 1 + rng.uniform(0, 1, (int(large.sum()), F))
        x *= np.where(row % 3 == 0, -1, 1)[:, None]
    elif kind == "all_binades":  # spans more than both cuts of a run
        x = rng.standard_normal((n, F)) * 2.0 ** rng.uniform(-60, 0, (n, F))
    elif kind == "subnormal":  # the second cut's power of two is below FP32's range
        x = rng.standard_normal((n, F)) * 2.0 ** rng.uniform(-149, -105, (n, F))
    else:
        x = rng.standard_normal((n, F)) * np.exp(4 * rng.standard_normal((n, 1)))
    return x.astype(np.float32)


@pytest.mark.parametrize("n", [300, 16_384, 20_001])
@pytest.mark.parametrize("kind", ["one_large", "all_binades", "subnormal", "log_normal"])
def test_rests(kind, n):
    import torch

    import paper_2511_09376_gb300 as wdf
    x = _rows(kind, n)
    ctx = wdf.ctx_create(0)
    ma, mn = wdf.global_attribution(ctx, torch.from_numpy(x).cuda())
    ma, mn = ma.cpu().numpy(), mn.cpu().numpy()
    ctx.close()
    d = x.astype(np.float64).T
    want_abs = np.array([math.fsum(c) for c in np.abs(d)]) / n
    want = np.array([math.fsum(c) for c in d]) / n
    assert (np.abs(ma - want_abs) <= TOL * want_abs).all()
    assert (np.abs(mn - want) <= TOL * want_abs).all()

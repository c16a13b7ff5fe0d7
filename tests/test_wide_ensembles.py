"""Wide ensembles: the widths whose tile of 32 rows needs the wide form of the consumer kernel.

On the CPU: every ensemble whose tile fits in the form with one or two bytes per code and a
tree or two staged per block (its size is restated here) fits a block in one of the kernel's two
forms.  On the GPU: at the largest of those widths, calls of few rows, of many, and batches give the
same bits, and values within the FP32 bar of the FP64 oracle."""
import ctypes

import numpy as np
import pytest

import oracle
import paper_2511_09376_gb300 as wdf
from conftest import assert_phi_close
from paper_2511_09376_gb300 import synth

SHARED = 232_448  # of a block
FLUSH = {2: 8, 3: 16, 4: 24, 5: 32, 6: 64, 7: 136, 8: 264}  # flush positions of a tree, per form below


def _up(v, to=16):
    return -(-v // to) * to


def _bytes_form(D, F, columns, code_bytes=1):
    """Codes of one or two bytes, phi rows of 33 floats, metadata and records of the staged trees."""
    trees, record = (1, 16) if D >= 7 else (2, 8)
    return (_up(32 * columns * code_bytes) + _up((F + 1) * 132) + _up(trees * 64) + (_up(trees * 48) if D <= 6 else 0) +
            _up(trees * (2 ** D - 1) * record) + _up(trees * FLUSH[D] * (2 if D >= 7 else 4)))


def _fits(D, F, quads):
    f = getattr(ctypes.CDLL(wdf.library_path()), "_ZN3wdf18explain_smem_bytesEiiiib")
    f.argtypes, f.restype = [ctypes.c_int] * 4 + [ctypes.c_bool], ctypes.c_size_t
    return min(f(D, F, quads, 32, False), f(D, F, quads, 32, True)) + 16 <= SHARED


def _widest(D, columns):
    return max(F for F in range(1, 1800) if _bytes_form(D, F, columns(F)) <= SHARED)


# quads of a column: 2 of 16 to 255 thresholds, 51 when 65,535 are cut into 17 columns
@pytest.mark.parametrize("depth", range(2, 9))
@pytest.mark.parametrize("columns,code_bytes,quads", [(lambda F: F, 1, 2), (lambda F: F, 2, 51), (lambda F: min(F, 1), 1, 1),
                                                      (lambda F: min(F, 300), 1, 2), (lambda F: F // 2, 2, 6)])
def test_widths_fit(depth, columns, code_bytes, quads):
    for F in range(1, 1800):
        if _bytes_form(depth, F, columns(F), code_bytes) <= SHARED:
            assert _fits(depth, F, quads * _up(columns(F), 8)), F


def _ensemble(rng, D, F, used, per_feature):
    """Complete trees whose nodes take the first `used` features in turn, per_feature or more thresholds each."""
    n_in, nodes = 2 ** D - 1, 2 ** (D + 1) - 1
    T = -(-used * per_feature // n_in)
    inner = np.tile(np.arange(nodes) < n_in, T)
    child = np.tile(np.arange(nodes), T)
    feature = np.full(T * nodes, -1, np.int32)
    feature[inner] = rng.permutation(T * n_in) % used
    return synth.Ensemble(F, nodes * np.arange(T + 1, dtype=np.int64), feature,
                          np.where(inner, rng.standard_normal(T * nodes), 0).astype(np.float32),
                          np.where(inner, 2 * child + 1, -1).astype(np.int32),
                          np.where(inner, 2 * child + 2, -1).astype(np.int32),
                          np.where(inner, 0, rng.normal(0, 0.1, T * nodes)).astype(np.float32))


@pytest.mark.gpu
@pytest.mark.parametrize("depth,few", [(2, False), (5, False), (6, False), (7, False), (8, False), (3, True), (7, True)])
def test_widest(depth, few):
    import torch
    rng = np.random.default_rng(depth)
    F = _widest(depth, (lambda f: min(f, 40)) if few else (lambda f: f))
    ens = _ensemble(rng, depth, F, 40 if few else F, 17)
    B = rng.standard_normal((130, F)).astype(np.float32)
    C = torch.from_numpy(rng.standard_normal((4003, F)).astype(np.float32)).cuda()
    ctx = wdf.ctx_create(0)
    e = wdf.load_ensemble(ctx, ens)
    wdf.set_background(e, torch.from_numpy(B).cuda())
    many = wdf.explain(e, C)
    rows = np.unique(np.concatenate([[0, 1, 31, 32, 33, 4002], rng.integers(0, 4003, 10)]))
    want = oracle.values_hist(ens, oracle.bg_hist(ens, B), B.shape[0], C.cpu().numpy()[rows])
    assert_phi_close(many.cpu().numpy()[rows], want, f"D={depth} F={F}")
    for n in (1, 33, 70):
        np.testing.assert_array_equal(wdf.explain(e, C[:n]).cpu().numpy(), many[:n].cpu().numpy())
    narrow_np, _, Bn = synth.make(synth.Workload("n", 5, 1, 60, 9, 9, 12, depth, 0.3, 0.1, False))
    narrow = wdf.load_ensemble(ctx, narrow_np)
    wdf.set_background(narrow, torch.from_numpy(Bn).cuda())
    Cn = C[:100, :9].contiguous()
    batch = wdf.batch_create(ctx, [narrow, e])
    reqs = [(1, C[:33]), (0, Cn), (1, C)]

    def check():
        got = wdf.batch_explain(batch, reqs)
        np.testing.assert_array_equal(got[0].cpu().numpy(), many[:33].cpu().numpy())
        np.testing.assert_array_equal(got[1].cpu().numpy(), wdf.explain(narrow, Cn).cpu().numpy())
        np.testing.assert_array_equal(got[2].cpu().numpy(), many.cpu().numpy())

    check()
    wdf.batch_autotune(batch, reqs, reps=1)
    check()
    batch.close()
    ctx.close()

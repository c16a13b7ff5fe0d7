"""Host threads inside wdf_explain at once, each with its own ensemble and stream: every call
succeeds and gives the bits that it gives alone.  The ensembles differ in what their kernels ask
for per block (thresholds to encode, features, trees).  Native threads, released together
before every call, so that the calls' launches interleave; row counts of the node-value route
and of tiles."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2511_09376_gb300 import synth

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
LIB = os.path.join(os.path.dirname(HERE), "paper_2511_09376_gb300", "libwoodelf.so")

HAMMER = r"""
#include <atomic>
#include <thread>
#include <vector>
#include "woodelf.h"
struct Job { wdf_ensemble *e; const float *C; int64_t n, F; float *phi; void *stream; };
extern "C" int hammer(decltype(&wdf_explain) explain, const Job *jobs, int count, int calls) {
    std::atomic<int> failed{0}, waiting{0}, turn{0};
    std::vector<std::thread> threads;
    for (int k = 0; k < count; ++k)
        threads.emplace_back([&, k] {
            const Job &j = jobs[k];
            for (int i = 0; i < calls; ++i) {
                if (waiting.fetch_add(1) + 1 == count) {  // a spinning barrier
                    waiting.store(0);
                    turn.store(i + 1);
                } else {
                    while (turn.load() < i + 1) {}
                }
                if (explain(j.e, j.C, j.n, j.F, WDF_MEM_DEVICE, j.phi, j.F, j.stream) != WDF_OK) failed.fetch_add(1);
            }
        });
    for (auto &t : threads) t.join();
    return failed.load();
}
"""


class _Job(ctypes.Structure):
    _fields_ = [("e", ctypes.c_void_p), ("C", ctypes.c_void_p), ("n", ctypes.c_int64), ("F", ctypes.c_int64),
                ("phi", ctypes.c_void_p), ("stream", ctypes.c_void_p)]


@pytest.mark.parametrize("rows,calls", [(40, 4000), (9000, 300)])
def test_explain_from_threads(tmp_path, rows, calls):
    import torch

    import paper_2511_09376_gb300 as wdf
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, so = tmp_path / "hammer.cpp", tmp_path / "hammer.so"
    src.write_text(HAMMER)
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-pthread", "-I",
                    os.path.join(os.path.dirname(HERE), "include"), str(src), "-o", str(so)], check=True)
    hammer = ctypes.CDLL(str(so)).hammer
    explain = ctypes.cast(ctypes.CDLL(LIB).wdf_explain, ctypes.c_void_p)
    ctx = wdf.ctx_create(0)
    held, jobs = [], (_Job * 4)()
    for k, (T, D, F) in enumerate([(3, 4, 10), (400, 6, 127), (12, 6, 300), (90, 4, 60)]):
        ens, C, B = synth.make(synth.Workload(f"t{k}", 40 + k, rows, 400, F, F, T, D, 0.2, 0.1, False))
        e = wdf.load_ensemble(ctx, ens)
        wdf.set_background(e, torch.from_numpy(B).cuda())
        C = torch.from_numpy(C).cuda()
        want, phi, stream = wdf.explain(e, C).cpu().numpy(), torch.empty_like(C), torch.cuda.Stream()
        jobs[k] = _Job(e.handle, C.data_ptr(), rows, F, phi.data_ptr(), stream.cuda_stream)
        held.append((e, C, phi, want, stream))
    torch.cuda.synchronize()
    failed = hammer(explain, jobs, len(held), calls)
    torch.cuda.synchronize()
    assert failed == 0
    for e, _, phi, want, _ in held:
        np.testing.assert_array_equal(phi.cpu().numpy(), want)
        e.close()
    ctx.close()

"""Calls inside a user's stream capture: the graph's replays, on changed rows, give the bits of
plain calls -- few rows (node values, dependent launches), whole tiles, split tiles and their
slices, wide tiles, a new background, pair values and global attribution, whose scratch then
belongs to the graph."""
import numpy as np
import pytest

from paper_2511_09376_gb300 import synth

pytestmark = pytest.mark.gpu


def _setup(D, T, F):
    import torch

    import paper_2511_09376_gb300 as wdf
    ctx = wdf.ctx_create(0)
    ens, _, B = synth.make(synth.Workload("g", 90 + D, 1, 700, F, F, T, D, 0.3, 0.1, False))
    e = wdf.load_ensemble(ctx, ens)
    wdf.set_background(e, torch.from_numpy(B).cuda())
    return torch, wdf, ctx, e


def _captured(torch, call):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    return graph


# node values (one tree, one row; several parts), whole tiles, parts on several blocks, slices, wide tiles
@pytest.mark.parametrize("D,T,F,n", [(6, 1, 9, 1), (7, 120, 20, 70), (4, 30, 40, 30_001), (8, 101, 40, 5_000),
                                     (8, 100, 134, 90_000), (6, 40, 1_700, 3_000)])
def test_explain(D, T, F, n):
    torch, wdf, ctx, e = _setup(D, T, F)
    C = torch.randn((n, F), device="cuda")
    out = torch.empty_like(C)
    wdf.explain(e, C, out)
    torch.cuda.synchronize()
    graph = _captured(torch, lambda: wdf.explain(e, C, out))
    for seed in (1, 2):
        C.copy_(torch.randn((n, F), device="cuda", generator=torch.Generator("cuda").manual_seed(seed)))
        out.fill_(float("nan"))
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        got = out.clone()
        assert torch.equal(got, wdf.explain(e, C))
    del graph
    ctx.close()


def test_background_pairs_and_global():
    torch, wdf, ctx, e = _setup(6, 20, 12)
    B, C = torch.randn((900, 12), device="cuda"), torch.randn((333, 12), device="cuda")
    phi, pairs = torch.empty_like(C), torch.empty((333, 12, 12), device="cuda")
    means = []

    def call():
        wdf.set_background(e, B)
        wdf.explain(e, C, phi)
        wdf.explain_interactions(e, C, pairs)
        means[:] = wdf.global_attribution(ctx, phi)

    call()
    torch.cuda.synchronize()
    graph = _captured(torch, call)
    B.copy_(torch.randn((900, 12), device="cuda"))
    C.copy_(torch.randn((333, 12), device="cuda"))
    graph.replay()
    torch.cuda.synchronize()
    got = [phi.clone(), pairs.clone(), *[m.clone() for m in means]]
    call()
    torch.cuda.synchronize()
    assert torch.equal(got[0], phi)
    np.testing.assert_allclose(got[1].cpu().numpy(), pairs.cpu().numpy(), rtol=1e-5, atol=1e-6)  # scheduling-dependent
    assert torch.equal(got[2], means[0]) and torch.equal(got[3], means[1])
    del graph
    ctx.close()

"""Contraction into few, large clusters: clusters of many vertices without
entries are not one warp's walk, warps whose vertices share a cluster and warps
whose vertices do not (with vertex weights and without), and a cut mesh costs no
more than one contracted as in coarsening, give or take a small factor."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _ms(f):
    f()
    best = []
    for _ in range(3):
        torch.cuda.synchronize()
        b, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        b.record()
        r = f()
        e.record()
        torch.cuda.synchronize()
        best.append(b.elapsed_time(e))
        del r
    return min(best)


def test_vertices_without_entries():
    n = 1 << 22
    g = tp.graph_from_csr(torch.zeros(n + 1, dtype=torch.int64, device="cuda"),
                          torch.zeros(0, dtype=torch.int32, device="cuda"))
    u = torch.arange(n, dtype=torch.int32, device="cuda")
    for C, nc in ((torch.full_like(u, 7), 1), (u % 64, 64)):
        cg, mp = tp.contract(g, C)
        x, a, vw, ew = cg.export_csr()
        assert len(x) == nc + 1 and len(a) == len(ew) == 0 and bool((vw == n // nc).all())
        assert torch.equal(mp, C - C.min())
    usual = _ms(lambda: tp.contract(g, u // 64))
    assert _ms(lambda: tp.contract(g, torch.full_like(u, 7))) < 10 * usual
    assert _ms(lambda: tp.contract(g, u % 64)) < 10 * usual


def test_cut_mesh():
    n = 1 << 22
    z = tp.graph_from_csr(*synth.rgg2d(n, 16.0, 3)).compress()
    u = torch.arange(n, dtype=torch.int64, device="cuda")
    usual = _ms(lambda: tp.contract(z, (u // 16).to(torch.int32)))
    assert _ms(lambda: tp.contract(z, (u * 64 // n).to(torch.int32))) < 3 * usual


@pytest.mark.parametrize("graph", ["mesh", "skewed", "dense"])
@pytest.mark.parametrize("weighted", [False, True])
def test_contraction_equals_oracle(graph, weighted):
    xadj, adj = {"mesh": lambda: synth.rgg2d(30011, 16.0, 3), "skewed": lambda: synth.rmat(13, 24, seed=4),
                 "dense": lambda: synth.gnm(2003, 90000, 5)}[graph]()
    n = len(xadj) - 1
    vw = ew = None
    if weighted:
        u = np.repeat(np.arange(n, dtype=np.int64), np.diff(xadj))
        ew = (np.minimum(u, adj) * 7919 + np.maximum(u, adj) * 104729) % 9 + 1
        vw = np.arange(n, dtype=np.int64) % 5 + 1
    og, g = oracle.Graph(xadj, adj, vw, ew), tp.graph_from_csr(xadj, adj, vw, ew)
    ids = np.arange(n, dtype=np.int64)
    for C in (ids * 4 // n, ids * 64 // n * 3, ids % 5, np.where(ids % 70 < 64, 0, ids), 0 * ids):
        C = C.astype(np.int32)
        want, want_map = oracle.contract(og, C)
        for q in [g] if weighted else [g, g.compress()]:
            cg, mp = tp.contract(q, torch.from_numpy(C).cuda())
            x, a, w, e = (t.cpu().numpy() for t in cg.export_csr())
            assert np.array_equal(mp.cpu().numpy(), want_map)
            assert np.array_equal(x, want.xadj) and np.array_equal(a, want.adj)
            assert np.array_equal(w, want.vw) and np.array_equal(e, want.ew)

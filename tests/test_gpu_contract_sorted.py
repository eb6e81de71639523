"""Contractions whose rows are all sorted at once (skewed graphs of a middle
size, and small compressed ones with long records, by chunks), on both sides of
the bounds, against the oracle; and what they cost beside a mesh of the size."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _check(g, og, C):
    want, want_map = oracle.contract(og, C)
    cg, mp = tp.contract(g, torch.from_numpy(C).cuda())
    x, a, w, e = (t.cpu().numpy() for t in cg.export_csr())
    assert np.array_equal(mp.cpu().numpy(), want_map)
    assert np.array_equal(x, want.xadj) and np.array_equal(a, want.adj)
    assert np.array_equal(w, want.vw) and np.array_equal(e, want.ew)


@pytest.mark.parametrize("scale", [12, 14, 16, 18])  # 1e5 to 8e6 entries
def test_skewed_graphs_equal_oracle(scale):
    xadj, adj = synth.rmat(scale, 18, seed=scale)
    n = len(xadj) - 1
    u = np.repeat(np.arange(n, dtype=np.int64), np.diff(xadj))
    lo, hi = np.minimum(u, adj), np.maximum(u, adj)
    vw = np.arange(n, dtype=np.int64) % 5 + 1
    g = tp.graph_from_csr(xadj, adj)
    z = g.compress()
    for cap in (8, n // 60):
        C = tp.lp_cluster(g, cap).cpu().numpy()
        for q in (g, z):
            _check(q, oracle.Graph(xadj, adj), C)
        for top in (50, 1 << 40):  # weights beside the keys, and apart
            ew = (lo * 7919 + hi * 104729) % top + 1
            _check(tp.graph_from_csr(xadj, adj, vw, ew), oracle.Graph(xadj, adj, vw, ew), C)


def test_chunked_records_without_a_copy():
    """A hub of 70 chunks in a compressed graph that is not decoded."""
    n, d = 90001, 70001
    mesh = synth.rgg2d(n, 6.0, 3)
    u = np.repeat(np.arange(n, dtype=np.int64), np.diff(mesh[0]))
    spokes = np.arange(1, d + 1, dtype=np.int64)
    key = np.unique(np.concatenate([u * n + mesh[1], spokes, spokes * n]))
    xadj = np.zeros(n + 1, np.int64)
    np.add.at(xadj, key // n + 1, 1)
    xadj, adj = np.cumsum(xadj), (key % n).astype(np.int32)
    z = tp.graph_from_csr(xadj, adj).compress()
    for C in (np.arange(n), np.arange(n) // 7 * 7, np.arange(n) * 3 // n):
        _check(z, oracle.Graph(xadj, adj), C.astype(np.int32))


def test_small_skewed_graphs_cost_little():
    def ms(f):
        f()
        best = []
        for _ in range(5):
            torch.cuda.synchronize()
            b, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            b.record()
            f()
            e.record()
            torch.cuda.synchronize()
            best.append(b.elapsed_time(e))
        return min(best)

    n = 1 << 16
    skewed, mesh = (tp.graph_from_csr(*x).compress() for x in (synth.rmat(16, 12, seed=2), synth.rgg2d(n, 20.0, 2)))
    Cs, Cm = tp.lp_cluster(skewed, n // 60), tp.lp_cluster(mesh, n // 60)
    assert ms(lambda: tp.contract(skewed, Cs)) < 4 * ms(lambda: tp.contract(mesh, Cm))

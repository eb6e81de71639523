"""Device memory of the contraction: the rows of its tables take the room that
they need (and are summed again where a sample of the graph promised too few
inter-cluster entries), and a compressed graph with long records that there is
no room to decode is contracted from its records."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _equal(cg, mp, want, want_map):
    x, a, w, e = (t.cpu().numpy() for t in cg.export_csr())
    assert np.array_equal(mp.cpu().numpy(), want_map)
    assert np.array_equal(x, want.xadj) and np.array_equal(a, want.adj)
    assert np.array_equal(w, want.vw) and np.array_equal(e, want.ew)


def test_peak_of_a_mesh():
    """The labels, weights and mover lists of clustering are the peak, not the
    entries of the contraction."""
    n = 1 << 21
    g = tp.graph_from_csr(*synth.rgg2d(n, 16.0, 5))
    for q in (g, g.compress()):
        _, st = tp.partition(q, 64, 0.03)
        assert st["peak_bytes"] < 125 * n


@pytest.mark.parametrize("weighted", [False, True])
def test_sample_that_falls_short(weighted):
    """A path in clusters of 64, and, between two sampled vertices, 800 vertices
    of which each half is joined to all of the other, alone in their clusters."""
    n, at, half = 1 << 20, (1 << 19) + 100, 400
    u = np.arange(n - 1, dtype=np.int64)
    left = at + np.arange(half)
    heavy = np.stack([np.repeat(left, half), np.tile(left + half, half)], 1)
    e = np.concatenate([np.stack([u, u + 1], 1), heavy])
    e = np.concatenate([e, e[:, ::-1]])
    key = np.unique(e[:, 0] * n + e[:, 1])
    x = np.zeros(n + 1, np.int64)
    np.add.at(x, key // n + 1, 1)
    xadj, adj = np.cumsum(x), (key % n).astype(np.int32)
    C = (np.arange(n) // 64 * 64).astype(np.int32)
    C[at - 100 : at + 2 * half + 100] = np.arange(at - 100, at + 2 * half + 100)
    vw = ew = None
    if weighted:
        src = np.repeat(np.arange(n, dtype=np.int64), np.diff(xadj))
        ew = (np.minimum(src, adj) * 7919 + np.maximum(src, adj) * 104729) % 9 + (1 << 40)
        vw = np.arange(n, dtype=np.int64) % 5 + 1
    want, want_map = oracle.contract(oracle.Graph(xadj, adj, vw, ew), C)
    g = tp.graph_from_csr(xadj, adj, vw, ew)
    for q in [g] if weighted else [g, g.compress()]:
        _equal(*tp.contract(q, torch.from_numpy(C).cuda()), want, want_map)


def test_no_room_to_decode():
    """With less memory than the decoded copy and the rows take together the
    records are contracted, with far less than either the call fails cleanly."""
    n, d = 700001, 5000  # a mesh with a hub, more than 2^23 entries (smaller ones are not decoded)
    mesh = synth.rgg2d(n, 16.0, 3)
    u = np.repeat(np.arange(n, dtype=np.int64), np.diff(mesh[0]))
    spokes = np.arange(1, d + 1, dtype=np.int64) * (n // (d + 1))
    key = np.unique(np.concatenate([u * n + mesh[1], spokes, spokes * n]))
    xadj = np.zeros(n + 1, np.int64)
    np.add.at(xadj, key // n + 1, 1)
    xadj, adj = np.cumsum(xadj), (key % n).astype(np.int32)
    assert len(adj) > 1 << 23 and np.diff(xadj).max() > 1024
    z = tp.graph_from_csr(xadj, adj).compress()
    C = tp.lp_cluster(z, 300)
    want, want_map = oracle.contract(oracle.Graph(xadj, adj), C.cpu().numpy())
    live, peak, limit = {}, [0], [1 << 60]

    def alloc(nbytes, stream):
        if sum(live.values()) + nbytes > limit[0]:
            return 0
        p = torch.cuda.caching_allocator_alloc(nbytes, stream=stream)
        live[p] = nbytes
        peak[0] = max(peak[0], sum(live.values()))
        return p

    def free(ptr, nbytes, stream):
        live.pop(ptr)
        torch.cuda.caching_allocator_delete(ptr)

    tp.set_allocator(alloc, free)
    try:
        cg, mp = tp.contract(z, C)
        _equal(cg, mp, want, want_map)
        del cg
        base = sum(live.values())
        limit[0] = peak[0] - 1  # the copy and its rows do not fit together
        for _ in range(2):
            peak[0] = base
            cg, mp = tp.contract(z, C)
            _equal(cg, mp, want, want_map)
            del cg, mp
        limit[0] = 4 * len(adj)  # not even the copy: refused as before, nothing leaks
        with pytest.raises(tp.TpError):
            tp.contract(z, C)
        torch.cuda.synchronize()
        assert sum(live.values()) == base
    finally:
        tp.set_allocator(None, None)

"""Contraction through every table size and the sort behind them: coarse
vertices whose distinct neighbours just fit a table or just overflow it (and
move on to the next), many members per coarse vertex and one, rows walked by a
lane or a warp, sums in 32 and 64 bits, against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402

DEGREES = (31, 32, 33, 192, 193, 768, 769, 2816, 2817, 4096, 4097, 8192, 8193, 10240, 10241, 41000)


@pytest.fixture(scope="module")
def csr():
    """Hubs of those degrees among 41 000 leaves that form a path."""
    leaves, hubs = 41000, len(DEGREES)
    n = hubs + leaves
    pairs = [np.stack([np.full(d, h), hubs + (np.arange(d) * 7 % leaves if d < leaves else np.arange(d))], 1)
             for h, d in enumerate(DEGREES)]
    v = hubs + np.arange(leaves)
    pairs.append(np.stack([v[:-1], v[1:]], 1))
    e = np.concatenate(pairs).astype(np.int64)
    e = np.concatenate([e, e[:, ::-1]])
    key = np.unique(e[:, 0] * n + e[:, 1])
    x = np.zeros(n + 1, np.int64)
    np.add.at(x, key // n + 1, 1)
    return np.cumsum(x), (key % n).astype(np.int32), hubs


def _weights(xadj, adj, top):
    n = len(xadj) - 1
    u = np.repeat(np.arange(n, dtype=np.uint64), np.diff(xadj))
    lo, hi = np.minimum(u, adj.astype(np.uint64)), np.maximum(u, adj.astype(np.uint64))
    h = (lo * np.uint64(0x9E3779B97F4A7C15) ^ hi * np.uint64(0xC2B2AE3D27D4EB4F)) >> np.uint64(13)
    return (h % np.uint64(top) + np.uint64(1)).astype(np.int64)


def _clusterings(n, hubs):
    ident = np.arange(n, dtype=np.int32)
    yield "each vertex", ident
    triples = ident.copy()
    triples[hubs:] = hubs + (ident[hubs:] - hubs) // 3 * 3
    yield "leaves in threes", triples
    wide = ident.copy()  # one cluster of many low-degree members, one of all hubs
    wide[hubs : hubs + 20000] = hubs + 11
    wide[:hubs] = 5
    yield "two large clusters", wide
    half = ident.copy()  # a cluster of 3000 members that reaches 3000 and more others
    half[hubs : hubs + 6000 : 2] = hubs
    yield "every second leaf", half
    yield "all", np.full(n, n - 1, np.int32)


@pytest.mark.parametrize("top", [0, 50, 1 << 40])
def test_contraction_equals_oracle(csr, top):
    xadj, adj, hubs = csr
    n = len(xadj) - 1
    ew = _weights(xadj, adj, top) if top else None
    vw = np.random.default_rng(3).integers(1, 9, n).astype(np.int64) if top else None
    og = oracle.Graph(xadj, adj, vw, ew)
    g = tp.graph_from_csr(xadj, adj, vw, ew)
    for name, C in _clusterings(n, hubs):
        want, want_map = oracle.contract(og, C)
        for gr in [g] if top else [g, g.compress()]:
            cg, mp = tp.contract(gr, torch.from_numpy(C).cuda())
            x, a, w, e = (t.cpu().numpy() for t in cg.export_csr())
            assert np.array_equal(mp.cpu().numpy(), want_map), name
            assert np.array_equal(x, want.xadj) and np.array_equal(a, want.adj), name
            assert np.array_equal(w, want.vw) and np.array_equal(e, want.ew), name

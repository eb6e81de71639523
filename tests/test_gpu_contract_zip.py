"""Contraction of compressed graphs whose degrees stay below the point from
which they are decoded first, through every table size and the sort behind
them: coarse vertices whose distinct neighbours just fit a table or just
overflow it (and move on to the next), records walked by a lane or a warp,
more long records than a block lists, against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402

# distinct neighbours of a group of hubs, each hub joined to up to REACH leaves
GROUPS = (31, 32, 33, 192, 193, 768, 769, 2816, 2817, 8192, 8193, 10240, 10241, 16500)
REACH = 1000
LEAVES = 16500


@pytest.fixture(scope="module")
def csr():
    """The groups' hubs, then leaves that form a path."""
    first, pairs, h = [], [], 0
    for d in GROUPS:
        first.append(h)
        for lo in range(0, d, REACH):
            leaf = np.arange(lo, min(lo + REACH, d))
            pairs.append(np.stack([np.full(len(leaf), h), leaf], 1))
            h += 1
    hubs = h
    e = np.concatenate(pairs).astype(np.int64)
    e[:, 1] += hubs
    v = hubs + np.arange(LEAVES)
    e = np.concatenate([e, np.stack([v[:-1], v[1:]], 1)])
    e = np.concatenate([e, e[:, ::-1]])
    n = hubs + LEAVES
    key = np.unique(e[:, 0] * n + e[:, 1])
    x = np.zeros(n + 1, np.int64)
    np.add.at(x, key // n + 1, 1)
    return np.cumsum(x), (key % n).astype(np.int32), np.array(first), hubs


def _clusterings(n, first, hubs):
    ident = np.arange(n, dtype=np.int32)
    yield "each vertex", ident
    group = ident.copy()
    group[:hubs] = first[np.searchsorted(first, np.arange(hubs), side="right") - 1]
    yield "groups", group
    both = group.copy()
    both[hubs:] = hubs + (ident[hubs:] - hubs) // 3 * 3
    yield "groups, leaves in threes", both
    one = ident.copy()
    one[:hubs] = 3
    yield "all hubs", one
    far = ident.copy()  # a cluster of many short records that reaches thousands of others
    far[hubs : hubs + 9000 : 2] = hubs
    yield "every second leaf", far
    yield "all", np.full(n, n - 1, np.int32)


def test_contraction_equals_oracle(csr):
    xadj, adj, first, hubs = csr
    n = len(xadj) - 1
    assert np.diff(xadj).max() <= 1024  # beyond that a compressed graph is decoded first
    og = oracle.Graph(xadj, adj)
    z = tp.graph_from_csr(xadj, adj).compress()
    for name, C in _clusterings(n, first, hubs):
        want, want_map = oracle.contract(og, C)
        cg, mp = tp.contract(z, torch.from_numpy(C).cuda())
        x, a, w, e = (t.cpu().numpy() for t in cg.export_csr())
        assert np.array_equal(mp.cpu().numpy(), want_map), name
        assert np.array_equal(x, want.xadj) and np.array_equal(a, want.adj), name
        assert np.array_equal(w, want.vw) and np.array_equal(e, want.ew), name


def test_many_long_records_in_one_cluster():
    """More records above the lane decoder's degree than a block lists."""
    import synth

    xadj, adj = synth.gnm(2003, 60000, 4)
    n = len(xadj) - 1
    for C in (np.where(np.arange(n) < 700, 0, np.arange(n)), np.arange(n) // 400 * 400):
        C = C.astype(np.int32)
        want, _ = oracle.contract(oracle.Graph(xadj, adj), C)
        cg, _ = tp.contract(tp.graph_from_csr(xadj, adj).compress(), torch.from_numpy(C).cuda())
        x, a, w, e = (t.cpu().numpy() for t in cg.export_csr())
        assert np.array_equal(x, want.xadj) and np.array_equal(a, want.adj)
        assert np.array_equal(w, want.vw) and np.array_equal(e, want.ew)

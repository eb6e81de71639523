"""Validation, encoding and decoding in tiles of adjacency entries: rows that
begin, end and span tile borders (2048 entries), empty rows there and at both
ends, chunked hubs, records decoded by a lane, by a warp and by chunks; and
what has to be refused."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _csr(n, pairs):
    e = np.concatenate([pairs, pairs[:, ::-1]])
    key = np.unique(e[:, 0].astype(np.int64) * n + e[:, 1])
    key = key[key // n != key % n]
    x = np.zeros(n + 1, np.int64)
    np.add.at(x, key // n + 1, 1)
    return np.cumsum(x), (key % n).astype(np.int32)


def _path(entries, lead, gap, trail):
    """A path with the given number of adjacency entries (even), its vertices
    `gap` ids apart, `lead` empty rows before and `trail` behind."""
    m = entries // 2
    v = lead + gap * np.arange(m + 1)
    return _csr(int(v[-1]) + 1 + trail, np.stack([v[:-1], v[1:]], 1))


def _star(leaves, at):
    """A hub numbered `at` among its leaves, which form a path."""
    v = np.array([x for x in range(leaves + 1) if x != at])
    return _csr(leaves + 1, np.concatenate([np.stack([np.full(leaves, at), v], 1),
                                            np.stack([v[:-1], v[1:]], 1)]))


CASES = {
    "empty": lambda: (np.zeros(1, np.int64), np.zeros(0, np.int32)),
    "no_edges": lambda: (np.zeros(5001, np.int64), np.zeros(0, np.int32)),
    **{f"path_{e}_{lead}_{gap}_{trail}": (lambda e=e, lead=lead, gap=gap, trail=trail:
                                         _path(e, lead, gap, trail))
       for e in (2, 2046, 2048, 2050, 4096, 6146)
       for lead, gap, trail in ((0, 1, 0), (3, 1, 2), (4000, 3, 5000))},
    **{f"star_{d}_{at}": (lambda d=d, at=at: _star(d, at))
       for d, at in ((127, 0), (128, 60), (129, 0), (2047, 2047), (2048, 5), (10000, 0),
                     (10001, 5000), (30500, 17), (30500, 30500))},
    # first codes and gaps of five bytes
    "wide_gaps": lambda: _csr((1 << 28) + 8, np.array([[0, (1 << 28) + 7], [5, (1 << 28) + 6], [5, 6]])),
    "rmat": lambda: synth.rmat(12, 16, seed=5),
    "rgg": lambda: synth.rgg2d(20011, 16.0, 2),
}


@pytest.mark.parametrize("name", CASES)
def test_round_trip_equals_oracle(name):
    xadj, adj = CASES[name]()
    n = len(xadj) - 1
    dx, da = torch.from_numpy(xadj).cuda(), torch.from_numpy(adj).cuda()
    g = tp.graph_from_csr(dx, da)
    z = g.compress()
    data, off = z.export_compressed()
    for d in (z, tp.graph_from_compressed(n, data, off)):
        x2, a2, _, _ = d.decompress().export_csr()
        assert torch.equal(x2, dx) and torch.equal(a2, da)
    if n < 1 << 20:
        want_data, want_off = oracle.encode(xadj, adj)
        assert np.array_equal(data.cpu().numpy(), want_data)
        assert np.array_equal(off.cpu().numpy().astype(np.uint64), want_off)


def _refused(make):
    with pytest.raises(tp.TpError) as e:
        make()
    assert e.value.code == 1


@pytest.mark.parametrize("name", ["path_4096_3_1_2", "star_10001_5000", "rmat"])
def test_invalid_csr_is_refused(name):
    xadj, adj = CASES[name]()
    n, m2 = len(xadj) - 1, len(adj)
    ew = np.ones(m2, np.int64)
    tp.graph_from_csr(xadj, adj, np.ones(n, np.int64), ew)
    u = np.repeat(np.arange(n), np.diff(xadj))
    for at in (0, m2 // 2, m2 - 1, 2047, 2048):
        at = min(at, m2 - 1)
        for value in (-1, n, int(u[at])):  # out of range, a loop
            bad = adj.copy()
            bad[at] = value
            _refused(lambda: tp.graph_from_csr(xadj, bad))
        w = ew.copy()
        w[at] = 0
        _refused(lambda: tp.graph_from_csr(xadj, adj, None, w))
        w[at] = 2  # its mirror still weighs 1
        _refused(lambda: tp.graph_from_csr(xadj, adj, None, w))
    # two neighbours swapped; a neighbour twice
    row = int(np.flatnonzero(np.diff(xadj) >= 2)[-1])
    b = int(xadj[row])
    bad = adj.copy()
    bad[b], bad[b + 1] = adj[b + 1], adj[b]
    _refused(lambda: tp.graph_from_csr(xadj, bad))
    bad[b] = bad[b + 1] = adj[b]
    _refused(lambda: tp.graph_from_csr(xadj, bad))
    # one entry without a mirror, above and below the diagonal: the entries
    # above and below still balance, or a lower mirror is missing
    for side in (1, -1):
        cand = np.flatnonzero((adj - u) * side > 0)
        for at in (cand[0], cand[-1]):
            keep = np.arange(m2) != at
            x = xadj.copy()
            x[u[at] + 1 :] -= 1
            _refused(lambda: tp.graph_from_csr(x, adj[keep]))
    x = xadj.copy()
    x[n // 2] = x[n] + 1
    _refused(lambda: tp.graph_from_csr(x, adj))
    x[n // 2] = -1
    _refused(lambda: tp.graph_from_csr(x, adj))
    vw = np.ones(n, np.int64)
    vw[n - 1] = 0
    _refused(lambda: tp.graph_from_csr(xadj, adj, vw))


def test_swapped_mirrors_are_refused():
    # 0-1, 2-3 stored as 0->1, 1->2, 2->1, 3->2: as many entries above the
    # diagonal as below, every row ascends, but 0->1 has no mirror
    xadj = np.array([0, 1, 2, 3, 4], np.int64)
    _refused(lambda: tp.graph_from_csr(xadj, np.array([1, 2, 1, 2], np.int32)))


@pytest.mark.parametrize("name", ["path_4096_3_1_2", "star_129_0", "star_10001_5000"])
def test_corrupt_streams_are_refused(name):
    xadj, adj = CASES[name]()
    n = len(xadj) - 1
    data, off = oracle.encode(xadj, adj)

    def refused(d, o=off):
        with pytest.raises(tp.TpError) as e:
            tp.graph_from_compressed(n, d, o)
        assert e.value.code == 4

    tp.graph_from_compressed(n, data, off)
    deg = np.diff(xadj)
    for u in (int(np.argmax(deg)), int(np.flatnonzero(deg)[0])):
        lo, hi = int(off[u]), int(off[u + 1])
        for p in {hi - 1, hi - 2, (lo + hi) // 2}:
            for v in (0x80, 0xFF):  # an unfinished or overlong VarInt
                bad = data.copy()
                bad[p] |= v
                if bad[p] != data[p]:
                    refused(bad)
        if deg[u] > 1:
            bad = data.copy()
            bad[hi - 1] = 0  # a gap of zero
            refused(bad)
    if deg.max() > 10000:  # chunk offsets out of order or behind the record
        u = int(np.argmax(deg))
        t = int(off[u]) + len(oracle.varint(int(xadj[u])))
        for raw in (0, 0x7FFFFFFF):
            bad = data.copy()
            bad[t : t + 4] = np.frombuffer(np.uint32(raw).tobytes(), np.uint8)
            refused(bad)
    o = off.copy()
    o[n // 2] = len(data)
    refused(data, o)
    o[n // 2] = off[n // 2 + 1] + 1
    refused(data, o)

"""Bisection nodes around the sizes and entry counts at which the kernel's form
changes, against the oracle: the shared-memory state holds 12 512 vertices, or
10 224 with 64-bit connectivity differences, and nodes of more than 2^19
entries go to clusters; as a root, as nodes of one depth side by side and as
children."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _edge_weights(xadj, adj, top):
    """Symmetric edge weights of 1 .. top."""
    n = len(xadj) - 1
    u = np.repeat(np.arange(n, dtype=np.uint64), np.diff(xadj))
    lo, hi = np.minimum(u, adj.astype(np.uint64)), np.maximum(u, adj.astype(np.uint64))
    h = (lo * np.uint64(0x9E3779B97F4A7C15) ^ hi * np.uint64(0xC2B2AE3D27D4EB4F)) >> np.uint64(13)
    return (h % np.uint64(top) + np.uint64(1)).astype(np.int64)


def _check(xadj, adj, ew, k):
    n = len(xadj) - 1
    l_max = 1030 * -(-n // k) // 1000
    want = oracle.initial_partition(oracle.Graph(xadj, adj, None, ew), k, l_max, oracle.Params(seed=5))
    got = tp.initial_partition(tp.graph_from_csr(xadj, adj, None, ew), k, l_max, tp.default_params(seed=5))
    assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("n", [12496, 12511, 12512, 12513, 12514, 12515, 12528, 12529])
def test_root_around_the_capacity(n):
    xadj, adj = synth.gnm(n, 3 * n, n)
    _check(xadj, adj, None, 2)


@pytest.mark.parametrize("n", [10208, 10223, 10224, 10225, 10239, 10240, 10241])
def test_root_around_the_capacity_of_wide_differences(n):
    xadj, adj = synth.gnm(n, 3 * n, n)
    _check(xadj, adj, _edge_weights(xadj, adj, 1 << 40), 2)


@pytest.mark.parametrize("m", [(1 << 18) - 1, 1 << 18, (1 << 18) + 1])  # 2^19 entries and around
def test_root_around_the_entries_of_a_cluster(m):
    xadj, adj = synth.gnm(3001, m, 7)
    _check(xadj, adj, None, 3)


@pytest.mark.parametrize("top", [0, 1 << 40])
def test_children_around_the_capacity(top):
    """Two equal halves without an edge between them: the root's split falls
    between them, or near it."""
    half = 10232 if top else 12513
    x, a = synth.gnm(half, 3 * half, 11)
    xadj = np.concatenate([x, x[-1] + x[1:]])
    adj = np.concatenate([a, a + half]).astype(np.int32)
    _check(xadj, adj, _edge_weights(xadj, adj, top) if top else None, 4)


def test_classes_of_one_depth_side_by_side():
    """A batch whose coarsest graphs are the graphs themselves (n <= 160 k):
    clusters, the largest shared-memory nodes and small ones in one depth."""
    sizes = [300, 2000, 7000, 12512, 12513, 12514, 12529, 16003]
    host = [synth.gnm(n, 3 * n, n) for n in sizes]
    k = 128
    graphs = [tp.graph_from_csr(x, a) for x, a in host]
    res = tp.partition_batch(graphs, [k] * len(sizes), 0.03, tp.default_params(seed=3))
    for (x, a), (part, st) in zip(host, res):
        want, wst = oracle.partition(oracle.Graph(x, a), k, 0.03, oracle.Params(seed=3))
        assert np.array_equal(part.cpu().numpy(), want) and st["cut"] == wst["cut"]


def _joined(parts):
    """The graphs side by side, an edge from each one's last vertex to the next one's first."""
    u, v, base = [], [], 0
    for x, a in parts:
        n = len(x) - 1
        u.append(np.repeat(np.arange(n), np.diff(x)) + base)
        v.append(a.astype(np.int64) + base)
        if base:
            u.append(np.array([base - 1, base]))
            v.append(np.array([base, base - 1]))
        base += n
    u, v = np.concatenate(u), np.concatenate(v)
    order = np.lexsort((v, u))
    x = np.zeros(base + 1, np.int64)
    np.add.at(x, u + 1, 1)
    return np.cumsum(x), v[order].astype(np.int32)


def _path(n):
    u = np.arange(n)
    a = np.stack([u - 1, u + 1], 1).reshape(-1)[1:-1].astype(np.int32)
    return np.concatenate([[0], 1 + 2 * np.arange(n - 1), [2 * (n - 1)]]).astype(np.int64), a


@pytest.mark.parametrize("parts", ["path", "narrow and wide", "star"])
def test_narrow_and_wide_levels_of_a_cluster(parts):
    """Nodes of clusters whose BFS has levels of a vertex or two, of hundreds
    and of thousands, in turn."""
    graphs = {"path": [_path(14003)],
              "narrow and wide": [_path(3000), synth.gnm(6001, 60000, 3), _path(2500),
                                  synth.gnm(3001, 500000, 4), _path(900)],
              "star": [_path(5000), (np.concatenate([[0], 8000 + np.arange(8001)]).astype(np.int64),
                                     np.concatenate([1 + np.arange(8000), np.zeros(8000)]).astype(np.int32)),
                       _path(700)]}[parts]
    xadj, adj = _joined(graphs)
    _check(xadj, adj, None, 3)


def test_narrow_levels_cost_a_cluster_no_more_than_one_block():
    """A path just too long for shared memory against one that just fits."""
    def ms(n):
        g = tp.graph_from_csr(*_path(n))
        best = []
        for _ in range(3):
            torch.cuda.synchronize()
            b, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            b.record()
            tp.initial_partition(g, 2, n)
            e.record()
            torch.cuda.synchronize()
            best.append(b.elapsed_time(e))
        return min(best)

    assert ms(13000) < 2 * ms(12500)

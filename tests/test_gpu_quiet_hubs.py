"""Rounds that leave quiet vertices out of a mesh with hubs among the movers:
vertices of every degree class that a move wakes (a thread, a warp, a block, a
block by chunks) and one beyond which it ends all marks, against the oracle;
and what hubs cost."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _mesh_with_spokes(n, deg, spokes):
    """A mesh and vertices joined to every (n // d)-th vertex."""
    xadj, adj = synth.rgg2d(n, deg, 4)
    u = np.repeat(np.arange(n), np.diff(xadj))
    e = [np.stack([u, adj], 1)]
    for h, d in spokes:
        v = np.arange(d) * (n // d)
        v = v[v != h]
        e += [np.stack([np.full(len(v), h), v], 1), np.stack([v, np.full(len(v), h)], 1)]
    e = np.concatenate(e)
    key = np.unique(e[:, 0].astype(np.int64) * n + e[:, 1])
    x = np.zeros(n + 1, np.int64)
    np.add.at(x, key // n + 1, 1)
    return np.cumsum(x), (key % n).astype(np.int32)


@pytest.mark.parametrize("hub", [9000, 65536, 70000, 79999])
def test_rounds_equal_oracle(hub):
    n = 80001
    spokes = [(11, hub), (40000, 20000), (777, 10001), (60000, 9999), (123, 600), (4567, 300), (70001, 90)]
    xadj, adj = _mesh_with_spokes(n, 16.0, spokes)
    rng = np.random.default_rng(3)
    vw = rng.integers(1, 4, n).astype(np.int64)
    u = np.repeat(np.arange(n, dtype=np.int64), np.diff(xadj))
    ew = (np.minimum(u, adj) * 7919 + np.maximum(u, adj) * 104729) % 5 + 1
    unit = tp.graph_from_csr(xadj, adj)
    forms = [(oracle.Graph(xadj, adj), unit), (oracle.Graph(xadj, adj), unit.compress()),
             (oracle.Graph(xadj, adj, vw, ew), tp.graph_from_csr(xadj, adj, vw, ew))]
    op = oracle.Params(seed=6, cluster_rounds=12, refine_rounds=12)
    gp = tp.default_params(seed=6, cluster_rounds=12, refine_rounds=12, use_graphs=0)
    k = 5
    hubs = [h for h, _ in spokes]
    for og, g in forms:
        W = int(og.vw.sum())
        want = oracle.cluster(og, 400, op, 0)
        assert np.array_equal(tp.lp_cluster(g, 400, gp, 0).cpu().numpy(), want)
        # stripes, some vertices and all hubs displaced: the hubs move back
        part = (np.arange(n) * k // n).astype(np.int32)
        part[rng.integers(0, n, n // 300)] = 1
        for h in hubs:
            part[h] = (part[h] + 2) % k
        B = oracle.block_weights(og, part, k)
        l_max = max(int(B.max()), 1030 * -(-W // k) // 1000)
        want = part.copy()
        oracle.refine(og, want, B, k, l_max, op, 1)
        assert any(want[h] != part[h] for h in hubs)
        got = torch.from_numpy(part).cuda()
        tp.lp_refine(g, k, l_max, got, gp, level=1)
        assert np.array_equal(got.cpu().numpy(), want)


def test_hubs_cost_little():
    n, k = 1 << 20, 64
    mesh = tp.graph_from_csr(*synth.rgg2d(n, 16.0, 4))
    hubs = tp.graph_from_csr(*_mesh_with_spokes(n, 16.0, [(11, n - 1), (n // 2, n // 8), (n // 3, 9000)]))
    part = (torch.arange(n, device="cuda") * k // n).to(torch.int32)

    def ms(f):
        f()
        best = []
        for _ in range(3):
            torch.cuda.synchronize()
            b, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            b.record()
            f()
            e.record()
            torch.cuda.synchronize()
            best.append(b.elapsed_time(e))
        return min(best)

    p = tp.default_params(seed=1, cluster_rounds=8)
    for g in (hubs, hubs.compress()):
        m = mesh if g is hubs else mesh.compress()
        for f in (lambda q: tp.lp_cluster(q, 8192, p), lambda q: tp.lp_refine(q, k, n // k * 2, part.clone(), p)):
            assert ms(lambda: f(g)) < 2.5 * ms(lambda: f(m))

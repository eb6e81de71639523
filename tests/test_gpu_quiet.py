"""Rounds that leave quiet vertices out (lane tier, few movers) against the
oracle: refinement of nearly settled partitions and many clustering rounds,
unit weights, weighted and compressed, with vertices of higher tiers among the
movers, and the rounds and sub-rounds at which marks are not used."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _mesh_with_spokes(n, spokes):
    """A mesh and a few vertices joined to many others across it."""
    xadj, adj = synth.rgg2d(n, 12.0, 4)
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


GRAPHS = {
    "mesh": lambda: synth.rgg2d(30011, 16.0, 2),
    "spokes": lambda: _mesh_with_spokes(20000, ((3, 50), (777, 600), (5000, 10500))),
    "sparse": lambda: synth.gnm(9001, 12000, 5),
}


@pytest.mark.parametrize("name", GRAPHS)
@pytest.mark.parametrize("rounds,S", [(1, 8), (3, 8), (12, 8), (40, 8), (6, 32), (4, 33), (5, 1)])
def test_rounds_equal_oracle(name, rounds, S):
    xadj, adj = GRAPHS[name]()
    n = len(xadj) - 1
    rng = np.random.default_rng(11)
    vw = rng.integers(1, 4, n).astype(np.int64)
    u = np.repeat(np.arange(n, dtype=np.uint64), np.diff(xadj))
    lo, hi = np.minimum(u, adj.astype(np.uint64)), np.maximum(u, adj.astype(np.uint64))
    ew = ((lo * np.uint64(7919) + hi * np.uint64(104729)) % np.uint64(5) + np.uint64(1)).astype(np.int64)
    unit = tp.graph_from_csr(xadj, adj)
    forms = [(oracle.Graph(xadj, adj), unit), (oracle.Graph(xadj, adj), unit.compress()),
             (oracle.Graph(xadj, adj, vw, ew), tp.graph_from_csr(xadj, adj, vw, ew))]
    op = oracle.Params(seed=6, sub_rounds=S, cluster_rounds=rounds, refine_rounds=rounds)
    # rounds launched step by step, as on levels beyond the one-launch kernel
    gp = tp.default_params(seed=6, sub_rounds=S, cluster_rounds=rounds, refine_rounds=rounds, use_graphs=0)
    k = 5
    for og, g in forms:
        W = int(og.vw.sum())
        want = oracle.cluster(og, 40, op, 0)
        got = tp.lp_cluster(g, 40, gp, 0)
        assert np.array_equal(got.cpu().numpy(), want)
        # stripes with some vertices displaced: most of a block is settled
        part = (np.arange(n) * k // n).astype(np.int32)
        part[rng.integers(0, n, n // 200)] = 1
        B = oracle.block_weights(og, part, k)
        l_max = max(int(B.max()), 1030 * -(-W // k) // 1000)
        want = part.copy()
        oracle.refine(og, want, B, k, l_max, op, 1)
        got = torch.from_numpy(part).cuda()
        tp.lp_refine(g, k, l_max, got, gp, level=1)
        assert np.array_equal(got.cpu().numpy(), want)

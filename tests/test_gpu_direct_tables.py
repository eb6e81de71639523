"""Refinement and rebalancing with direct label tables (few blocks) and with
hash tables (many), in every degree tier, with ratings in 32 and 64 bits,
against the oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _all_tiers():
    """Skewed graph with vertices of every tier up to hubs above degree 10 000."""
    xadj, adj = synth.rmat(14, 16, seed=4)
    n = len(xadj) - 1
    u = np.repeat(np.arange(n), np.diff(xadj))
    extra = []
    for hub, d in ((5, 11000), (9, 6000), (17, 3000), (33, 1500), (65, 700), (129, 300)):
        v = np.arange(n - d, n)
        extra += [np.stack([np.full(d, hub), v], 1), np.stack([v, np.full(d, hub)], 1)]
    e = np.concatenate([np.stack([u, adj], 1)] + extra)
    key = np.unique(e[:, 0].astype(np.int64) * n + e[:, 1])
    key = key[key // n != key % n]
    x = np.zeros(n + 1, np.int64)
    np.add.at(x, key // n + 1, 1)
    return np.cumsum(x), (key % n).astype(np.int32)


@pytest.fixture(scope="module")
def csr():
    return _all_tiers()


def _weights(xadj, adj, top):
    n = len(xadj) - 1
    u = np.repeat(np.arange(n, dtype=np.uint64), np.diff(xadj))
    lo, hi = np.minimum(u, adj.astype(np.uint64)), np.maximum(u, adj.astype(np.uint64))
    h = (lo * np.uint64(0x9E3779B97F4A7C15) ^ hi * np.uint64(0xC2B2AE3D27D4EB4F)) >> np.uint64(13)
    return (h % np.uint64(top) + np.uint64(1)).astype(np.int64)


@pytest.mark.parametrize("k", [2, 128, 129, 1024, 1025])
# unit weights; 32-bit sums; the first weights whose sum does not fit them; wide ones
@pytest.mark.parametrize("top", [0, 900, 1 << 13, 1 << 40])
def test_refine_and_rebalance_equal_oracle(csr, k, top):
    xadj, adj = csr
    n = len(xadj) - 1
    ew = _weights(xadj, adj, top) if top else None
    og = oracle.Graph(xadj, adj, None, ew)
    g = tp.graph_from_csr(xadj, adj, None, ew)
    graphs = [g] if top else [g, g.compress()]
    l_max = oracle.block_cap(n, k, 30000)
    part = ((np.arange(n) * 7919 % n) * k // n).astype(np.int32)
    part[n // 2 : n // 2 + 10] = k - 1
    want = part.copy()
    B = oracle.block_weights(og, want, k)
    oracle.refine(og, want, B, k, l_max, oracle.Params(seed=4), 2)
    # a few vertices too many in block 0, so that rebalancing makes some moves
    unb = want.copy()
    Bu = oracle.block_weights(og, unb, k)
    move = np.flatnonzero(unb != 0)[: max(0, l_max - Bu[0]) + 5]
    unb[move] = 0
    reb = unb.copy()
    oracle.rebalance(og, reb, oracle.block_weights(og, unb, k), k, l_max)
    for gr in graphs:
        got = torch.from_numpy(part).cuda()
        tp.lp_refine(gr, k, l_max, got, tp.default_params(seed=4), level=2)
        assert np.array_equal(got.cpu().numpy(), want)
        got = torch.from_numpy(unb).cuda()
        tp.rebalance(gr, k, l_max, got)
        assert np.array_equal(got.cpu().numpy(), reb)

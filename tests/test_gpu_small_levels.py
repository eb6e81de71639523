"""The rounds of a small level in one launch (clusters of 1 to 16 CTAs) against
the oracle: unit weights, weighted and compressed; lane and warp tiers; 1, 8
and 32 sub-rounds; label caps that contest hardly any or most targets (warps
and blocks pick the prefix); and sizes just beyond the kernel's range."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _weights(xadj, adj, top):
    n = len(xadj) - 1
    u = np.repeat(np.arange(n, dtype=np.uint64), np.diff(xadj))
    lo, hi = np.minimum(u, adj.astype(np.uint64)), np.maximum(u, adj.astype(np.uint64))
    h = (lo * np.uint64(0x9E3779B97F4A7C15) ^ hi * np.uint64(0xC2B2AE3D27D4EB4F)) >> np.uint64(13)
    return (h % np.uint64(top) + np.uint64(1)).astype(np.int64)


GRAPHS = {
    "one": lambda: synth.gnm(1, 0, 1),
    "tiny": lambda: synth.gnm(40, 60, 1),
    "mesh_300": lambda: synth.rgg2d(300, 12.0, 1),
    "mesh_20k": lambda: synth.rgg2d(20011, 16.0, 2),
    "mesh_130k": lambda: synth.rgg2d(130003, 8.0, 3),
    "deg_100": lambda: synth.gnm(1501, 75000, 4),    # warp tiers
    "deg_500": lambda: synth.gnm(901, 190000, 5),    # around the largest degree (512)
    "entries": lambda: synth.gnm(4001, 1050000, 6),  # just beyond the entry limit
}


@pytest.mark.parametrize("name", GRAPHS)
@pytest.mark.parametrize("S", [1, 8, 32])
def test_rounds_equal_oracle(name, S):
    xadj, adj = GRAPHS[name]()
    n = len(xadj) - 1
    rng = np.random.default_rng(7)
    vw = rng.integers(1, 6, n).astype(np.int64)
    ew = _weights(xadj, adj, 30)
    unit = tp.graph_from_csr(xadj, adj)
    forms = [(oracle.Graph(xadj, adj), unit), (oracle.Graph(xadj, adj), unit.compress()),
             (oracle.Graph(xadj, adj, vw, ew), tp.graph_from_csr(xadj, adj, vw, ew))]
    op = oracle.Params(seed=3, sub_rounds=S)
    gp = tp.default_params(seed=3, sub_rounds=S)
    for og, g in forms:
        W = int(og.vw.sum())
        for cap in (7, max(8, W // 20)):
            want = oracle.cluster(og, cap, op, 1)
            got = tp.lp_cluster(g, cap, gp, 1)
            assert np.array_equal(got.cpu().numpy(), want), cap
        for k, slack in ((2, 1001), (37, 1030)):
            part = ((np.arange(n) * 7919 % n) * k // n).astype(np.int32)
            B = oracle.block_weights(og, part, k)
            l_max = max(int(B.max()), slack * -(-W // k) // 1000)
            want = part.copy()
            oracle.refine(og, want, B, k, l_max, op, 2)
            got = torch.from_numpy(part).cuda()
            tp.lp_refine(g, k, l_max, got, gp, level=2)
            assert np.array_equal(got.cpu().numpy(), want), k

"""The bisection kernel's forms against the oracle: state in shared memory or
clusters with state in global memory (a node too large for shared memory, or
with too many edges for one SM), 32- and 64-bit connectivity differences,
adjacency groups of 4 to 32 lanes, and contested sides."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _weights(n, m2, xadj, adj, top, seed):
    """Vertex weights and symmetric edge weights up to top."""
    rng = np.random.default_rng(seed)
    vw = rng.integers(1, 9, n)
    u = np.repeat(np.arange(n, dtype=np.uint64), np.diff(xadj))
    lo, hi = np.minimum(u, adj.astype(np.uint64)), np.maximum(u, adj.astype(np.uint64))
    h = (lo * np.uint64(0x9E3779B97F4A7C15) ^ hi * np.uint64(0xC2B2AE3D27D4EB4F)) >> np.uint64(13)
    return vw.astype(np.int64), (h % np.uint64(top) + np.uint64(1)).astype(np.int64)


CASES = {
    # above the shared-memory capacity (about 12 500 vertices): clusters of 16
    "large_mesh": (lambda: synth.rgg2d(20001, 5.0, 3), 1, 5),
    # few vertices, more than 2^19 entries: clusters although the state would fit
    "dense": (lambda: synth.gnm(1501, 300000, 4), 7, 3),
    # weighted degrees beyond 32 bits, in both forms
    "wide_smem": (lambda: synth.gnm(2500, 20000, 5), 1 << 40, 6),
    "wide_cluster": (lambda: synth.gnm(14003, 60000, 6), 1 << 40, 4),
    # isolated vertices and several components, the smallest groups
    "sparse": (lambda: synth.gnm(3001, 2000, 7), 5, 9),
    "hubs": (lambda: synth.rmat(13, 16, seed=8), 1, 16),
    "tiny": (lambda: synth.gnm(9, 12, 9), 3, 4),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("slack", [1000, 1030])  # side caps that contest movers, or hardly do
def test_bisection_equals_oracle(name, slack):
    make, top, k = CASES[name]
    xadj, adj = make()
    n = len(xadj) - 1
    vw, ew = _weights(n, len(adj), xadj, adj, top, 1)
    l_max = slack * -(-int(vw.sum()) // k) // 1000
    want = oracle.initial_partition(oracle.Graph(xadj, adj, vw, ew), k, l_max, oracle.Params(seed=5))
    g = tp.graph_from_csr(xadj, adj, vw, ew)
    got = tp.initial_partition(g, k, l_max, tp.default_params(seed=5))
    assert np.array_equal(got.cpu().numpy(), want)

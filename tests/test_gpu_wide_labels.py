"""Refinement of weighted graphs over more blocks than the lane tier's 32-bit
sort keys can tell apart (label and slot: 2^27 - 1 labels), against the oracle:
the rounds of a small level in one launch are not for it, and the kernels that
are sort 64-bit keys; and one block count that the short keys just hold."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402

LIMIT = (1 << 27) - 1


@pytest.mark.parametrize("k", [LIMIT, LIMIT + 1, LIMIT + 40])
@pytest.mark.parametrize("use_graphs", [0, 1])
def test_refinement_equals_oracle(k, use_graphs):
    xadj, adj = synth.rgg2d(4001, 14.0, 3)  # most vertices in the lane tier
    n = len(xadj) - 1
    u = np.repeat(np.arange(n, dtype=np.int64), np.diff(xadj))
    ew = (np.minimum(u, adj) * 7919 + np.maximum(u, adj) * 104729) % 9 + 1
    vw = np.arange(n, dtype=np.int64) % 3 + 1
    # the last labels, and the first, which some of them are without their top bit
    labels = np.concatenate([k - 1 - np.arange(20, dtype=np.int64), np.arange(40)])
    assert 0 <= labels.min() and labels.max() < k
    part = labels[np.random.default_rng(2).integers(0, len(labels), n)].astype(np.int32)
    og = oracle.Graph(xadj, adj, vw, ew)
    B = np.bincount(part, weights=vw, minlength=k).astype(np.int64)
    l_max = int(B.max()) + 40
    want = part.copy()
    oracle.refine(og, want, B, k, l_max, oracle.Params(seed=6), 1)
    got = torch.from_numpy(part).cuda()
    g = tp.graph_from_csr(xadj, adj, vw, ew)
    tp.lp_refine(g, k, l_max, got, tp.default_params(seed=6, use_graphs=use_graphs), level=1)
    assert np.array_equal(got.cpu().numpy(), want)

"""Levels on both sides of the line between the one-launch kernel of small
levels and the kernels of the sub-rounds, against the oracle; and beyond the
line, where the one launch would take up to twice as long, it is not taken."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402

SIDES = {
    "sparse": ((90001, 8), (140001, 8)),
    "warp tiers": ((4001, 60), (20001, 60)),
    "mixed": ((15001, 30), (40001, 30)),
}


@pytest.mark.parametrize("name", SIDES)
def test_both_sides_equal_oracle(name):
    for n, deg in SIDES[name]:
        xadj, adj = synth.gnm(n, n * deg // 2, n)
        og, g = oracle.Graph(xadj, adj), tp.graph_from_csr(xadj, adj)
        op, gp = oracle.Params(seed=4), tp.default_params(seed=4)
        for q in (g, g.compress()):
            assert np.array_equal(tp.lp_cluster(q, n // 200, gp, 1).cpu().numpy(),
                                  oracle.cluster(og, n // 200, op, 1))


@pytest.mark.parametrize("n,deg", [(20001, 100), (60001, 34)])
def test_beyond_the_line_costs_no_more_than_the_kernels_of_the_sub_rounds(n, deg):
    g = tp.graph_from_csr(*synth.gnm(n, n * deg // 2, n))

    def ms(use_graphs):
        p = tp.default_params(seed=4, use_graphs=use_graphs)
        tp.lp_cluster(g, n // 200, p)
        best = []
        for _ in range(5):
            torch.cuda.synchronize()
            b, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            b.record()
            tp.lp_cluster(g, n // 200, p)
            e.record()
            torch.cuda.synchronize()
            best.append(b.elapsed_time(e))
        return min(best)

    assert ms(1) < 1.2 * ms(0)

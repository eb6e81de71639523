"""Contraction of unit-weight graphs of 2^31 adjacency entries, compressed and
CSR: a ring of n vertices, each joined to the eight before and the eight behind
it, in clusters of 64 consecutive vertices. The coarse graph is a ring of
n / 64 vertices whose edges weigh 1 + 2 + ... + 8 = 36 (the pairs of distance
at most eight across a cluster's end). Everything stays on the device."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402

REACH, CLUSTER = 8, 64


def _ring(n):
    """CSR of the ring; rows ascending (the first and last rows wrap around)."""
    deg = 2 * REACH
    xadj = torch.arange(n + 1, dtype=torch.int64, device="cuda") * deg
    adj = torch.empty(n * deg, dtype=torch.int32, device="cuda")
    step = torch.tensor([d for d in range(-REACH, REACH + 1) if d], device="cuda")
    rows = 1 << 24
    for lo in range(0, n, rows):
        u = torch.arange(lo, min(lo + rows, n), device="cuda")
        v = (u[:, None] + step) % n
        if lo == 0 or lo + rows >= n:
            v = v.sort(1).values
        adj[lo * deg : lo * deg + v.numel()] = v.reshape(-1).to(torch.int32)
    return xadj, adj


def test_weights_of_2_31_entries():
    n = 1 << 27
    nc = n // CLUSTER
    g = tp.graph_from_csr(*_ring(n))
    assert g.info()["m2"] == 1 << 31
    C = torch.arange(n, dtype=torch.int32, device="cuda") // CLUSTER * CLUSTER
    a = torch.arange(nc, device="cuda")
    want = torch.stack([(a - 1) % nc, (a + 1) % nc], 1).sort(1).values.reshape(-1).to(torch.int32)
    z = g.compress()
    for q in (z, g):
        cg, cmap = tp.contract(q, C)
        x, adj, vw, ew = cg.export_csr()
        assert torch.equal(x, torch.arange(nc + 1, device="cuda") * 2)
        assert torch.equal(adj, want)
        assert bool((vw == CLUSTER).all()) and bool((ew == REACH * (REACH + 1) // 2).all())
        assert torch.equal(cmap, C // CLUSTER)
        del cg, cmap, x, adj, vw, ew

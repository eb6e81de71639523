"""Long runs of rows without entries: a tile of entries behind such a run has
more rows than its block walks one by one (65 536). Validation, encoding and
decoding against the oracle, runs in front, inside, at tile ends and behind;
malformed graphs behind a run are still refused; and a run costs no more than
as many rows with entries."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2410_19119_gb300 as tp  # noqa: E402


def _spread(xadj, adj, gaps):
    """The graph with gaps[i] empty rows put in front of row i (i = n: at the end)."""
    n = len(xadj) - 1
    pad = np.zeros(n + 1, np.int64)
    for i, c in gaps.items():
        pad[i] += c
    at = np.arange(n) + np.cumsum(pad)[:n]
    total = n + int(pad.sum())
    deg = np.zeros(total, np.int64)
    deg[at] = np.diff(xadj)
    x = np.zeros(total + 1, np.int64)
    np.cumsum(deg, out=x[1:])
    return x, at[adj].astype(np.int32)


MANY = 65536
CASES = {
    "front": {0: 3 * MANY},
    "behind": {5000: 2 * MANY + 7},
    "inside": {1700: MANY - 1, 2500: MANY, 2501: MANY + 1, 4000: 5, 4100: 31, 4200: 32, 4300: 33},
    "all": {0: MANY + 5, 1: 1, 2222: 4 * MANY, 4999: 100000, 5000: MANY},
    "short": {100: 1, 200: 64, 300: 4095, 400: 9000},
}
GRAPHS = {
    "mesh": lambda: synth.rgg2d(5000, 9.0, 3),
    "sparse": lambda: synth.gnm(5000, 3100, 4),  # empty rows of its own, few tiles
    "hub": lambda: synth.rmat(13, 16, seed=2),
}


@pytest.mark.parametrize("graph", GRAPHS)
@pytest.mark.parametrize("case", CASES)
def test_streams_equal_oracle(graph, case):
    xadj, adj = _spread(*GRAPHS[graph](), CASES[case])
    n = len(xadj) - 1
    g = tp.graph_from_csr(xadj, adj)
    z = g.compress()
    data, off = z.export_compressed()
    want, woff = oracle.encode(xadj, adj)
    assert np.array_equal(data.cpu().numpy(), want) and np.array_equal(off.cpu().numpy(), woff)
    for q in (z.decompress(), tp.graph_from_compressed(n, data, off).decompress()):
        x, a, _, _ = q.export_csr()
        assert np.array_equal(x.cpu().numpy(), xadj) and np.array_equal(a.cpu().numpy(), adj)


def test_last_entry_in_the_first_of_two_tiles_and_only_empty_rows_behind():
    """2048 entries exactly: the last tile holds no entry, only rows."""
    n = 1025
    xadj = np.concatenate([[0], 1 + np.arange(0, 2 * (n - 2) + 1, 2), [2 * (n - 1)]])
    u = np.arange(n)
    adj = np.stack([u - 1, u + 1], 1).reshape(-1)[1:-1].astype(np.int32)
    assert len(adj) == 2048 == xadj[-1]
    for gaps in ({n: 2 * MANY}, {0: 2 * MANY, n: MANY}):
        x, a = _spread(xadj, adj, gaps)
        data, off = tp.graph_from_csr(x, a).compress().export_compressed()
        want, woff = oracle.encode(x, a)
        assert np.array_equal(data.cpu().numpy(), want) and np.array_equal(off.cpu().numpy(), woff)


def test_faults_behind_a_run_are_refused():
    xadj, adj = _spread(*synth.rgg2d(5000, 9.0, 3), {2500: 3 * MANY})
    b = int(xadj[2600 + 3 * MANY])  # a row behind the run
    assert xadj[2601 + 3 * MANY] - b >= 2
    for change in ("order", "loop", "mirror", "range"):
        a = adj.copy()
        if change == "order":
            a[b], a[b + 1] = a[b + 1], a[b]
        elif change == "loop":
            a[b] = 2600 + 3 * MANY
        elif change == "mirror":
            a[b] -= 1
        else:
            a[b] = len(xadj) - 1
        with pytest.raises(tp.TpError):
            tp.graph_from_csr(xadj, a)
    tp.graph_from_csr(xadj, adj)


def test_a_run_costs_no_more_than_rows_with_entries():
    n, edge = 1 << 24, 1000
    pairs = torch.arange(n - 1, device="cuda")

    def csr(u):
        key = torch.cat([u * n + u + 1, (u + 1) * n + u]).sort().values
        x = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        x[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
        return x, (key % n).to(torch.int32)

    def ms(f):
        f()
        best = []
        for _ in range(3):
            torch.cuda.synchronize()
            b, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            b.record()
            r = f()
            e.record()
            torch.cuda.synchronize()
            best.append(b.elapsed_time(e))
            del r
        return min(best)

    path = csr(pairs)
    run = csr(torch.cat([pairs[:edge], pairs[-edge:]]))
    assert ms(lambda: tp.graph_from_csr(*run)) < 2 * ms(lambda: tp.graph_from_csr(*path))
    gp, gr = tp.graph_from_csr(*path), tp.graph_from_csr(*run)
    assert ms(gr.compress) < 2 * ms(gp.compress)

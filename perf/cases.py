"""The calls that users of the partitioner make, as timed cases.

A case is one call chain through the public entry points of
paper_2410_19119_gb300 on one kind of graph:

  partition  the whole multilevel partitioner on a graph that is in device memory
  batch      many small independent graphs partitioned in one call
  encode     CSR arrays to a validated graph handle, compressed, exported
  decode     a compressed stream to a validated handle, decompressed, exported
  cluster    size-constrained label propagation of one coarsening level
  contract   one contraction, the coarse graph exported
  refine     k-way refinement of a projected partition, then its cut and block weights
  initial    recursive bisection of a coarsest graph

Graphs: "rgg" (2D random geometric, ids in row-major cell order: meshes, road
networks), "rmat" (skewed degrees up to hubs: social and web graphs), "gnm"
(uniform random, no locality). They are made on the GPU from the seed alone.
All results are whole numbers, so there is nothing to compare in 64 bits.
"""
import math

import torch

import paper_2410_19119_gb300 as tp

EPS = 0.03


def listed():
    return [
        # the smallest call in earnest (and the size of the framework's own
        # smoke run): one small graph; launches, synchronisations and the
        # serial parts of a phase are all there is
        {"name": "partition_gnm_4k", "op": "partition", "graph": "gnm", "n": 4096, "deg": 16.0,
         "k": 8, "zip": False},
        # an ordinary mesh of a million vertices (an odd number of them) as plain CSR
        {"name": "partition_rgg_1m", "op": "partition", "graph": "rgg", "n": 1000003, "deg": 16.0,
         "k": 16, "zip": False},
        # the headline: the large mesh in the compressed format (the benchmark's size)
        {"name": "partition_rgg_16m_zip", "op": "partition", "graph": "rgg", "n": 1 << 24,
         "deg": 16.0, "k": 64, "zip": True},
        # a social network in the compressed format: hubs, chunked records, dense coarse levels
        {"name": "partition_rmat_4m_zip", "op": "partition", "graph": "rmat", "n": 1 << 22,
         "deg": 32.0, "k": 256, "zip": True},
        # a service's queue of small graphs, partitioned together
        {"name": "batch_160", "op": "batch", "graph": "mixed", "n": 1 << 16, "count": 160,
         "deg": 12.0, "k": 32, "zip": False},
        # loading a mesh: arrays to a validated, compressed graph
        {"name": "encode_rgg_4m", "op": "encode", "graph": "rgg", "n": 4194301, "deg": 16.0,
         "k": 0, "zip": False},
        # loading a skewed graph: hubs in the validation and in the chunked encoder
        {"name": "encode_rmat_1m", "op": "encode", "graph": "rmat", "n": 1 << 20, "deg": 32.0,
         "k": 0, "zip": False},
        # reading a stored compressed graph back to CSR
        {"name": "decode_rgg_3m", "op": "decode", "graph": "rgg", "n": 3000001, "deg": 16.0,
         "k": 0, "zip": True},
        # coarsening alone on a skewed compressed graph (the clustering kernel of the library's
        # paper, all degree tiers); users with their own contraction call this
        {"name": "cluster_rmat_2m_zip", "op": "cluster", "graph": "rmat", "n": 2000003,
         "deg": 32.0, "k": 64, "zip": True},
        # one contraction of a large compressed mesh
        {"name": "contract_rgg_4m_zip", "op": "contract", "graph": "rgg", "n": 4194301,
         "deg": 16.0, "k": 64, "zip": True},
        # uncoarsening step on a weighted, dense coarse level of a skewed graph
        {"name": "refine_rmat_coarse", "op": "refine", "graph": "rmat", "n": 1 << 20,
         "deg": 32.0, "k": 64, "zip": False},
        # the coarsest weighted graph of a mesh, recursively bisected
        {"name": "initial_rgg_coarse", "op": "initial", "graph": "rgg", "n": 1 << 20,
         "deg": 16.0, "k": 64, "zip": False},
    ]


def draw(rng):
    op = rng.choice(["partition", "partition", "partition", "batch", "encode", "decode", "cluster",
                     "contract", "refine", "initial"])
    if op == "batch":
        return {"op": op, "graph": "mixed", "n": int(2 ** rng.uniform(12, 16)),
                "count": rng.randint(3, 160), "deg": rng.uniform(6.0, 16.0),
                "k": rng.choice([4, 8, 16, 32]), "zip": False}
    graph = rng.choice(["rgg", "rgg", "rmat", "gnm"])
    # levels below the input (refine, initial) start from an input large enough to be coarsened
    lo = 15 if op in ("refine", "initial") else 10
    hi = {"rgg": 23, "rmat": 20, "gnm": 20}[graph]
    n = int(2 ** rng.uniform(lo, hi))
    deg = {"rgg": rng.uniform(8.0, 24.0), "rmat": rng.uniform(16.0, 40.0),
           "gnm": rng.uniform(6.0, 20.0)}[graph]
    k = rng.choice([2, 3, 8, 13, 16, 32, 64, 100, 256])
    while k > 2 and n < 160 * k:  # (a graph this small would not be coarsened at all)
        k //= 2
    zipped = op == "decode" or (op in ("partition", "cluster", "contract") and rng.random() < 0.5)
    return {"op": op, "graph": graph, "n": n, "deg": deg, "k": k, "zip": zipped}


# ---------------------------------------------------------------- inputs

def _csr(n, u, v):
    """CSR of directed entries (u, v) that are sorted by (u, v)."""
    xadj = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    xadj[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    return xadj, v.to(torch.int32)


def _symmetric(n, u, v):
    """Symmetric CSR without loops or duplicates of the pairs (u, v)."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    return _csr(n, key // n, key % n)


def _gnm(n, deg, gen):
    m = int(n * deg / 2)
    u = torch.randint(0, n, (m,), generator=gen, device="cuda")
    v = torch.randint(0, n, (m,), generator=gen, device="cuda")
    return _symmetric(n, u, v)


def _rmat(n, deg, gen, probs=(0.57, 0.19, 0.19)):
    """R-MAT pairs of the next power of two, those among the first n vertices kept."""
    scale = max(1, (n - 1).bit_length())
    a, b, c = probs
    m = int(n * deg / 2)
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        r = torch.rand(m, generator=gen, device="cuda")
        u = 2 * u + (r >= a + b)
        v = 2 * v + (((r >= a) & (r < a + b)) | (r >= a + b + c))
    keep = (u < n) & (v < n)
    return _symmetric(n, u[keep], v[keep])


def _rgg(n, deg, gen):
    """Points in the unit square, joined within the radius of average degree deg; ids by grid
    cell in row-major order, then x."""
    r = math.sqrt(deg / (math.pi * n))
    dim = max(1, int(1.0 / r))
    p = torch.rand(2, n, generator=gen, device="cuda", dtype=torch.float64)
    cx = (p[0] * dim).long().clamp_(max=dim - 1)
    cy = (p[1] * dim).long().clamp_(max=dim - 1)
    order = torch.argsort((cy * dim + cx) + (p[0] * dim - cx).clamp_(0, 0.999999))
    x, y, cx, cy = p[0][order], p[1][order], cx[order], cy[order]
    start = torch.zeros(dim * dim + 1, dtype=torch.int64, device="cuda")
    start[1:] = torch.cumsum(torch.bincount(cy * dim + cx, minlength=dim * dim), 0)
    us, vs = [], []
    step = 1 << 21
    for lo in range(0, n, step):  # bounds the candidate lists
        ids = torch.arange(lo, min(lo + step, n), device="cuda")
        ax, ay = cx[ids], cy[ids]
        first, count = [], []
        for dy in (-1, 0, 1):  # three runs of candidates per vertex: ids stay ascending
            row = ay + dy
            ok = (row >= 0) & (row < dim)
            base = row.clamp(0, dim - 1) * dim
            b = start[base + (ax - 1).clamp(min=0)]
            e = start[base + (ax + 1).clamp(max=dim - 1) + 1]
            first.append(b)
            count.append(torch.where(ok, e - b, torch.zeros_like(b)))
        first, count = torch.stack(first, 1).reshape(-1), torch.stack(count, 1).reshape(-1)
        end = torch.cumsum(count, 0)
        run = torch.repeat_interleave(torch.arange(len(count), device="cuda"), count)
        v = torch.arange(len(run), device="cuda") - (end - count)[run] + first[run]
        u = lo + run // 3
        dx, dy = x[u] - x[v], y[u] - y[v]
        keep = (dx * dx + dy * dy <= r * r) & (u != v)
        us.append(u[keep])
        vs.append(v[keep].to(torch.int32))
    return _csr(n, torch.cat(us), torch.cat(vs))


def _arrays(kind, n, deg, gen):
    return {"gnm": _gnm, "rmat": _rmat, "rgg": _rgg}[kind](n, deg, gen)


def _cluster_cap(weight, k):
    return max(1, int(EPS * 1e6) * weight // (1000000 * k))


def _block_cap(weight, k):
    return (1000000 + int(EPS * 1e6)) * -(-weight // k) // 1000000


def _coarser(g, cap, level=0):
    return tp.contract(g, tp.lp_cluster(g, cap, level=level))


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    op, n, k = case["op"], case["n"], case["k"]
    if op == "batch":
        graphs, ks = [], []
        for i in range(case["count"]):  # sizes spread evenly over the logarithm of 2^8 .. n
            ni = int(2 ** (8 + (math.log2(n) - 8) * (i * 0.6180339887 % 1)))
            xadj, adj = _arrays(("gnm", "rgg", "rmat")[i % 3], ni, case["deg"], gen)
            graphs.append(tp.graph_from_csr(xadj, adj))
            ks.append(2 << int(math.log2(k) * (i * 0.4142135624 % 1)))
        out = torch.empty(sum(g.n for g in graphs), dtype=torch.int32, device="cuda")
        outs = list(torch.split(out, [g.n for g in graphs]))
        return {"op": op, "graphs": graphs, "ks": ks, "out": out, "outs": outs}
    xadj, adj = _arrays(case["graph"], n, case["deg"], gen)
    # the caller's buffers for results whose length is known after the call only (zero beyond it)
    most = int(1.05 * n * case["deg"]) + 4096

    def buffers(**sizes):
        return {name: torch.zeros(size, dtype=dtype, device="cuda")
                for name, (size, dtype) in sizes.items()}

    if op == "encode":
        return {"op": op, "xadj": xadj, "adj": adj,
                "out": buffers(bytes=(6 * n + 4 * most, torch.uint8),
                               offsets=(n + 1, torch.int64))}
    g = tp.graph_from_csr(xadj, adj)
    if case["zip"]:
        g = g.compress()
    if op == "decode":
        data, off = g.export_compressed()
        return {"op": op, "n": n, "data": data, "off": off,
                "out": buffers(xadj=(n + 1, torch.int64), adj=(most, torch.int32))}
    state = {"op": op, "g": g, "k": k}
    if op == "cluster":
        state["cap"] = _cluster_cap(n, k)
    elif op == "contract":
        state["cluster"] = tp.lp_cluster(g, _cluster_cap(n, k))
        state["out"] = buffers(xadj=(n + 1, torch.int64), adj=(most, torch.int32),
                               vw=(n, torch.int64), ew=(most, torch.int64),
                               map=(n, torch.int32))
    elif op == "refine":  # the first coarse level, its partition projected from the next one
        cap = _cluster_cap(n, k)
        g1, _ = _coarser(g, cap)
        g2, m2 = _coarser(g1, cap, 1)
        part, _ = tp.partition(g2, k, EPS)
        state.update(g=g1, part=part[m2.long()].contiguous(), cap=_block_cap(n, k),
                     out=buffers(part=(n, torch.int32)))
    elif op == "initial":  # coarsened as the partitioner does, to about 160 k vertices
        cap, level = _cluster_cap(n, k), 0
        while g.n > 160 * k and level < 8:
            coarse, _ = _coarser(g, cap, level)
            if 20 * coarse.n > 19 * g.n:
                break
            g, level = coarse, level + 1
        state.update(g=g, cap=_block_cap(n, k), out=buffers(part=(n, torch.int32)))
    return state


# ---------------------------------------------------------------- one pass

def _into(out, **results):
    """Results of a length known only now, copied into the caller's buffers."""
    for name, t in results.items():
        out[name][: len(t)].copy_(t)
    return out


def run(state):
    op = state["op"]
    if op == "partition":
        part, stats = tp.partition(state["g"], state["k"], EPS)
        return {"part": part, "cut": stats["cut"], "heaviest": stats["max_block_weight"],
                "levels": stats["levels"]}
    if op == "batch":
        res = tp.partition_batch(state["graphs"], state["ks"], EPS, outs=state["outs"])
        return {"part": state["out"], "cut": torch.tensor([st["cut"] for _, st in res])}
    if op == "encode":
        z = tp.graph_from_csr(state["xadj"], state["adj"]).compress()
        data, off = z.export_compressed()
        return _into(state["out"], bytes=data, offsets=off)
    if op == "decode":
        g = tp.graph_from_compressed(state["n"], state["data"], state["off"]).decompress()
        xadj, adj, _, _ = g.export_csr()
        return _into(state["out"], xadj=xadj, adj=adj)
    if op == "cluster":
        return {"cluster": tp.lp_cluster(state["g"], state["cap"])}
    if op == "contract":
        coarse, cmap = tp.contract(state["g"], state["cluster"])
        xadj, adj, vw, ew = coarse.export_csr()
        return _into(state["out"], xadj=xadj, adj=adj, vw=vw, ew=ew, map=cmap)
    if op == "refine":
        part = tp.lp_refine(state["g"], state["k"], state["cap"], state["part"].clone())
        cut, weights = tp.metrics(state["g"], part, state["k"])
        return {**_into(state["out"], part=part), "cut": cut, "weights": weights}
    return _into(state["out"], part=tp.initial_partition(state["g"], state["k"], state["cap"]))


def work(case):
    """Bytes of the inputs and outputs of one pass (sizes as expected of the random graphs:
    a compressed entry takes about 1.8 bytes in meshes and 2.8 in graphs without locality)."""
    n, m2 = case["n"], case["n"] * case["deg"]
    if case["op"] == "batch":  # sizes are spread over the logarithm of 2^8 .. n
        mean = (n - 256) / math.log(n / 256)
        n, m2 = case["count"] * mean, case["count"] * mean * case["deg"]
    csr = 8 * n + 4 * m2
    packed = 4 * n + m2 * (1.8 if case["graph"] == "rgg" else 2.8)
    graph = packed if case["zip"] else csr
    # coarse levels: about an eighth of the vertices, half of the entries, 12 bytes an entry
    coarse = 16 * n / 8 + 12 * m2 / 2
    total = {
        "partition": graph + 4 * n,
        "batch": csr + 4 * n,
        "encode": csr + packed + 4 * n,
        "decode": packed + 4 * n + csr + 8 * m2 + 8 * n,
        "cluster": graph + 4 * n,
        "contract": graph + 4 * n + coarse + 4 * n,
        "refine": coarse + 8 * n / 8,
        "initial": 16 * 160 * case["k"] + 12 * 160 * case["k"] * 16,
    }[case["op"]]
    return {"bytes": total, "flops": 0}


def exact(case, seed):
    """Every output is a whole number: there is no value in 64 bits to compare with."""
    return None

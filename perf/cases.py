"""The work that users of the partitioner have it do, as cases for timing.

A case names a call of the Python binding (``op``), the graph it gets and its options. Graphs are the
families of ``graphgen`` (4-neighbour grids, random geometric graphs of average degree 12, R-MAT graphs
of edge factor 16 with and without edge weights 1..8), drawn on the GPU from the case's seed.
"""
import math

import numpy as np
import torch

import paper_1710_08231_gb300 as gp

EPS = 0.03  # the imbalance of every configuration
DEG = 12.0  # average degree of the random geometric graphs
EDGE_FACTOR = 16
SHAPE = 11  # seed of the graphs whose entries or clusters decide the size of a result
M31, M63 = 0x7FFFFFFF, 0x7FFFFFFFFFFFFFFF


def listed():
    return [
        # the smallest graph of a batch clustered alone: latency and launches decide
        dict(name="cluster_rgg_1000", op="cluster", graph="rgg", n=1000, weights="unit", k=2),
        # level 0 of coarsening a large power-law graph: hubs beside millions of short rows
        dict(name="cluster_rmat_21", op="cluster", graph="rmat", scale=21, weights="unit", k=64),
        # refinement of a projected partition on a coarse mesh level: 64-bit weights and offsets, odd sizes
        dict(name="refine_rgg_777777_i64", op="refine", graph="rgg", n=777777, weights="int64", k=13),
        # contraction of a mesh level and of a power-law level (short rows; rows of millions of entries)
        dict(name="contract_rgg_2e20", op="contract", graph="rgg", n=1 << 20, weights="unit", k=16),
        dict(name="contract_rmat_22w", op="contract", graph="rmat", scale=22, weights="int32", k=64),
        # the learned scorer: inference on every entry of a level, and one gradient of its training
        dict(name="score_rmat_19w", op="score", graph="rmat", scale=19, weights="int32"),
        dict(name="grad_1000003", op="grad", n=1000003),
        # whole partitions: the smallest configuration, the mesh one, the power-law one
        dict(name="partition_grid_256", op="partition", graph="grid", rows=256, cols=256, weights="unit", k=2),
        dict(name="partition_rgg_2e20", op="partition", graph="rgg", n=1 << 20, weights="unit", k=16),
        dict(name="partition_rmat_22w", op="partition", graph="rmat", scale=22, weights="int32", k=64),
        # the paper's configuration of local search after every level's refinement
        dict(name="partition_mls_rgg_2e18", op="partition", graph="rgg", n=1 << 18, weights="unit", k=16, mls=3),
        # many small instances in one call
        dict(name="batch_512", op="batch", count=512, n_lo=1000, n_hi=200000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["cluster", "cluster", "refine", "contract", "contract", "score", "grad", "partition", "partition",
                     "partition", "mls", "batch"])
    if op == "grad":
        return dict(op="grad", n=_log(rng, 10000, 1000003))
    if op == "batch":
        return dict(op="batch", count=_log(rng, 8, 256), n_lo=1000, n_hi=_log(rng, 20000, 200000))
    c = dict(op="partition" if op == "mls" else op)
    graph = "rgg" if op in ("refine", "mls") else rng.choice(["rgg", "rmat"] + (["grid"] if op != "score" else []))
    c["graph"] = graph
    if graph == "rgg":
        c["n"] = _log(rng, 1000, (1 << 18) if op in ("mls", "score") else (1 << 20))
    elif graph == "grid":
        c["rows"], c["cols"] = _log(rng, 30, 1100), _log(rng, 30, 900)
    else:
        c["scale"] = rng.randint(12, 19 if op == "score" else 21)
    c["weights"] = rng.choice(["unit", "int32"] if op in ("score", "mls") else ["unit", "int32", "int64"])
    if op != "score":
        c["k"] = rng.choice([2, 4, 8, 13, 16, 32, 64]) if op != "mls" else rng.choice([4, 16, 64])
    if op == "mls":
        c["mls"] = 3
    return c


# ------------------------------------------------------------------------------------------ graphs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed & M63)


def _csr(src, dst, n):
    """Offsets of the rows of entries sorted by (src, dst)."""
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.bincount(src, minlength=n).cumsum(0)
    return off, dst.to(torch.int32)


def _rename(v, n, by):
    """Another name for every vertex: the graph stays the same up to its ids, near ids stay near."""
    return v ^ (by & (n - 1)) if n & (n - 1) == 0 else (v + by) % n


def _renamed(n, src, dst, by):
    """Offsets and adjacency of the entries (src, dst) with renamed vertices."""
    e = torch.sort(_rename(src, n, by) * n + _rename(dst, n, by)).values
    return _csr(e // n, e % n, n)


def _grid(rows, cols):
    n = rows * cols
    v = torch.arange(n, device="cuda")
    r, c = v // cols, v % cols
    nb = torch.stack([v - cols, v - 1, v + 1, v + cols], 1)  # ascending neighbour ids
    ok = torch.stack([r > 0, c > 0, c < cols - 1, r < rows - 1], 1)
    src = v[:, None].expand(n, 4)[ok]
    return n, _csr(src, nb[ok], n), r.double() / rows


def _rgg(n, gen):
    """Points in the unit square, an edge below distance sqrt(DEG / (pi n)); ids in generation order."""
    p = torch.rand(n, 2, dtype=torch.float64, device="cuda", generator=gen)
    r = math.sqrt(DEG / (math.pi * n))
    side = max(1, int(1.0 / r))  # cells at least r wide
    cell = (p * side).long().clamp_(max=side - 1)
    key = cell[:, 1] * side + cell[:, 0]
    order = torch.argsort(key)
    start = torch.searchsorted(key[order], torch.arange(side * side + 1, device="cuda"))
    pairs = []
    for dy in (-1, 0, 1):
        y = cell[:, 1] + dy
        x0, x1 = (cell[:, 0] - 1).clamp_(min=0), (cell[:, 0] + 1).clamp_(max=side - 1)
        ok = (y >= 0) & (y < side)
        yc = y.clamp(0, side - 1)
        b = start[yc * side + x0]
        cnt = torch.where(ok, start[yc * side + x1 + 1] - b, 0)
        src = torch.repeat_interleave(cnt)
        first = torch.cumsum(cnt, 0) - cnt
        dst = order[b[src] + torch.arange(src.numel(), device="cuda") - first[src]]
        d = p[src] - p[dst]
        near = ((d * d).sum(1) < r * r) & (src != dst)
        pairs.append(src[near] * n + dst[near])
    e = torch.sort(torch.cat(pairs)).values
    return n, _csr(e // n, e % n, n), p[:, 0]


def _rmat(scale, gen):
    """R-MAT quadrants (.57, .19, .19, .05), symmetrised, without loops and duplicates."""
    n, m = 1 << scale, EDGE_FACTOR << scale
    key = torch.zeros(2, m, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        u = torch.rand(m, device="cuda", generator=gen)
        down = u >= 0.76
        right = ((u >= 0.57) & ~down) | (u >= 0.95)
        key.mul_(2)
        key[0] += down
        key[1] += right
    a, b = key[0], key[1]
    keep = a != b
    a, b = a[keep], b[keep]
    e = torch.unique(torch.cat([(a << scale) | b, (b << scale) | a]))
    return n, _csr(e >> scale, e & (n - 1), n), None


def _mix(x):
    x = (x ^ (x >> 31)) * 0x7FB5D329728EA185
    x = (x ^ (x >> 27)) * 0x01DADEF4BC2DD44D
    return (x ^ (x >> 33)) & M63


def _graph(case, seed, by=None):
    """(DeviceGraph, a coordinate in [0, 1) of every vertex or None). by: the graph that SHAPE gives, with
    renamed vertices and with weights of the seed."""
    gen = _gen(seed if by is None else SHAPE)
    if case["graph"] == "grid":
        n, (off, adj), x = _grid(case["rows"], case["cols"])
    elif case["graph"] == "rgg":
        n, (off, adj), x = _rgg(case["n"], gen)
    else:
        n, (off, adj), x = _rmat(case["scale"], gen)
    if by:
        off, adj = _renamed(n, torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1]), adj.long(), by)
        gen = _gen(seed)
    vw = ew = None
    if case["weights"] != "unit":
        # symmetric edge weights 1..8; 64-bit weights (a level of a hierarchy) come with vertex weights
        wide = case["weights"] == "int64"
        src = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
        lo, hi = torch.minimum(src, adj), torch.maximum(src, adj)
        ew = (1 + (_mix(lo * n + hi + (seed & M31)) & 7)).to(torch.int64 if wide else torch.int32)
        if wide:
            vw = torch.randint(1, 21, (n,), device="cuda", generator=gen)
    if case["weights"] != "int64":
        off = off.to(torch.int32)
    return gp.DeviceGraph(n, off, adj, vw, ew), x


def _bounds(dg, k):
    total = dg.n if dg.vw is None else int(dg.vw.sum())
    most = 1 if dg.vw is None else int(dg.vw.max())
    lmax = gp.lmax(total, k, EPS)
    return lmax, max(most, lmax // 14)


def _weights(seed):
    """A scorer (32 hidden units) with weights of the size that training gives them."""
    rng = np.random.default_rng(seed)
    return rng.normal(0, 0.2, (32, 8)), rng.normal(0, 0.1, 32), rng.normal(0, 0.2, 32), float(rng.normal(0, 0.1))


def _weights64(seed):
    """The same after the rounding that the scorer stores them with (bfloat16 weights, float32 biases)."""
    w1, b1, w2, b2 = (torch.as_tensor(v, device="cuda").float() for v in _weights(seed))
    return w1.bfloat16().double(), b1.double(), w2.bfloat16().double(), b2.double()


def _features(n, seed):
    """Features as rows of R-MAT graphs have them, and targets."""
    gen = _gen(seed)
    u = torch.rand(n, 8, device="cuda", generator=gen)
    lo, hi = 1 + 6 * u[:, 0], 3 + 9 * u[:, 1]
    c0, c1 = 1 + 3 * u[:, 3], 1 + 4 * u[:, 4]
    feat = torch.stack([torch.minimum(lo, hi), torch.maximum(lo, hi), 1 + 2.2 * u[:, 2], torch.minimum(c0, c1),
                        torch.maximum(c0, c1), (u[:, 5] * u[:, 5] * 64).floor() / 64, u[:, 6] * u[:, 6],
                        (u[:, 7] * 8).floor() / 16], 1)
    y = (torch.rand(n, device="cuda", generator=gen) < torch.sigmoid(2 * feat[:, 5] + feat[:, 6] - 0.5)).float()
    return feat.contiguous(), y


# ------------------------------------------------------------------------------------------ passes
def prepare(case, seed):
    s = dict(op=case["op"], seed=seed & M31)
    if case["op"] == "grad":
        s["feat"], s["y"] = _features(case["n"], seed)
        s["mlp"] = gp.mlp_pack(*_weights(seed & M31))
        return s
    if case["op"] == "batch":
        sizes, rng = np.random.default_rng(SHAPE), np.random.default_rng(seed & M31)
        s["graphs"], s["ks"], s["seeds"] = [], [], []
        for i in range(case["count"]):
            n = int(round(math.exp(sizes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
            if sizes.integers(2):
                rows = math.isqrt(n)
                c = dict(graph="grid", rows=rows, cols=-(-n // rows), weights="unit")
            else:
                c = dict(graph="rgg", n=n, weights="unit")
            s["graphs"].append(_graph(c, 1000 * (seed & M31) + i)[0])
            s["ks"].append(int((2, 4, 8)[rng.integers(3)]))
            s["seeds"].append(int(rng.integers(1 << 31)))
        return s
    if case["op"] == "contract":
        # a clustering of the coarsening phase, moved with the vertices to the seed's names
        base, by = _graph(case, SHAPE, 0)[0], 1 + (seed & M31)
        labels = gp.lp_cluster(base, _bounds(base, case["k"])[1], 10, SHAPE)[0].long()
        s["dg"] = _graph(case, seed, by)[0]
        n, v = base.n, torch.arange(base.n, device="cuda")
        s["labels"] = torch.empty(n, dtype=torch.int32, device="cuda")
        s["labels"][_rename(v, n, by)] = _rename(labels, n, by).to(torch.int32)
        return s
    dg, x = _graph(case, seed, 1 + (seed & M31) if case["op"] == "score" else None)
    s["dg"] = dg
    if case["op"] == "score":
        s["mlp"] = gp.mlp_pack(*_weights(seed & M31))
        return s
    s["k"] = k = case["k"]
    s["lmax"], s["U"] = _bounds(dg, k)
    if case["op"] == "refine":
        # strips with 3 % of the vertices in a neighbouring one, as a projected partition has ragged borders
        gen = _gen(seed + 1)
        part = (x * k).long().clamp_(max=k - 1)
        stray = torch.rand(dg.n, device="cuda", generator=gen) < 0.03
        s["part"] = torch.where(stray, (part + 1) % k, part).to(torch.int32)
    if case["op"] == "partition":
        s["params"] = gp.default_params(mls_global_iters=case.get("mls", 0))
    return s


class _Device:
    def __init__(self, ptr, count, kind):
        self.__cuda_array_interface__ = dict(shape=(count,), typestr=kind, data=(int(ptr), False), version=3, strides=None)


def run(s):
    op = s["op"]
    if op == "cluster":
        labels, st = gp.lp_cluster(s["dg"], s["U"], 10, s["seed"])
        return [labels, st["rounds"], st["moves"]]
    if op == "refine":
        part, bw, st = gp.lp_refine(s["dg"], s["part"], s["k"], s["lmax"], 25, s["seed"])
        return [part, bw, st["moves"]]
    if op == "contract":
        c, f2c = gp.contract(s["dg"], s["labels"])
        s["coarse"] = c  # owns the arrays returned below
        d = c.desc
        return [f2c] + [torch.as_tensor(_Device(p, m, t), device="cuda") for p, m, t in
                        ((d.offsets, c.n + 1, "<i8"), (d.adj, c.m_dir, "<i4"), (d.vwgt, c.n, "<i8"), (d.ewgt, c.m_dir, "<i8"))]
    if op == "score":
        return list(gp.mlp_score(s["dg"], 1, s["mlp"]))
    if op == "grad":
        return list(gp.mlp_grad(s["feat"], s["y"], s["mlp"]))
    if op == "batch":
        parts, res = gp.partition_batch(s["graphs"], s["ks"], EPS, s["seeds"])
        return [torch.cat(parts), np.array([r.cut for r in res])]
    part, res = gp.partition(s["dg"], s["k"], EPS, s["seed"], s["params"])
    return [part, res.cut, res.max_block_weight]


# ------------------------------------------------------------------------------------------ work
def _size(case):
    """Vertices and (nearly) the CSR entries of the case's graph."""
    if case["graph"] == "grid":
        a, b = case["rows"], case["cols"]
        return a * b, 4 * a * b - 2 * (a + b)
    if case["graph"] == "rgg":
        return case["n"], int(DEG * case["n"])
    return 1 << case["scale"], int((0.97 - 0.8 * 0.82 ** case["scale"]) * 2 * EDGE_FACTOR) << case["scale"]


def work(case):
    op = case["op"]
    if op == "grad":  # forward, and the two products of the backward pass
        return dict(bytes=36 * case["n"], flops=case["n"] * (2 * 288 + 4 * 288))
    if op == "batch":  # half grids (4 entries a vertex), half geometric graphs (12)
        n = case["count"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        return dict(bytes=int(n * (4 + 4 * 8 + 4)), flops=0)
    n, m = _size(case)
    wide = case["weights"] == "int64"
    size = (8 if wide else 4) * (n + 1) + 4 * m
    if case["weights"] != "unit":
        size += (8 if wide else 4) * m + (8 * n if wide else 0)
    if op == "score":
        return dict(bytes=size + 8 * m, flops=2 * 288 * m)
    if op == "contract":  # a coarse graph of about a third of a mesh's and all of a power-law graph's entries
        mc = m // 3 if case["graph"] != "rmat" else m // 2
        return dict(bytes=size + 8 * n + 12 * mc + 16 * (n // 4), flops=0)
    return dict(bytes=size + 4 * n + (4 * n if op == "refine" else 0), flops=0)


# ------------------------------------------------------------------------------------------ 64 bits
def exact(case, seed):
    if case["op"] == "grad":
        feat, y = _features(case["n"], seed)
        w1, b1, w2, b2 = _weights64(seed & M31)
        x, y = feat.double(), y.double()
        pre = x @ w1.T + b1
        h = pre.clamp(min=0)
        z = h @ w2 + b2
        loss = (z.clamp(min=0) - y * z + torch.log1p(torch.exp(-z.abs()))).mean()
        dz = (torch.sigmoid(z) - y) / y.numel()
        dh = torch.where(pre > 0, dz[:, None] * w2, 0.0)
        g = torch.cat([(dh.T @ x).reshape(-1), dh.sum(0), h.T @ dz, dz.sum().reshape(1)])
        return [float(loss), g.cpu().numpy()]
    if case["op"] != "score":
        return None
    dg = _graph(case, seed, 1 + (seed & M31))[0]
    w1, b1, w2, b2 = _weights64(seed & M31)
    n, m, off, adj = dg.n, dg.m_dir, dg.off.long(), dg.adj.long()
    deg = off[1:] - off[:-1]
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    ew = torch.ones(m, dtype=torch.float64, device="cuda") if dg.ew is None else dg.ew.double()
    wdeg = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, src, ew)
    pos = torch.arange(m, device="cuda") - off[src]
    heads = (src * n + adj)[pos < 64]  # (vertex, neighbour) of each vertex's first 64 neighbours, ascending
    out = torch.empty(m, dtype=torch.float64, device="cuda")
    for e0 in range(0, m, 1 << 22):
        v, u, w = src[e0:e0 + (1 << 22)], adj[e0:e0 + (1 << 22)], ew[e0:e0 + (1 << 22)]
        shared = torch.zeros(v.numel(), dtype=torch.float64, device="cuda")
        for t in range(64):
            at = (deg[u] > t).nonzero().reshape(-1)
            want = v[at] * n + adj[off[u[at]] + t]
            i = torch.searchsorted(heads, want).clamp_(max=heads.numel() - 1)
            shared[at] += heads[i] == want
        dv, du = deg[v].double(), deg[u].double()
        one = torch.ones_like(w)
        f = torch.stack([torch.log2(1 + torch.minimum(dv, du)), torch.log2(1 + torch.maximum(dv, du)), torch.log2(1 + w),
                         one, one, shared / 64, w / torch.maximum(wdeg[v], wdeg[u]), one / 16], 1)
        out[e0:e0 + (1 << 22)] = torch.sigmoid(torch.relu(f @ w1.T + b1) @ w2 + b2)
    return [out, None]

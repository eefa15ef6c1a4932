"""Kernels at the edges of their tiles, tables and size rules, against the oracle.

Label propagation, contraction, local search and placement work in whole numbers, so the results are equal;
features are sums of at most a few thousand terms, the scorer's bounds are those of its own tests."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gp():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_1710_08231_gb300 as m
    m.build()
    m.lp_set_schedule(0, 0)
    return m


def _from_pairs(n, a, b, weight=None, vw=None):
    """Symmetric CSR from pairs (duplicates and loops dropped); weight(lo, hi) gives int64 edge weights."""
    a, b = np.asarray(a, np.int64), np.asarray(b, np.int64)
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    key = np.unique((lo * n + hi)[lo != hi])
    lo, hi = key // n, key % n
    w = weight(lo, hi).astype(np.int64) if weight else None
    src, dst = np.concatenate([lo, hi]), np.concatenate([hi, lo])
    order = np.lexsort((dst, src))
    off = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int64)
    return gg.Graph(n, off, dst[order].astype(np.int32), vw, None if w is None else np.concatenate([w, w])[order], "pairs")


def _ring(n, d, weight=None):
    """Every vertex is joined to its d // 2 next ones on a ring (degree d), with shuffled ids."""
    p = np.random.default_rng(n + d).permutation(n)
    i = np.arange(n)
    a = np.concatenate([p[i]] * (d // 2))
    b = np.concatenate([p[(i + s) % n] for s in range(1, d // 2 + 1)])
    return _from_pairs(n, a, b, weight)


_SMALL = lambda lo, hi: 1 + (lo * 31 + hi * 17) % 9
_WIDE = lambda lo, hi: (1 + (lo * 31 + hi * 17) % 5) << np.where((lo + hi) % 11 == 0, 30, 3)


def _lp_same(gp, g, U, k):
    import torch
    dg = gp.DeviceGraph.from_host(g)
    lab, st = gp.lp_cluster(dg, U, 6, 77)
    lab_o, _, st_o = O.lp_cluster(g, U, 6, 77)
    assert np.array_equal(lab.cpu().numpy(), lab_o)
    assert (st["moves"], st["visits"], st["edges"]) == (st_o.moves, st_o.visits, st_o.edges)
    part = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
    lm = O.lmax(int(O.vertex_weights(g).sum()), k, 0.03)
    p, bw, _ = gp.lp_refine(dg, torch.from_numpy(part).cuda(), k, lm, 8, 5)
    p_o, bw_o, _ = O.lp_refine(g, part, k, lm, 8, 5)
    assert np.array_equal(p.cpu().numpy(), p_o) and np.array_equal(bw.cpu().numpy(), bw_o)


@pytest.mark.parametrize("n,d", [(7, 2), (8, 4), (2047, 8), (2049, 10), (4096, 16), (5000, 18), (3000, 32), (3000, 34),
                                 (1500, 128), (1500, 130), (1300000, 4)])
@pytest.mark.parametrize("weight", [None, _SMALL, _WIDE], ids=["unit", "small", "wide"])
def test_lp_row_lengths(gp, n, d, weight):
    """Rows at the limits of the bins (8, 16, 32), of the block-owned form (128), blocks of one and several tiles, and
    weights whose sums do not fit 32 bits."""
    if n > 100000 and weight is _SMALL:
        pytest.skip("covered by the other two")
    _lp_same(gp, _ring(n, d, weight), 40, 5)


@pytest.mark.parametrize("d", [256, 257, 1024, 1025, 2048, 2049, 4097])
def test_lp_long_rows(gp, d):
    """A few vertices of one long degree over a mesh: warp, team, block and hub tables at their limits, with contests
    above and below the size whose moves all blocks make."""
    n = 3 * d + 500
    rng = np.random.default_rng(d)
    hubs = rng.permutation(n)[:3]
    i = np.arange(n - 1)
    a = [i] + [np.full(d, h) for h in hubs]
    b = [i + 1] + [rng.permutation(n)[:d] for _ in hubs]
    _lp_same(gp, _from_pairs(n, np.concatenate(a), np.concatenate(b), _SMALL), n // 3, 3)


@pytest.mark.parametrize("n", [3, 1000, 40000, 70000])
@pytest.mark.parametrize("parts", [1, 255, 257, 0])
def test_contract_widths(gp, n, parts):
    """Coarse ids of one and several digits, one coarse vertex, all of them, long stretches of vertices without edges,
    and 64-bit weight sums."""
    import torch
    rng = np.random.default_rng(n + parts)
    a = rng.integers(0, n // 3 + 1, 4 * n)
    b = rng.integers(0, n // 3 + 1, 4 * n)
    far = np.where(rng.random(4 * n) < 0.5, 0, n - n // 3 - 1)  # (the middle third has no edges)
    g = _from_pairs(n, a + far, b + far, _WIDE)
    lab = np.arange(n, dtype=np.int32) if parts == 0 else (rng.integers(0, min(parts, n), n)).astype(np.int32)
    cg, f2c = gp.contract(gp.DeviceGraph.from_host(g), torch.from_numpy(lab).cuda())
    h = cg.to_host()
    co, f2c_o = O.contract(g, lab)
    assert h.n == co.n and np.array_equal(f2c.cpu().numpy(), f2c_o)
    for x in ("off", "adj", "vw", "ew"):
        assert np.array_equal(getattr(h, x), getattr(co, x)), x


def test_dropped_coarse_graph_frees_late(gp):
    """A coarse graph that goes out of scope keeps its arrays until the library allocates again."""
    import torch
    g = gg.grid(60, 60)
    dg = gp.DeviceGraph.from_host(g)
    lab = torch.from_numpy((np.arange(g.n) // 4).astype(np.int32)).cuda()
    want = None
    for _ in range(50):
        cg, _ = gp.contract(dg, lab)
        h = cg.to_host()
        want = want or h
        assert np.array_equal(h.adj, want.adj) and np.array_equal(h.off, want.off)
        del cg


@pytest.mark.parametrize("d", [2, 14, 16, 18, 64, 1100])
def test_features_list_lengths(gp, d):
    """Lists of one and several lookup steps, and rows above the table's slots."""
    g = _ring(1500, d, _SMALL)
    g.ew = g.ew.astype(np.int32)
    f = gp.edge_features(gp.DeviceGraph.from_host(g), 2).cpu().numpy().astype(np.float64)
    assert np.allclose(f, O.edge_features(g, 2), rtol=2e-6, atol=2e-6)


@pytest.mark.parametrize("m", [1, 31, 33, 257])
def test_gradients_few_entries(gp, m):
    import torch
    rng = np.random.default_rng(m)
    feat = rng.random((m, 8)).astype(np.float32)
    y = (rng.random(m) < 0.5).astype(np.float32)
    mlp = gp.mlp_pack(rng.normal(0, 0.3, (32, 8)).astype(np.float32), rng.normal(0, 0.3, 32).astype(np.float32),
                      rng.normal(0, 0.3, 32).astype(np.float32), np.float32(0.1))
    loss, grad = gp.mlp_grad(torch.from_numpy(feat).cuda(), torch.from_numpy(y).cuda(), mlp)
    w1, b1, w2, b2 = gp.mlp_unpack(mlp)
    loss64, gw1, gb1, gw2, gb2 = O.mlp_loss_grad(feat.astype(np.float64), y.astype(np.float64), w1, b1, w2, b2)
    want = np.concatenate([gw1.reshape(-1), gb1, gw2, [gb2]])
    got = grad.astype(np.float64)
    assert ((np.abs(got - want) <= 1e-3) | (np.abs(got - want) <= 2e-2 * np.abs(want))).all()
    assert abs(loss - loss64) <= 1e-4 * max(1.0, abs(loss64))


@pytest.mark.parametrize("k,weighted", [(2, True), (64, False), (65, True), (256, False)])
def test_mls_many_blocks_and_long_lists(gp, k, weighted):
    """k around the limit of the connections per lane; a random start makes every vertex a boundary vertex, which is
    more than one launch ranks."""
    import torch
    g = gg.rgg(10000, 9.0, 8)
    if weighted:
        src = np.repeat(np.arange(g.n), np.diff(g.off))
        g.ew = _SMALL(np.minimum(src, g.adj), np.maximum(src, g.adj)).astype(np.int32)
    part0 = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
    lmax = int(np.bincount(part0, minlength=k).max()) + 3
    p = gp.mls_default_params(global_iters=1, max_local=3)
    po = O.mls_default_params()
    po.global_iters, po.max_local = 1, 3
    out, st = gp.mls(gp.DeviceGraph.from_host(g), torch.from_numpy(part0).cuda(), k, lmax, 3, p)
    out_o, st_o = O.mls(g, part0, k, lmax, 3, po)
    assert np.array_equal(out.cpu().numpy(), out_o) and st == st_o


@pytest.mark.parametrize("k,extra,weighted", [(1, 5, False), (33, 1000, False), (1024, 3000, False), (1025, 3000, False),
                                              (3, 700, True), (40, 700, True)])
def test_placement_of_isolated_vertices(gp, k, extra, weighted):
    """Degree-0 vertices by the closed form (up to 1024 blocks with sorted weights, above without) and one by one."""
    base = gg.rgg(4000, 8.0, 9)
    n = base.n + extra
    off = np.concatenate([base.off, np.full(extra, base.off[-1], dtype=base.off.dtype)])
    vw = np.random.default_rng(4).integers(1, 9, n).astype(np.int32) if weighted else None
    g = gg.Graph(n, off, base.adj, vw, None, "rgg+isolated")
    part, res = gp.partition(gp.DeviceGraph.from_host(g), k, 0.05, 5)
    part_o, res_o = O.partition(g, k, 0.05, 5)
    assert np.array_equal(part.cpu().numpy(), part_o)
    assert (res.cut, res.n_isolated, res.max_block_weight) == (res_o.cut, res_o.n_isolated, res_o.max_block_weight)

"""Label propagation on block-owned vertices, rows of 33 to 128 entries by tables of four or eight warps, against the
oracle (whole numbers, so everything is equal)."""
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
    m.lp_set_tiles(0, 0)
    return m


def _mixed(n, share, weighted):
    """A ring of degree 4 where a share of the vertices is joined to the next 40 ones as well (degree 44 and more,
    at most 128 by the share's spacing)."""
    i = np.arange(n)
    h = i[:: max(1, round(1 / share))]
    a = np.concatenate([i, i] + [h] * 40)
    b = np.concatenate([(i + 1) % n, (i + 2) % n] + [(h + s) % n for s in range(3, 43)])
    lo, hi = np.minimum(a, b).astype(np.int64), np.maximum(a, b).astype(np.int64)
    key = np.unique(lo * n + hi)
    lo, hi = key // n, key % n
    w = 1 + (lo * 31 + hi * 17) % 9
    src, dst = np.concatenate([lo, hi]), np.concatenate([hi, lo])
    order = np.lexsort((dst, src))
    off = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int64)
    g = gg.Graph(n, off, dst[order].astype(np.int32), None,
                 np.concatenate([w, w])[order].astype(np.int32) if weighted else None, "mixed")
    assert 32 < np.diff(off).max() <= 128
    return g


@pytest.mark.parametrize("n", [3000, 45000])
@pytest.mark.parametrize("share", [1 / 50, 1 / 17, 1 / 15, 1 / 2])
@pytest.mark.parametrize("weighted,scored", [(False, False), (True, False), (False, True), (True, True)])
def test_tables_of_four_and_eight_warps(gp, n, share, weighted, scored):
    """Shares of long rows around the line between the two, one tile a block and several problems' worth of blocks;
    the refinement of a random partition has contests whose keys cover the rows kept beside the tables."""
    import torch
    g = _mixed(n, share, weighted)
    dg = gp.DeviceGraph.from_host(g)
    q = None
    if scored:
        src = np.repeat(np.arange(n), np.diff(g.off))
        q = ((np.minimum(src, g.adj) * 7 + np.maximum(src, g.adj) * 13) % 32769).astype(np.int32)
    for vpb in (0, 4096):
        gp.lp_set_tiles(0, vpb)
        lab, st = gp.lp_cluster(dg, 90, 6, 3, None if q is None else torch.from_numpy(q).cuda())
        part = np.random.default_rng(1).integers(0, 6, n).astype(np.int32)
        lm = O.lmax(n, 6, 0.03)
        p, bw, st_r = gp.lp_refine(dg, torch.from_numpy(part).cuda(), 6, lm, 6, 5)
        gp.lp_set_tiles(0, 0)
        if vpb == 0:
            lab_o, _, st_o = O.lp_cluster(g, 90, 6, 3, q)
            p_o, bw_o, st_ro = O.lp_refine(g, part, 6, lm, 6, 5)
        assert np.array_equal(lab.cpu().numpy(), lab_o) and st["moves"] == st_o.moves
        assert np.array_equal(p.cpu().numpy(), p_o) and np.array_equal(bw.cpu().numpy(), bw_o)
        assert st_r["moves"] == st_ro.moves


@pytest.mark.parametrize("n", [250, 600, 5000, 20000, 45000])
@pytest.mark.parametrize("k", [2, 9])
@pytest.mark.parametrize("weighted", [False, True])
def test_contests_decided_by_one_block(gp, n, k, weighted):
    """Random partitions: contests of a few, hundreds and thousands of proposals, whose moves are made by the block that
    decides them or by all blocks of the problem."""
    import torch
    g = gg.rgg(n, 9.0, 12)
    if weighted:
        src = np.repeat(np.arange(n), np.diff(g.off))
        g.ew = (1 + (np.minimum(src, g.adj).astype(np.int64) * 31 + np.maximum(src, g.adj) * 17) % 9).astype(np.int32)
        g.vw = np.random.default_rng(n).integers(1, 6, n).astype(np.int64)
    part = np.random.default_rng(k).integers(0, k, n).astype(np.int32)
    lm = O.lmax(int(O.vertex_weights(g).sum()), k, 0.02)
    p, bw, st = gp.lp_refine(gp.DeviceGraph.from_host(g), torch.from_numpy(part).cuda(), k, lm, 12, 5)
    p_o, bw_o, st_o = O.lp_refine(g, part, k, lm, 12, 5)
    assert np.array_equal(p.cpu().numpy(), p_o) and np.array_equal(bw.cpu().numpy(), bw_o)
    assert (st["moves"], st["visits"]) == (st_o.moves, st_o.visits)


@pytest.mark.parametrize("n", [40, 3001, 90000])
@pytest.mark.parametrize("extra", [0, 1, 6])
@pytest.mark.parametrize("weighted,scored", [(False, False), (True, False), (False, True), (True, True)])
def test_groups_of_four_and_eight_lanes(gp, n, extra, weighted, scored):
    """Rows of at most 4 entries only (four lanes each), one row of 5, and one of 10 (no row of 5 to 8 but longer
    ones), with tiles too small for a thread per row and larger ones."""
    import torch
    i = np.arange(n)
    a, b = np.concatenate([i, i]), np.concatenate([(i + 1) % n, (i + 7) % n])
    a, b = np.concatenate([a, [3] * extra]), np.concatenate([b, (3 + 9 + 2 * np.arange(extra)) % n])
    lo, hi = np.minimum(a, b).astype(np.int64), np.maximum(a, b).astype(np.int64)
    if extra == 6:  # (the row of 10 has its new neighbours' other edges taken out: they have 1 + at most 3)
        keep = ~(np.isin(lo, (3 + 9 + 2 * np.arange(6)) % n) & (hi == lo + 1))
        lo, hi = lo[keep], hi[keep]
    if extra == 1:
        keep = ~((lo == (3 + 9) % n) & (hi == lo + 1))
        lo, hi = lo[keep], hi[keep]
    key = np.unique(lo * n + hi)
    lo, hi = key // n, key % n
    w = 1 + (lo * 31 + hi * 17) % 9
    src, dst = np.concatenate([lo, hi]), np.concatenate([hi, lo])
    order = np.lexsort((dst, src))
    off = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int64)
    g = gg.Graph(n, off, dst[order].astype(np.int32), None,
                 np.concatenate([w, w])[order].astype(np.int32) if weighted else None, "four")
    d = np.diff(off)
    assert (d.max(), ((d > 4) & (d <= 8)).sum()) == {0: (4, 0), 1: (5, 1), 6: (10, 0)}[extra]
    q = None
    if scored:
        s = np.repeat(i, d)
        q = ((np.minimum(s, g.adj) * 7 + np.maximum(s, g.adj) * 13) % 32769).astype(np.int32)
    dg = gp.DeviceGraph.from_host(g)
    for vpb in (0, 4096):
        gp.lp_set_tiles(0, vpb)
        lab, st = gp.lp_cluster(dg, 30, 6, 3, None if q is None else torch.from_numpy(q).cuda())
        gp.lp_set_tiles(0, 0)
        lab_o, _, st_o = O.lp_cluster(g, 30, 6, 3, q)
        assert np.array_equal(lab.cpu().numpy(), lab_o) and st["moves"] == st_o.moves

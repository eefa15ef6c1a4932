"""Label propagation with edge weights whose connections and gains need more than 32 bits, against the oracle: whole
numbers, so labels, block weights and counters are equal. Weights are multiples of 2^26 .. 2^50, which leaves the low
half of every gain zero from 2^32 on."""
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


def _weighted(g, shift, kind=np.int64):
    src = np.repeat(np.arange(g.n), np.diff(g.off))
    lo, hi = np.minimum(src, g.adj).astype(np.int64), np.maximum(src, g.adj).astype(np.int64)
    g.ew = ((1 + (lo * 31 + hi * 17) % 8) << shift).astype(kind)
    return g


def _same(gp, g, U, k, q=None):
    import torch
    dg = gp.DeviceGraph.from_host(g)
    qd = None if q is None else torch.from_numpy(q).cuda()
    lab, st = gp.lp_cluster(dg, U, 8, 3, qd)
    lab_o, _, st_o = O.lp_cluster(g, U, 8, 3, q)
    assert np.array_equal(lab.cpu().numpy(), lab_o)
    assert (st["moves"], st["visits"], st["edges"]) == (st_o.moves, st_o.visits, st_o.edges)
    part = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
    lm = O.lmax(g.n, k, 0.03)
    p, bw, st = gp.lp_refine(dg, torch.from_numpy(part).cuda(), k, lm, 8, 5)
    p_o, bw_o, st_o = O.lp_refine(g, part, k, lm, 8, 5)
    assert np.array_equal(p.cpu().numpy(), p_o) and np.array_equal(bw.cpu().numpy(), bw_o)
    assert st["moves"] == st_o.moves


@pytest.mark.parametrize("shift", [31, 32, 36, 50])
@pytest.mark.parametrize("n,deg", [(3000, 12.0), (30000, 12.0), (3000, 120.0)],
                         ids=["one tile a block", "many blocks", "long rows"])
def test_gains_above_32_bits(gp, n, deg, shift):
    """Contested moves are ordered by gains of which only the high half differs from zero."""
    _same(gp, _weighted(gg.rgg(n, deg, 4), shift), 60, 13)


@pytest.mark.parametrize("shift", [32, 40])
def test_scored_gains_above_32_bits(gp, shift):
    g = _weighted(gg.rgg(4000, 12.0, 6), shift)
    src = np.repeat(np.arange(g.n), np.diff(g.off))
    q = ((np.minimum(src, g.adj) * 7 + np.maximum(src, g.adj) * 13) % 32769).astype(np.int32)
    _same(gp, g, 40, 5, q)


@pytest.mark.parametrize("shift,kind", [(26, np.int32), (30, np.int64), (40, np.int64)])
@pytest.mark.parametrize("deg", [6.0, 12.0])
def test_wide_weights_of_short_rows(gp, deg, shift, kind):
    """Enough vertices for a thread per row (rows of up to 8 and 16 entries), weights whose sums do not fit there."""
    _same(gp, _weighted(gg.rgg(60000, deg, 9), shift, kind), 30, 7)


@pytest.mark.parametrize("n,deg", [(2000, 20.0), (60000, 24.0), (60000, 9.0)])
@pytest.mark.parametrize("shift", [None, 0, 27])
def test_scored_rows_of_lane_groups(gp, n, deg, shift):
    """Rows of up to 32 entries with scores: connections and score sums over equal labels, few or many of them."""
    g = gg.rgg(n, deg, 6)
    if shift is not None:
        g = _weighted(g, shift)
    src = np.repeat(np.arange(g.n), np.diff(g.off))
    q = ((np.minimum(src, g.adj) * 7 + np.maximum(src, g.adj) * 13) % 32769).astype(np.int32)
    _same(gp, g, 60, 5, q)

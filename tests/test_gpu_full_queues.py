"""Multi-try search with queues that are full most of the time, rows on both sides of what a lane walks alone (64
entries) and block counts on both sides of the connections per lane (64), against the oracle."""
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
    return m


@pytest.mark.parametrize("k", [2, 16, 64, 65])
@pytest.mark.parametrize("cap", [1, 5, 40, 256])
def test_full_queues(gp, k, cap):
    import torch
    weights = ("unit", "int32", "int64")[(k + cap) % 3]
    g = gg.rmat(10, 12, seed=3)
    deg = np.diff(g.off)
    assert (deg > 64).sum() > 20 and (deg <= 64).sum() > 500
    if weights != "unit":
        src = np.repeat(np.arange(g.n), deg)
        w = 1 + (np.minimum(src, g.adj) * 31 + np.maximum(src, g.adj) * 17) % 9
        g = gg.Graph(g.n, g.off, g.adj, None, w.astype(weights), g.name)
    part0 = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
    lmax = int(np.bincount(part0, minlength=k).max()) + 3
    p, po = gp.mls_default_params(global_iters=1, max_local=2, max_moves=12, queue_cap=cap), O.mls_default_params()
    po.global_iters, po.max_local, po.max_moves, po.queue_cap = 1, 2, 12, cap
    out, st = gp.mls(gp.DeviceGraph.from_host(g), torch.from_numpy(part0).cuda(), k, lmax, 3, p)
    out_o, st_o = O.mls(g, part0, k, lmax, 3, po)
    assert np.array_equal(out.cpu().numpy(), out_o) and st == st_o

"""A device wait that runs out returns GP_ERR_TIMEOUT in every kernel whose blocks meet: LP in its list form (rows above
128 entries) and the contraction. The context stays usable and the next call gives the oracle's result."""
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
    m.lp_set_hub_keep(0, 0)
    return m


def _runs_out(gp, call):
    gp.set_wait_limit(1)
    try:
        with pytest.raises(gp.GpError) as ei:
            call()
        assert ei.value.status == gp.GP_ERR_TIMEOUT
        assert "barrier" in str(ei.value)
    finally:
        gp.set_wait_limit(0)


def test_lp_list_form(gp):
    g = gg.rmat(15, 16, seed=3)
    assert int(np.diff(g.off).max()) > 128
    dg = gp.DeviceGraph.from_host(g)
    _runs_out(gp, lambda: gp.lp_cluster(dg, 60, 10, 3))
    lab, _ = gp.lp_cluster(dg, 60, 10, 3)
    assert np.array_equal(lab.cpu().numpy(), O.lp_cluster(g, 60, 10, 3)[0])


@pytest.mark.parametrize("weights", ["unit", "int32", "int64"])
def test_contraction(gp, weights):
    import torch
    g = gg.rgg(100_000, 12.0, 4)  # about 300 tiles of pairs
    if weights != "unit":
        src = np.repeat(np.arange(g.n), np.diff(g.off))
        w = (np.minimum(src, g.adj) * 7 + np.maximum(src, g.adj) * 13) % 8 + 1
        g = gg.Graph(g.n, g.off, g.adj, None, w.astype(weights), g.name)
    lab = (np.arange(g.n) // 3).astype(np.int32)
    dg, dlab = gp.DeviceGraph.from_host(g), torch.from_numpy(lab).cuda()
    _runs_out(gp, lambda: gp.contract(dg, dlab))
    cg, f2c = gp.contract(dg, dlab)
    h = cg.to_host()
    co, f2c_o = O.contract(g, lab)
    assert np.array_equal(f2c.cpu().numpy(), f2c_o)
    for x in ("off", "adj", "vw", "ew"):
        assert np.array_equal(getattr(h, x), getattr(co, x)), x

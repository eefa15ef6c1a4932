"""Initial partitioning on both sides of the line (32 entries a row on average) above which a large BFS frontier is taken
from the side of the vertices without a distance, against the oracle."""
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


def _ring(n, d):
    """Every vertex is joined to its d // 2 next ones on a ring, with shuffled ids."""
    p = np.random.default_rng(n + d).permutation(n)
    i = np.arange(n)
    src = np.concatenate([p[i]] * (d // 2) + [p[(i + s) % n] for s in range(1, d // 2 + 1)])
    dst = np.concatenate([p[(i + s) % n] for s in range(1, d // 2 + 1)] + [p[i]] * (d // 2))
    order = np.lexsort((dst, src))
    return gg.Graph(n, np.arange(n + 1, dtype=np.int64) * d, dst[order].astype(np.int32), None, None, "ring")


@pytest.mark.parametrize("graph", ["ring32", "ring34", "rmat_dense", "rmat_thin", "grid"])
@pytest.mark.parametrize("k", [2, 7, 40])
def test_partition(gp, graph, k):
    g = {"ring32": lambda: _ring(1500, 32), "ring34": lambda: _ring(1500, 34), "rmat_dense": lambda: gg.rmat(10, 64, seed=3),
         "rmat_thin": lambda: gg.rmat(11, 6, seed=3), "grid": lambda: gg.grid(50, 41)}[graph]()
    assert (g.adj.size > 32 * g.n) == (graph in ("ring34", "rmat_dense"))
    p, po = gp.default_params(coarse_min=4000), O.default_params()
    po.coarse_min = 4000  # (no coarsening: the bisection sees the graph itself)
    part, res = gp.partition(gp.DeviceGraph.from_host(g), k, 0.03, 5, p)
    part_o, res_o = O.partition(g, k, 0.03, 5, po)
    assert np.array_equal(part.cpu().numpy(), part_o) and (res.cut, res.levels) == (res_o.cut, res_o.levels)

"""Scores of short rows, which are staged across rows and scored 32 at a time: entries that end inside, at and one past a
step of 32, rows from one entry to more than a step, segments that end inside rows."""
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


def _csr(n, pairs, weighted):
    lo, hi = np.array(sorted(pairs), dtype=np.int64).reshape(-1, 2).T
    src, dst = np.concatenate([lo, hi]), np.concatenate([hi, lo])
    order = np.lexsort((dst, src))
    off = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int64)
    w = (1 + (lo * 31 + hi * 17) % 9).astype(np.int64)
    return gg.Graph(n, off, dst[order].astype(np.int32), None, np.concatenate([w, w])[order] if weighted else None, "csr")


def _path(n):
    return n, {(i, i + 1) for i in range(n - 1)}


def _star(leaves):
    return leaves + 1, {(0, i) for i in range(1, leaves + 1)}


def _mixed(n):
    # rows of 2 to 70 entries, with vertices without entries between them
    e = {(i, i + 1) for i in range(0, n - 1) if i % 7}
    return n, e | {(h, x) for h in range(3, n, 97) for x in range(h + 2, min(n, h + 70))}


GRAPHS = {"path2": _path(2), "path16": _path(16), "path17": _path(17), "path18": _path(18), "path33": _path(33),
          "star31": _star(31), "star32": _star(32), "star33": _star(33), "mixed40": _mixed(40), "mixed3001": _mixed(3001)}


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("name", [*GRAPHS, "grid", "rgg"])
def test_scores(gp, name, weighted):
    if name in GRAPHS:
        g = _csr(*GRAPHS[name], weighted)
    else:  # (grid: long enough for segments of more than 32 entries)
        g = gg.grid(700, 401) if name == "grid" else gg.rgg(20011, 11.0, 2)
    rng = np.random.default_rng(5)
    mlp = gp.mlp_pack(rng.normal(0, 0.5, (32, 8)).astype(np.float32), rng.normal(0, 0.3, 32).astype(np.float32),
                      rng.normal(0, 0.5, 32).astype(np.float32), np.float32(0.1))
    s, q = (t.cpu().numpy() for t in gp.mlp_score(gp.DeviceGraph.from_host(g), 1, mlp))
    s64 = O.mlp_forward(O.edge_features(g, 1), *gp.mlp_unpack(mlp))
    # the bound that the scorer is specified with: BF16 features and hidden units
    assert np.abs(s.astype(np.float64) - s64).max() <= 1e-2
    assert np.array_equal(q, np.rint(s * np.float32(32768.0)).astype(np.int32))
    src = np.repeat(np.arange(g.n), np.diff(g.off))
    assert np.array_equal(q[np.lexsort((g.adj, src))], q[np.lexsort((src, g.adj))])

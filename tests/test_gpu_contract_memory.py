"""Contraction with an allocator that gives a bounded number of bytes: the pairs are sorted in parts where they do not
fit at once, with the same coarse graph."""
import ctypes

import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu

gp_alloc_fn = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)
gp_free_fn = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)


@pytest.fixture(scope="module")
def gp():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_1710_08231_gb300 as m
    m.build()
    return m


class _Bounded:
    """Allocator callback on PyTorch's allocator that refuses what would exceed `most` bytes in use."""

    def __init__(self, most):
        import torch
        self.most, self.used, self.refused, self.live = most, 0, 0, {}

        @gp_alloc_fn
        def alloc(nbytes, stream, ctx):
            if self.used + nbytes > self.most:
                self.refused += 1
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)
            self.live[p] = int(nbytes)
            self.used += int(nbytes)
            return p

        @gp_free_fn
        def free(ptr, nbytes, stream, ctx):
            if ptr:
                self.used -= self.live.pop(ptr)
                torch.cuda.caching_allocator_delete(ptr)

        self.alloc, self.free = alloc, free


def _weighted(g, kind, rng):
    """Symmetric edge weights of the kind, with odd vertex weights for 64 bits."""
    if kind == "unit":
        return g
    src = np.repeat(np.arange(g.n), np.diff(g.off))
    lo, hi = np.minimum(src, g.adj), np.maximum(src, g.adj)
    w = (lo * 7 + hi * 13) % 8 + 1
    ew = w.astype(np.int32) if kind == "int32" else w.astype(np.int64) << 33
    vw = rng.integers(1, 20, g.n) if kind == "int64" else None
    return gg.Graph(g.n, g.off, g.adj, vw, ew, g.name)


@pytest.mark.parametrize("kind", ["unit", "int32", "int64"])
@pytest.mark.parametrize("labels", ["identity", "pairs", "blocks", "mod", "giant"])
def test_contract_in_parts(gp, kind, labels):
    import torch
    rng = np.random.default_rng(5)
    g = _weighted(gg.rgg(131101, 12.0, 4), kind, rng)
    n, m = g.n, g.adj.size
    v = np.arange(n)
    # (giant: one cluster of a fifth of the entries, so that a part is one row of more than an eighth of them)
    lab = {"identity": v, "pairs": v // 2, "blocks": v // 64, "mod": rng.integers(0, 3000, n),
           "giant": np.where(v % 5 == 0, 7, v)}[labels].astype(np.int32)
    co, f2c_o = O.contract(g, lab)
    dg, dlab = gp.DeviceGraph.from_host(g), torch.from_numpy(lab).cuda()
    mc = co.adj.size
    # 12 bytes per entry and 60 per vertex of scratch beside the coarse graph (3 MB for rounding)
    bounded = _Bounded(12 * m + 60 * n + 12 * mc + 16 * co.n + (3 << 20))
    gp.lib().gp_set_allocator(ctypes.cast(bounded.alloc, ctypes.c_void_p), ctypes.cast(bounded.free, ctypes.c_void_p), None)
    try:
        cg, f2c = gp.contract(dg, dlab)
        assert bounded.refused, "the pairs fitted: the parts were not reached"
        h = cg.to_host()
        cg.free()
        gp.free_cached()
        assert not bounded.live
    finally:
        gp.free_cached()
        gp._install_torch_allocator(gp.lib())
    assert h.n == co.n and np.array_equal(f2c.cpu().numpy(), f2c_o)
    for x in ("off", "adj", "vw", "ew"):
        assert np.array_equal(getattr(h, x), getattr(co, x)), x


def test_partition_with_little_memory(gp):
    """A whole partition whose contractions run in parts, against the oracle (degree classes come with them)."""
    g = gg.rgg(60000, 12.0, 9)
    dg = gp.DeviceGraph.from_host(g)
    ref, res = gp.partition(dg, 8, 0.03, 3)
    ref = ref.cpu().numpy()
    part_o, res_o = O.partition(g, 8, 0.03, 3)
    assert np.array_equal(ref, part_o)
    got = 0
    for most in range(20 << 20, 60 << 20, 2 << 20):
        b = _Bounded(most)
        gp.lib().gp_set_allocator(ctypes.cast(b.alloc, ctypes.c_void_p), ctypes.cast(b.free, ctypes.c_void_p), None)
        try:
            part, r = gp.partition(dg, 8, 0.03, 3)
        except gp.GpError as e:
            assert e.status == gp.GP_ERR_OOM
            continue
        finally:
            gp.free_cached()
            assert not b.live
            gp._install_torch_allocator(gp.lib())
        assert np.array_equal(part.cpu().numpy(), ref) and r.cut == res.cut
        got += b.refused > 0
    assert got, "no bound between refusing everything and everything fitting at once"

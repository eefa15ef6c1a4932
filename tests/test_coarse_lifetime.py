"""The arrays of a coarse graph live as long as their CoarseGraph or the map that came with it, and no longer."""
import copy
import ctypes
import gc
import pickle
import types

import numpy as np
import pytest

import paper_1710_08231_gb300 as gp


class _FakeLib:
    """gp_contract and the calls on its result; records the handles given back."""

    def __init__(self):
        self.made, self.freed, self.graph = 0, [], gp.GpGraph()
        self.graph.n, self.graph.m_dir = 3, 4

    def gp_contract(self, g, labels, coarse, f2c, stream):
        self.made += 1
        ctypes.cast(coarse, ctypes.POINTER(ctypes.c_void_p))[0] = self.made
        return gp.GP_OK

    def gp_coarse_graph(self, handle):
        return ctypes.pointer(self.graph)

    def gp_coarse_free(self, handle, stream):
        self.freed.append(handle.value)

    gp_coarse_drop = gp_coarse_free


@pytest.fixture
def fake(monkeypatch):
    import torch
    f = _FakeLib()
    monkeypatch.setattr(gp, "lib", lambda: f)
    monkeypatch.setattr(gp, "_stream", lambda s=None: None)
    dg = types.SimpleNamespace(n=5, adj=torch.zeros(1, dtype=torch.int32), desc=gp.GpGraph())
    return f, lambda: gp.contract(dg, torch.zeros(5, dtype=torch.int32))


@pytest.mark.parametrize("first", ["graph", "map"])
def test_last_holder_gives_back(fake, first):
    f, contract = fake
    cg, f2c = contract()
    if first == "graph":
        del cg
        gc.collect()
        assert f.freed == []
        kept = f2c.numpy()  # (other views of the map's storage do not count)
        del f2c
    else:
        del f2c
        gc.collect()
        assert f.freed == [] and cg.handle.value == 1
        del cg
    gc.collect()
    assert f.freed == [1]


def test_free_at_once(fake):
    f, contract = fake
    cg, f2c = contract()
    cg.free()
    assert f.freed == [1] and cg.handle is None
    cg.free()
    del cg, f2c
    gc.collect()
    assert f.freed == [1]


def test_copies_of_the_map(fake):
    f, contract = fake
    cg, f2c = contract()
    twin, again = copy.deepcopy(f2c), pickle.loads(pickle.dumps(f2c))
    del cg, f2c
    gc.collect()
    assert f.freed == [1] and twin.shape == again.shape == (5,)


@pytest.mark.gpu
def test_views_beside_the_map(_gpu):
    """What a tensor made from the descriptor's addresses reads after the CoarseGraph is gone, with other calls and
    allocations between; then the memory goes back without a further call."""
    import torch

    import graphgen as gg
    import oracle as O
    live = {}
    alloc_t = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)
    free_t = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)

    @alloc_t
    def alloc(nbytes, stream, ctx):
        p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)
        live[p] = int(nbytes)
        return p

    @free_t
    def free(ptr, nbytes, stream, ctx):
        if ptr:
            del live[ptr]
            torch.cuda.caching_allocator_delete(ptr)

    g = gg.grid(1600, 1600)
    lab = np.arange(g.n, dtype=np.int32)  # (a coarse graph as large as the fine one: 76 MB of edge weights)
    lab[1::7] -= 1
    co, _ = O.contract(g, lab)
    dg, dlab = gp.DeviceGraph.from_host(g), torch.from_numpy(lab).cuda()
    other = torch.zeros(g.n, dtype=torch.int32, device="cuda")
    gp.lib().gp_set_allocator(ctypes.cast(alloc, ctypes.c_void_p), ctypes.cast(free, ctypes.c_void_p), None)
    try:
        cg, f2c = gp.contract(dg, dlab)
        adj, ew = (gp._wrap(p, cg.m_dir, t) for p, t in ((cg.desc.adj, "<i4"), (cg.desc.ewgt, "<i8")))
        del cg
        o, of = gp.contract(dg, other)
        o.free()
        noise = [torch.full((co.adj.size,), -1, dtype=torch.int64, device="cuda") for _ in range(4)]
        assert np.array_equal(adj.cpu().numpy(), co.adj) and np.array_equal(ew.cpu().numpy(), co.ew)
        torch.cuda.synchronize()
        del noise, o, of
        assert max(live.values()) >= 8 * co.adj.size
        del f2c
        assert max(live.values(), default=0) < 8 * co.adj.size  # (smaller blocks are kept for reuse)
        gp.free_cached()
        assert not live
    finally:
        gp.free_cached()
        gp._install_torch_allocator(gp.lib())


@pytest.fixture(scope="module")
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    gp.build()

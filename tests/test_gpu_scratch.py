"""Scratch of the solves: only what the call uses, and solves near a limit run without the
restriction to reached rows instead of being refused."""
import ctypes
import os

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_06384_gb300 import kb as _kb
    if not os.path.exists(_kb.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    return _kb


@pytest.fixture(scope="module")
def graph():
    return synth.grid_graph((2000, 2000))


def _restricted(kb, G, method, M, m, **kw):
    """(bytes, bytes under no_frontier = 1)"""
    return [kb.kb_workspace_bytes(G, method, "exp", kb.make_params(t=0.1, no_frontier=nf, **kw), M, m) for nf in (0, 1)]


# bytes of the plans before the tile lists of all steps, on 152 SMs
@pytest.mark.parametrize("n,method,phi,M,m,kw,most", [
    (2000, "cheb", "exp", 1, 3, {}, 395008),
    (2000, "sbl", "exp", 1, 3, {}, 598528),
    (2000, "cbl", "spline", 4, 6, dict(s=1.5), 1516288),
    (20000, "cheb", "exp", 16, 300, {}, 3945728),
    (20000, "cbl", "exp", 33, 20, {}, 121915392),
    (20000, "cbl", "exp", 72, 20, {}, 253943552),
    (20000, "cbl", "exp", 112, 20, {}, 265778432),
    (20000, "cbl", "exp", 4, 40, dict(tol=1e-6, reorth=2), 53355264),
    (20000, "cbl", "spline", 64, 40, dict(tol=1e-6, reorth=2), 238324480),
])
def test_small_solves_take_no_more_than_they_use(kb, n, method, phi, M, m, kw, most):
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the recorded sizes are of 152 SMs")
    kw = dict(kw)
    p = kb.make_params(t=1.0, eps=0.5, s=kw.pop("s", 1.0), **kw)
    with kb.Graph.from_csr(synth.cycle_graph(n)) as G:
        assert kb.kb_workspace_bytes(G, method, phi, p, M, m) <= most


def test_server_takes_a_request_that_fits_without_the_restriction(kb, graph):
    import torch
    nodes = synth.sample_nodes(graph.n, 3, seed=1)
    with kb.Graph.from_csr(graph) as G:
        full, less = _restricted(kb, G, "cheb", 3, 60)
        assert less < full
        want = kb.kernel_columns(G, "cheb", "exp", nodes, 60, t=0.1, no_frontier=1)
        Y = torch.zeros_like(want)
        torch.cuda.synchronize()
        with kb.Server(streams=1, memory_budget=less) as sv:
            info, _ = sv.poll(sv.submit(G, "cheb", "exp", kb.make_params(t=0.1), nodes, 60, Y), -1)
            assert info["status"] == 0
        with kb.Server(streams=1, memory_budget=less - 1) as sv:
            with pytest.raises(kb.KbError) as e:
                sv.submit(G, "cheb", "exp", kb.make_params(t=0.1), nodes, 60, Y)
            assert kb.STATUS[e.value.code] == "KB_ERR_NOMEM"
        assert torch.equal(Y, want)


class PoolProps(ctypes.Structure):   # CUmemPoolProps
    _fields_ = [("allocType", ctypes.c_int), ("handleTypes", ctypes.c_int), ("locationType", ctypes.c_int),
                ("locationId", ctypes.c_int), ("win32", ctypes.c_void_p), ("maxSize", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


@pytest.mark.parametrize("method", ["cheb", "gbl"])
def test_full_pool_runs_without_the_restriction(kb, graph, method):
    """The device's pool holds what a solve on all rows takes, and not the tile lists as well."""
    import torch
    nodes = synth.sample_nodes(graph.n, 2, seed=2)
    cu = ctypes.CDLL("libcuda.so.1")
    dev, old, pool = torch.cuda.current_device(), ctypes.c_void_p(), ctypes.c_void_p()
    with kb.Graph.from_csr(graph) as G:
        kw = dict(two_pass=1) if method == "gbl" else {}
        full, less = _restricted(kb, G, method, 2, 250, **kw)
        slack = 64 << 20   # (sizes of a pool are rounded)
        assert full > less + 1.5 * slack
        want = kb.kernel_columns(G, method, "exp", nodes, 250, t=0.1, no_frontier=1, **kw)
        torch.cuda.synchronize()
        assert cu.cuDeviceGetMemPool(ctypes.byref(old), dev) == 0
        props = PoolProps(allocType=1, locationType=1, locationId=dev, maxSize=less + slack // 2)
        assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
        try:
            assert cu.cuDeviceSetMemPool(dev, pool) == 0
            Y, info = kb.kernel_columns(G, method, "exp", nodes, 250, t=0.1, info=True, **kw)
            torch.cuda.synchronize()
            assert info["status"] == 0 and torch.equal(Y, want)
            with pytest.raises(kb.KbError) as e:   # and one that does not fit either way
                kb.kernel_columns(G, method, "exp", synth.sample_nodes(graph.n, 40, seed=3), 250, t=0.1, **kw)
            assert kb.STATUS[e.value.code] == "KB_ERR_NOMEM"
        finally:
            torch.cuda.synchronize()
            assert cu.cuDeviceSetMemPool(dev, old) == 0
            assert cu.cuMemPoolDestroy(pool) == 0


def test_failed_allocation_is_reported_once(kb):
    """The call after one that ran out of memory does not report that again."""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    dev, old, pool = torch.cuda.current_device(), ctypes.c_void_p(), ctypes.c_void_p()
    g = synth.grid_graph((1000, 1000))
    nodes = synth.sample_nodes(g.n, 16, seed=1)
    with kb.Graph.from_csr(g) as G:
        want = kb.kernel_columns(G, "cheb", "exp", nodes, 5, t=0.1)
        torch.cuda.synchronize()
        assert cu.cuDeviceGetMemPool(ctypes.byref(old), dev) == 0
        props = PoolProps(allocType=1, locationType=1, locationId=dev, maxSize=32 << 20)   # (three blocks take 192 MB)
        assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
        try:
            assert cu.cuDeviceSetMemPool(dev, pool) == 0
            with pytest.raises(kb.KbError) as e:
                kb.kernel_columns(G, "cheb", "exp", nodes, 5, t=0.1)
            assert kb.STATUS[e.value.code] == "KB_ERR_NOMEM"
        finally:
            torch.cuda.synchronize()
            assert cu.cuDeviceSetMemPool(dev, old) == 0
            assert cu.cuMemPoolDestroy(pool) == 0
        assert torch.equal(kb.kernel_columns(G, "cheb", "exp", nodes, 5, t=0.1), want)
    with kb.Graph.from_csr(synth.path_graph(9)):
        pass

"""Solves that run out of scratch."""
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


class PoolProps(ctypes.Structure):   # CUmemPoolProps
    _fields_ = [("allocType", ctypes.c_int), ("handleTypes", ctypes.c_int), ("locationType", ctypes.c_int),
                ("locationId", ctypes.c_int), ("win32", ctypes.c_void_p), ("maxSize", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


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

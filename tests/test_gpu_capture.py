"""Solves recorded in a CUDA graph (stream capture): the launches that a captured stream treats
differently (side stream of the spline factors, cooperative, cluster and dependent launches) give
what the direct call gives, at every replay."""
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


@pytest.fixture(scope="module", params=[3000, 70003])   # all rows; restricted to the reached rows at M = 64
def graph(request):
    return synth.random_geometric_graph(request.param, 10, seed=3)


@pytest.mark.parametrize("method,M,kw", [
    ("cbl", 64, dict(phi="exp", t=0.7)),
    ("cbl", 64, dict(phi="spline", eps=0.5, s=1.0)),
    ("cbl", 64, dict(phi="spline", eps=0.5, s=2.5)),
    ("cbl", 64, dict(phi="spline", eps=0.5, s=1.0, tol=1e-3, reorth=2)),
    ("cbl", 20, dict(phi="exp", t=0.7, reorth=1)),
    ("cbl", 33, dict(phi="exp", t=0.7, basis="f64")),
    ("cbl", 64, dict(phi="exp", t=0.7, two_pass=1, basis="bf16")),
    ("gbl", 64, dict(phi="exp", t=0.7)),
    ("sbl", 64, dict(phi="spline", eps=0.5, s=1.5)),
    ("cheb", 64, dict(phi="exp", t=0.7)),
    ("cheb2", 140, dict(phi="exp", t=0.7)),
])
def test_recorded_solve(kb, graph, method, M, kw):
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    kw = dict(kw)
    phi = kw.pop("phi")
    m = 9
    lab_deg = np.diff(graph.rowptr)
    nodes = np.random.default_rng(4).choice(np.nonzero(lab_deg > 6)[0], size=M, replace=False).astype(np.int32)
    p = kb.make_params(**kw)
    s = torch.cuda.Stream()
    vp = ctypes.c_void_p
    with kb.Graph.from_csr(graph) as G:
        want = torch.empty(graph.n, M, device="cuda")
        Y = torch.zeros(graph.n, M, device="cuda")
        torch.cuda.synchronize()
        kb.kb_krylov_apply(G, method, phi, p, nodes, M, m, want, stream=s)
        s.synchronize()
        cg, ge = vp(), vp()
        assert cu.cuStreamBeginCapture_v2(vp(s.cuda_stream), 1) == 0   # (thread-local mode)
        try:
            kb.kb_krylov_apply(G, method, phi, p, nodes, M, m, Y, stream=s)
        finally:
            rc = cu.cuStreamEndCapture(vp(s.cuda_stream), ctypes.byref(cg))
        assert rc == 0
        assert not Y.any()   # recorded, not run
        assert cu.cuGraphInstantiateWithFlags(ctypes.byref(ge), cg, ctypes.c_ulonglong(0)) == 0
        try:
            for _ in range(2):
                Y.zero_()
                torch.cuda.synchronize()
                assert cu.cuGraphLaunch(ge, vp(s.cuda_stream)) == 0
                s.synchronize()
                assert bool(torch.isfinite(want).all()) and torch.equal(Y, want)
        finally:
            assert cu.cuGraphExecDestroy(ge) == 0 and cu.cuGraphDestroy(cg) == 0

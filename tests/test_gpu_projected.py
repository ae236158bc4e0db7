"""The projected problem of cbl at the edges of its launch rules: the series of e^{-tH} in one
launch with one, two and four items per CTA, term by term and in several chunks of
coefficients, and the spline factors kept across the checks of the stopping rule, with
processes that end before, at and between checks."""
import numpy as np
import pytest

import synth
from oracle import dense

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24


@pytest.fixture(scope="module")
def kb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import os
    from paper_2301_06384_gb300 import kb as _kb
    if not os.path.exists(_kb.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    return _kb


# items of a series = m ceil(M / 8): one, two, four per CTA, or a launch per term above that.
# The Lanczos error at these t is below 1e-9, so the exact kernel is the reference; FP32 bar
# max(1e-6, t Lambda u) = 1e-6
@pytest.mark.parametrize("m,t", [(6, 0.02), (16, 0.5), (32, 0.5), (48, 0.5)])
@pytest.mark.parametrize("M", [97, 128])
def test_series_launches(kb, M, m, t):
    g = synth.grid_graph((128, 128))
    nodes = synth.sample_nodes(g.n, M, seed=M)
    with kb.Graph.from_csr(g) as G:
        Y, info = kb.kernel_columns(G, "cbl", "exp", nodes, m, info=True, t=t, reorth=2)
    ref = dense.grid_exp_columns((128, 128), nodes, t)
    assert info["steps_done"] == m
    assert np.linalg.norm(Y.cpu().numpy() - ref) / np.linalg.norm(ref) < 1e-6


def test_series_in_chunks(kb):
    # more terms than one launch takes coefficients (440); the FP64 mode runs term by term
    g = synth.grid_graph((128, 128))
    nodes = synth.sample_nodes(g.n, 16, seed=3)
    t = 800.0
    assert len(kb.kb_exp_series_coeffs(t, 8.0)) > 440
    with kb.Graph.from_csr(g) as G:
        Y, Y64 = [kb.kernel_columns(G, "cbl", "exp", nodes, 20, t=t, basis=b).double() for b in ("f32", "f64")]
    assert float((Y - Y64).norm() / Y64.norm()) < t * 8.0 * U32


# path of n nodes, start at its centre: the invariant space has (n + 1) / 2 dimensions (stops
# by itself at step 4, 8, 11, 12 or 20: before, at and between checks)
@pytest.mark.parametrize("n", [7, 15, 21, 23, 39])
@pytest.mark.parametrize("phi,kw", [("spline", dict(eps=0.5, s=1.0)), ("spline", dict(eps=0.5, s=2.0)),
                                    ("spline", dict(eps=0.5, s=2.5)), ("exp", dict(t=1.0))])
def test_process_ends_by_itself_between_checks(kb, n, phi, kw):
    import torch
    g = synth.path_graph(n)
    nodes = np.array([n // 2], np.int32)
    with kb.Graph.from_csr(g) as G:
        Y, info = kb.kernel_columns(G, "cbl", phi, nodes, n, info=True, tol=1e-300, basis="f64", **kw)
        Yn = kb.kernel_columns(G, "cbl", phi, nodes, n, tol=1e-300, basis="f64", **kw)   # enqueues all steps
        torch.cuda.synchronize()
    assert info["steps_done"] == (n + 1) // 2
    assert torch.equal(Y, Yn)
    ref = dense.kernel_columns(dense.laplacian_dense(g.n, g.rowptr, g.col, g.val), nodes, dense.phi_function(phi, **kw))
    assert np.linalg.norm(Y.cpu().numpy() - ref) / np.linalg.norm(ref) < 2 * U32


# the stopping rule with and without info (which lets the host stop enqueueing) and the call
# with m = the stopping step give the same bits
@pytest.mark.parametrize("tol", [1e-2, 1e-5, 1e-300])
@pytest.mark.parametrize("phi,kw", [("spline", dict(eps=0.3, s=1.0)), ("spline", dict(eps=0.3, s=2.0)),
                                    ("exp", dict(t=2.0))])
def test_stopped_process_with_and_without_info(kb, tol, phi, kw):
    import torch
    g = synth.random_geometric_graph(20000, 10, seed=1)
    nodes = synth.sample_nodes(g.n, 16, seed=21)
    with kb.Graph.from_csr(g) as G:
        Y, info = kb.kernel_columns(G, "cbl", phi, nodes, 40, info=True, tol=tol, reorth=2, **kw)
        Yn = kb.kernel_columns(G, "cbl", phi, nodes, 40, tol=tol, reorth=2, **kw)
        Yf = kb.kernel_columns(G, "cbl", phi, nodes, info["steps_done"], reorth=2, **kw)
        torch.cuda.synchronize()
    assert info["spmm_launches"] == 40
    assert torch.equal(Y, Yn)
    assert torch.equal(Y, Yf)

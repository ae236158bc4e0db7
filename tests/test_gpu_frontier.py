"""The restriction to reached rows on blocks large enough that the library chooses it (16 MiB
and more): all methods and storage types against the all-rows run and the FP64 oracle, the
replayed second pass and the tensor-core products."""
import numpy as np
import pytest

import synth
from oracle import krylov

pytestmark = pytest.mark.gpu

N1, N2 = 60001, 10007   # reached component, component without a node (both end inside a tile)
M_STEPS = 12


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


@pytest.fixture(scope="module")
def case():
    from scipy.sparse.csgraph import connected_components
    parts = [synth.random_geometric_graph(N1, 10, seed=61), synth.random_geometric_graph(N2, 10, seed=62)]
    src, dst = [], []
    for g, off in zip(parts, (0, N1)):
        r = np.repeat(np.arange(g.n), np.diff(g.rowptr))
        keep = r < g.col
        src.append(r[keep] + off)
        dst.append(g.col[keep] + off)
    g = synth.from_edges(N1 + N2, np.concatenate(src), np.concatenate(dst))
    L = krylov.laplacian(g.n, g.rowptr, g.col, g.val)
    lab = connected_components(L)[1][:N1]
    big = np.nonzero(lab == np.bincount(lab).argmax())[0]
    return g, L, np.random.default_rng(7).choice(big, size=128, replace=False).astype(np.int32)


def _pair(kb, case, method, M, **kw):
    import torch
    g, L, nodes = case
    with kb.Graph.from_csr(g) as G:
        Y = [kb.kernel_columns(G, method, "exp", nodes[:M], M_STEPS, t=1.0, no_frontier=nf, **kw) for nf in (0, 1)]
        torch.cuda.synchronize()
    return [y.cpu().numpy().astype(np.float64) for y in Y]


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("method", ["cbl", "gbl", "sbl", "cheb", "cheb2"])
@pytest.mark.parametrize("M,basis", [(64, "f32"), (33, "f32"), (97, "f32"), (33, "bf16"), (5, "f64"), (33, "f64")])
def test_restricted_matches_all_rows(kb, case, method, M, basis):
    Yf, Ya = _pair(kb, case, method, M, basis=basis)
    assert np.all(Yf[N1:] == 0.0)
    if method in ("cheb", "cheb2"):
        assert np.array_equal(Yf, Ya)   # the same row arithmetic
    # sums in another order: FP32 rounding of the sums, of Y (FP64), or two runs each within
    # the bfloat16 mode's error 2e-2 of the exact result
    assert _rel(Yf, Ya) < {"f32": 1e-6, "f64": 2.0 ** -23, "bf16": 4e-2}[basis]
    if M != 33:
        return
    ref = krylov.apply(method, case[1], case[2][:M], M_STEPS, "exp", t=1.0).Y
    # (largest degree about 25: t Lambda u = 50 * 2^-24 = 3e-6 in FP32)
    assert _rel(Yf, ref) < {"f32": 3e-6, "f64": 2.0 ** -23, "bf16": 2e-2}[basis]


@pytest.mark.parametrize("method,kw", [("gbl", {}), ("sbl", {}), ("cbl", {}), ("cbl", dict(reorth=2))])
def test_second_pass_repeats_restricted_run(kb, case, method, kw):
    import torch
    g, _, nodes = case
    with kb.Graph.from_csr(g) as G:
        Y1, Y2 = [kb.kernel_columns(G, method, "exp", nodes[:64], M_STEPS, t=1.0, two_pass=tp, **kw) for tp in (0, 1)]
        torch.cuda.synchronize()
    assert torch.equal(Y1, Y2)


def test_tensor_core_products_on_listed_tiles(kb, case, monkeypatch):
    import torch
    g, L, nodes = case
    monkeypatch.setenv("KB_TENSOR_CORES", "1")
    with kb.Graph.from_csr(g) as G:
        Y1, Y2 = [kb.kernel_columns(G, "cbl", "exp", nodes[:64], M_STEPS, t=1.0, two_pass=tp) for tp in (0, 1)]
        torch.cuda.synchronize()
    assert torch.equal(Y1, Y2)
    ref = krylov.apply("cbl", L, nodes[:64], M_STEPS, "exp", t=1.0).Y
    assert _rel(Y1.cpu().numpy().astype(np.float64), ref) < 3e-6

"""Tall-skinny block kernels at the edges of their tiles: ragged widths and row counts, on
graphs large enough for the full-height tiles and small enough for the low ones, against the
FP64 oracle."""
import numpy as np
import pytest

import synth
from oracle import krylov

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


@pytest.fixture(scope="module")
def graphs():
    # 40961 rows: above 152 tiles of the tallest kind (256 rows), the last 32-row tile has one
    # row; 2025 rows: the low tiles, nine rows in the last one
    return {40961: synth.random_geometric_graph(40961, 10, seed=40961), 2025: synth.grid_graph((45, 45))}


@pytest.mark.parametrize("n", [40961, 2025])
@pytest.mark.parametrize("M", [3, 16, 21, 40, 64, 97, 128])
@pytest.mark.parametrize("kw", [dict(), dict(no_frontier=1), dict(reorth=1), dict(reorth=2), dict(basis="f64")],
                         ids=["plain", "all_rows", "full_reorth", "local_reorth", "f64"])
def test_cbl_edges(kb, graphs, n, M, kw):
    import torch
    f64 = kw.get("basis") == "f64"
    if f64 and M > 64:
        pytest.skip("FP64 blocks are at most 64 wide")
    g = graphs[n]
    # (a block with an isolated node is rank deficient)
    nodes = np.random.default_rng(M).choice(np.nonzero(np.diff(g.rowptr) >= 4)[0], size=M, replace=False).astype(np.int32)
    with kb.Graph.from_csr(g) as G:
        lam = G.lambda_max
        Y, info = kb.kernel_columns(G, "cbl", "exp", nodes, 6, info=True, t=0.5, **kw)
        torch.cuda.synchronize()
    assert info["steps_done"] == 6
    ref = krylov.apply("cbl", krylov.laplacian(g.n, g.rowptr, g.col, g.val), nodes, 6, "exp", t=0.5).Y
    err = np.linalg.norm(Y.cpu().numpy().astype(np.float64) - ref) / np.linalg.norm(ref)
    # FP64: the FP32 rounding of Y; FP32: 1e-6 or the first-order change t Lambda u of phi
    assert err < (2 * U32 if f64 else max(1e-6, 0.5 * lam * U32)), err

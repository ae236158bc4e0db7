"""Long rows (hubs) of the SpMM: the rule that lists them, and products on rows around its line and
around the rounds of a CTA's lane groups, against the FP64 oracle."""
import ctypes
import os

import numpy as np
import pytest

import synth
from oracle import krylov


@pytest.fixture(scope="module")
def kb():
    from paper_2301_06384_gb300 import kb as _kb
    if not os.path.exists(_kb.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    _kb.lib()
    return _kb


@pytest.mark.parametrize("degrees,line", [
    ([0], 64), ([0] * 100, 64), ([10] * 1000, 64), ([100] * 1000, 400),
    ([10] * 9999 + [9999], 64),                       # a star among others
    ([5] * 19000 + [105] * 1000, 128),                # one row in 20: too many
    ([5] * 19700 + [105] * 300, 64),                  # one in 66
    ([3] * 10 + [70, 600], 233),                      # small: one long row at most (4 * 700 / 12)
])
def test_rule_lists_few_rows(kb, degrees, line):
    f = ctypes.CDLL(kb.LIB_PATH)["_ZN2kb15long_row_degreeEPKilPSt6vectorIiSaIiEE"]
    f.restype, f.argtypes = ctypes.c_int32, [ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p]
    ptr = np.concatenate([[0], np.cumsum(degrees)]).astype(np.int32)
    rows = (ctypes.c_void_p * 3)()   # an empty std::vector<int32_t>
    assert f(ptr.ctypes.data, len(degrees), ctypes.addressof(rows)) == line
    count = ((rows[1] or 0) - (rows[0] or 0)) // 4
    got = list((ctypes.c_int32 * count).from_address(rows[0])) if count else []
    assert got == [i for i, d in enumerate(degrees) if d > line]
    assert count <= max(1, len(degrees) // 64)


# rows of the hubs: the line itself (64: an ordinary row) and around it; one round of the 128 groups of 4
# neighbours at W = 16, of the 16 groups at W = 128; many rounds
HUBS = [63, 64, 65, 68, 127, 128, 129, 511, 512, 513, 1000, 2049, 15001]


@pytest.fixture(scope="module")
def hubs():
    """A grid with hubs at rows 0, 1, ... (one unit of a warp) and at the last rows; weights too."""
    n = 70007
    rng = np.random.default_rng(5)
    at = list(range(len(HUBS))) + [n - 1 - i for i in range(len(HUBS))]
    body = np.arange(len(HUBS), n - len(HUBS))
    src, dst = [body[:-1], body[:-300]], [body[1:], body[300:]]   # (not beyond the body: hubs keep their degree)
    for h, d in zip(at, HUBS + HUBS):
        src.append(np.full(d, h))
        dst.append(rng.choice(body, size=d, replace=False))
    src, dst = np.concatenate(src), np.concatenate(dst)
    out = {}
    for w in (None, rng.uniform(0.5, 1.5, src.size).astype(np.float32)):
        g = synth.from_edges(n, src, dst, w)
        out[w is not None] = (g, krylov.laplacian(g.n, g.rowptr, g.col, g.val))
    nodes = np.concatenate([at, rng.choice(body, size=128 - len(at), replace=False)]).astype(np.int32)
    return out, nodes[np.random.default_rng(1).permutation(128)]


STEPS = 4


@pytest.mark.gpu
@pytest.mark.parametrize("method", ["cheb", "sbl"])   # without and with column dots
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("M,basis", [(1, "f32"), (16, "f32"), (29, "f32"), (64, "f32"), (101, "f32"), (13, "f64"), (64, "f64"),
                                     (16, "bf16"), (128, "bf16")])
def test_products_on_long_rows(kb, hubs, method, weighted, M, basis):
    import torch
    graphs, nodes = hubs
    g, L = graphs[weighted]
    t = 1e-4   # t Lambda about 3
    with kb.Graph.from_csr(g) as G:
        Y = [kb.kernel_columns(G, method, "exp", nodes[:M], STEPS, t=t, basis=basis, no_frontier=nf) for nf in (0, 1, 1)]
        torch.cuda.synchronize()
    assert torch.equal(Y[1], Y[2])
    if method == "cheb":
        assert torch.equal(Y[0], Y[1])   # the same row arithmetic
    ref = krylov.apply(method, L, nodes[:M], STEPS, "exp", t=t).Y
    # four products; the longest chain of a sum in FP32 is 15001 / 16 terms and 13 to combine
    # them, its rounding a random walk; FP64 results are rounded to FP32; bfloat16 blocks: the
    # mode's error
    tol = {"f32": STEPS * ((15001 / 16 + 13) ** 0.5) * 2.0 ** -24, "f64": 2.0 ** -23, "bf16": 2e-2}[basis]
    for y in Y:
        y = y.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(y - ref) / np.linalg.norm(ref) < tol

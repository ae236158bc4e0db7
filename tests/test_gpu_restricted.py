"""The restriction to reached rows at sizes where the library chooses it, over the forms that its
kernels take: all block widths, column groups, edge weights and diagonal excess, hubs, the normalized
Laplacian, the spline kernel, the stopping rule, reorthogonalisation and the second pass."""
import os

import numpy as np
import pytest

import synth
from oracle import krylov

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
STEPS = 10


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


class Case:
    """A graph with a component that no node reaches; its Laplacian; nodes in the other one."""

    def __init__(self, kind, n):
        rng = np.random.default_rng(n)
        if kind == "hubs":
            body = synth.barabasi_albert_graph(n - 500, 4, seed=2)
        else:
            body = synth.random_geometric_graph(n - 500, 10, seed=2)
        rest = synth.grid_graph((20, 25))
        src, dst = [], []
        for g, off in ((body, 0), (rest, n - 500)):
            r = np.repeat(np.arange(g.n), np.diff(g.rowptr))
            keep = r < g.col
            src.append(r[keep] + off)
            dst.append(g.col[keep] + off)
        src, dst = np.concatenate(src), np.concatenate(dst)
        w = rng.uniform(0.5, 1.5, src.size).astype(np.float32) if kind in ("weights", "hubs") else None
        self.g = g = synth.from_edges(n, src, dst, w)
        self.flags = 0
        if kind == "weights":   # generalized: more on the diagonal than the row sums
            d = np.nonzero(np.repeat(np.arange(n), np.diff(g.rowptr)) == g.col)[0]
            g.val[d] += rng.uniform(0.0, 2.0, n).astype(np.float32)
        self.L = krylov.laplacian(g.n, g.rowptr, g.col, g.val)
        self.lam = float(abs(self.L).sum(1).max())
        cut = n - 500
        deg = np.diff(self.L.indptr)[:cut]
        if kind == "hubs":
            self.nodes = rng.choice(np.nonzero(deg <= 8)[0], size=150, replace=False)
        else:
            from scipy.sparse.csgraph import connected_components
            lab = connected_components(self.L)[1][:cut]
            self.nodes = rng.choice(np.nonzero(lab == np.bincount(lab).argmax())[0], size=150, replace=False)
        self.nodes = self.nodes.astype(np.int32)
        self.cut = cut

    def solve(self, kb, method, phi, M, nf, info=False, m=STEPS, **kw):
        import torch
        with kb.Graph.from_csr(self.g) as G:
            if not nf:
                # the restriction is on: it takes scratch of its own
                a, b = [kb.kb_workspace_bytes(G, method, phi, kb.make_params(no_frontier=x, **kw), M, m) for x in (0, 1)]
                assert a > b
            r = kb.kernel_columns(G, method, phi, self.nodes[:M], m, no_frontier=nf, info=info, **kw)
            torch.cuda.synchronize()
        return (r[0].cpu().numpy().astype(np.float64), r[1]) if info else r.cpu().numpy().astype(np.float64)


    def twins(self, M):
        """Whether two of the nodes have the same neighbours and weights: L (e_a - e_b) is a multiple of
        e_a - e_b, so the second block of cbl is rank deficient."""
        L, seen = self.L, set()
        for v in self.nodes[:M]:
            cols, vals = L.indices[L.indptr[v]:L.indptr[v + 1]], L.data[L.indptr[v]:L.indptr[v + 1]]
            # (adjacent twins: the node itself counts among its neighbours)
            rows = [frozenset((c, x) for c, x in zip(cols, vals) if c != v), frozenset((c, 0.0) for c in cols)]
            if self.g.unit_weight and any(r in seen for r in rows):
                return True
            seen.update(rows)
        return False


CASES = {}


def case(kind, n):
    if (kind, n) not in CASES:
        CASES[kind, n] = Case(kind, n)
    return CASES[kind, n]


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# rows: 16 MiB in FP32 blocks of the width (16, 32, 64, 128 columns), and a part of a tile
SIZES = {5: 262144 + 7, 24: 131072 + 9, 50: 65536 + 15, 100: 32768 + 3}


@pytest.mark.parametrize("method", ["cbl", "gbl", "sbl", "cheb", "cheb2"])
@pytest.mark.parametrize("M", [5, 24, 50, 100])
@pytest.mark.parametrize("kind", ["plain", "weights"])
def test_widths(kb, method, M, kind):
    c = case(kind, SIZES[M])
    t = 1.0 if kind == "plain" else 0.5
    Yr, Ya = [c.solve(kb, method, "exp", M, nf, t=t) for nf in (0, 1)]
    if method in ("cheb", "cheb2"):
        assert np.array_equal(Yr, Ya)   # the same row arithmetic
        assert np.all(Yr[c.cut:] == 0.0)
    if method == "cbl" and c.twins(M):
        assert np.all(np.isnan(Yr)) and np.all(np.isnan(Ya))   # a breakdown either way
        with pytest.raises(krylov.Breakdown):
            krylov.apply(method, c.L, c.nodes[:M], STEPS, "exp", t=t)
        return
    tol = t * c.lam * U   # as the exponential's argument rounds in FP32
    assert rel(Yr, Ya) < tol
    if M in (5, 24):
        assert rel(Yr, krylov.apply(method, c.L, c.nodes[:M], STEPS, "exp", t=t).Y) < tol


@pytest.mark.parametrize("method", ["cheb", "sbl", "cheb2"])
@pytest.mark.parametrize("kind,n", [("plain", 40003), ("hubs", 40003)])
def test_column_groups(kb, method, kind, n):
    """128 and 22 columns: the second group runs in narrower rows of the same blocks."""
    c = case(kind, n)
    t = 1.0 if kind == "plain" else 2.0 / c.lam
    Yr, Ya = [c.solve(kb, method, "exp", 150, nf, t=t) for nf in (0, 1)]
    if method != "sbl":
        assert np.array_equal(Yr, Ya)
    # (short time: the rounding of the products, whose hub rows sum some 2000 terms in 16 chains or more)
    tol = t * c.lam * U if kind == "plain" else STEPS * ((2000 / 16) ** 0.5 + 5) * U
    assert rel(Yr, Ya) < tol
    assert rel(Yr, krylov.apply(method, c.L, c.nodes[:150], STEPS, "exp", t=t).Y) < tol


@pytest.mark.parametrize("method", ["cbl", "gbl", "sbl"])
@pytest.mark.parametrize("s", [1.0, 1.5])
@pytest.mark.parametrize("M", [24, 50])
def test_spline_kernel(kb, method, s, M):
    c = case("weights", SIZES[M])
    Yr, Ya = [c.solve(kb, method, "spline", M, nf, eps=0.5, s=s) for nf in (0, 1)]
    tol = s * (c.lam + 0.5) / 0.5 * U   # the condition number of the kernel's argument
    assert rel(Yr, Ya) < tol
    assert rel(Yr, krylov.apply(method, c.L, c.nodes[:M], STEPS, "spline", eps=0.5, s=s).Y) < tol


@pytest.mark.parametrize("phi,kw", [("exp", dict(t=1.0)), ("spline", dict(eps=2.0, s=1.0))])
@pytest.mark.parametrize("reorth", [0, 2])
@pytest.mark.parametrize("M", [24, 50])
def test_stopping_rule(kb, phi, kw, reorth, M):
    c = case("plain", SIZES[M])
    (Yr, ir), (Ya, ia) = [c.solve(kb, "cbl", phi, M, nf, info=True, m=60, tol=1e-4, reorth=reorth, **kw) for nf in (0, 1)]
    assert ir["steps_done"] < 60 and ia["steps_done"] < 60
    tol = (c.lam if phi == "exp" else (c.lam + 2.0) / 2.0) * U
    if ir["steps_done"] == ia["steps_done"]:
        assert abs(ir["est_change"] - ia["est_change"]) < 2 * tol
        assert rel(Yr, Ya) < tol
    else:   # a change at the threshold falls on either side of it with the rounding
        assert rel(Yr, Ya) < 2e-4


@pytest.mark.parametrize("reorth", [1, 2])
@pytest.mark.parametrize("M", [5, 24, 50, 100])
def test_reorthogonalised(kb, reorth, M):
    c = case("weights", SIZES[M])
    Yr = c.solve(kb, "cbl", "exp", M, 0, t=0.5, reorth=reorth)
    tol = 0.5 * c.lam * U
    assert rel(Yr, c.solve(kb, "cbl", "exp", M, 1, t=0.5, reorth=reorth)) < tol
    if M == 24:
        assert rel(Yr, krylov.apply("cbl", c.L, c.nodes[:M], STEPS, "exp", t=0.5, reorth=reorth == 1).Y) < tol


@pytest.mark.parametrize("method,kw", [("gbl", {}), ("sbl", {}), ("cbl", {}), ("cbl", dict(reorth=2))])
@pytest.mark.parametrize("M", [5, 24])
def test_second_pass(kb, method, kw, M):
    c = case("weights", SIZES[M])
    Y1, Y2 = [c.solve(kb, method, "exp", M, 0, t=0.5, two_pass=tp, **kw) for tp in (0, 1)]
    assert np.array_equal(Y1, Y2)


@pytest.mark.parametrize("method", ["cbl", "gbl", "sbl", "cheb"])
def test_normalized_laplacian(kb, method):
    import torch
    c = case("plain", SIZES[50])
    Y = []
    with kb.Graph.from_csr(c.g, flags=kb.KB_GRAPH_NORMALIZED) as G:
        for nf in (0, 1):
            Y.append(kb.kernel_columns(G, method, "exp", c.nodes[:50], STEPS, t=3.0, no_frontier=nf).cpu().numpy().astype(np.float64))
        a, b = [kb.kb_workspace_bytes(G, method, "exp", kb.make_params(t=3.0, no_frontier=x), 50, STEPS) for x in (0, 1)]
        torch.cuda.synchronize()
    assert a > b
    if method == "cheb":
        assert np.array_equal(Y[0], Y[1])
    assert rel(Y[0], Y[1]) < 3.0 * 2.0 * U * STEPS   # Lambda <= 2; the rounding of the steps

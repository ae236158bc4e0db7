"""Performance cases: kernel-column solves, serving and the RLS predictor through the public API.

A case is a dict of plain values; prepare() builds the graph handle, the node sets and the
output buffers a program keeps, run() makes one pass, exact() gives the same outputs in 64
bits with plain torch, and work() the bytes and operations a pass cannot do without.

Graphs are made on the GPU from the seed: random geometric graphs (mean degree 10, nodes in
cell-sorted order), 2-D and 3-D grids, and preferential-attachment graphs with weights in
[0.5, 1.5].  Nodes are drawn among those of degree >= 3, as a program samples nodes of the
graph proper and not of its isolated crumbs.
"""
import math

import numpy as np
import torch

from paper_2301_06384_gb300 import kb

DEV = "cuda"


# ---------------------------------------------------------------------- the cases
def _case(name, entry, graph, n, method, M, m, **kw):
    c = {"name": name, "entry": entry, "graph": graph, "n": n, "method": method, "M": M, "m": m,
         "phi": "exp", "t": 1.0, "eps": 0.0, "s": 0.0, "basis": "f32", "reorth": 0, "tol": 0.0,
         "requests": 1}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: 32 x 32 grid, latency and launches
        _case("grid32-cbl", "apply", "grid2", 1024, "cbl", 16, 20),
        # a small call of an odd width from a program that may not allocate
        _case("rgg2e4-cheb-fixed", "fixed", "rgg", 20000, "cheb", 37, 30),
        # a small learning task: predictor from 40 labels
        _case("rgg2e4-rls", "rls", "rgg", 20000, "cbl", 40, 20),
        # plain FP64 solve of an odd width
        _case("rgg1e5-cbl-f64", "apply", "rgg", 100003, "cbl", 33, 20, basis="f64"),
        # the throughput workload: 10^6 nodes, 64 columns, 30 products, block, global and
        # Chebyshev methods
        _case("rgg1e6-cbl", "apply", "rgg", 1000000, "cbl", 64, 30, t=2.0),
        _case("rgg1e6-gbl", "apply", "rgg", 1000000, "gbl", 64, 30, t=0.5),
        _case("rgg1e6-cheb", "apply", "rgg", 1000000, "cheb", 64, 30, t=2.0),
        # 3-D grid of the precision sweep: widest blocks, column by column, and narrow blocks
        # with many products
        _case("grid128c-sbl", "apply", "grid3", 2097152, "sbl", 128, 20),
        _case("grid128c-cbl", "apply", "grid3", 2097152, "cbl", 32, 40),
        # power-law graph, spline kernel, widest blocks, full reorthogonalisation
        _case("ba5e5-spline-reorth", "apply", "ba", 500000, "cbl", 128, 16, phi="spline", eps=0.1,
              s=2.0, reorth=1),
        # serving: four concurrent requests of different widths under the stopping rule
        _case("serve-rgg-spline", "server", "rgg", 55392, "cbl", 64, 100, phi="spline", eps=0.1, s=1.0,
              reorth=2, tol=1e-6, requests=4),
        _case("serve-ba-exp", "server", "ba", 23535, "cbl", 48, 100, t=0.5, reorth=2, tol=1e-6, requests=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply", "reorth", "server", "server", "fixed", "rls", "f64"])
    t = round(rng.uniform(0.1, 3.0), 3)
    c = _case("", kind, "rgg", 0, "cbl", 1, 1, t=t)
    del c["name"]
    c["entry"] = "apply" if kind in ("reorth", "f64") else kind
    if kind == "apply":
        c["graph"] = rng.choice(["rgg", "rgg", "grid2", "grid3"])
        c["n"] = _log(rng, 4000, 1000000)
        c["method"] = rng.choice(["cbl", "cbl", "gbl", "sbl", "cheb", "cheb2"])
        c["M"] = _log(rng, 8, 128)
        c["m"] = rng.randint(8, 40)
        if c["method"] == "cbl":
            # the block space stays well below n
            c["m"] = max(6, min(c["m"], c["n"] // (4 * c["M"])))
        if c["method"] in ("gbl", "sbl", "cheb") and rng.random() < 0.25:
            c["phi"], c["eps"], c["s"] = "spline", round(rng.uniform(0.5, 2.0), 3), rng.choice([0.5, 1.0, 1.5, 2.0])
    elif kind == "reorth":
        c["graph"], c["n"], c["M"], c["m"] = "ba", _log(rng, 20000, 400000), rng.randint(32, 128), rng.randint(8, 14)
        c["phi"], c["eps"], c["s"], c["reorth"] = "spline", round(rng.uniform(0.2, 1.0), 3), rng.choice([1.0, 2.0]), 1
    elif kind == "server":
        c["graph"] = rng.choice(["rgg", "ba"])
        c["n"], c["M"], c["m"] = _log(rng, 10000, 60000), rng.randint(16, 64), 100
        c["reorth"], c["tol"], c["requests"] = 2, 1e-6, rng.randint(2, 4)
        if c["graph"] == "ba":
            c["t"] = round(rng.uniform(0.1, 0.6), 3)
        elif rng.random() < 0.5:
            c["phi"], c["eps"], c["s"] = "spline", round(rng.uniform(0.1, 1.0), 3), 1.0
    elif kind == "fixed":
        c["n"], c["method"], c["M"], c["m"] = _log(rng, 1000, 20000), "cheb", rng.randint(1, 64), rng.randint(8, 60)
    elif kind == "rls":
        c["n"], c["M"], c["m"] = _log(rng, 10000, 100000), rng.randint(10, 100), rng.randint(10, 24)
    else:
        c["n"], c["M"], c["m"], c["basis"] = _log(rng, 10000, 100000), rng.randint(5, 40), rng.randint(8, 20), "f64"
    return c


# ---------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rgg(n, gen):
    """Random geometric graph of mean degree 10 in the unit square: CSR pattern without diagonal."""
    pts = torch.rand(n, 2, dtype=torch.float64, device=DEV, generator=gen)
    r = math.sqrt(10.0 / (math.pi * (n - 1)))
    nc = max(int(math.floor(1.0 / r)), 1)
    cxy = torch.clamp((pts * nc).long(), max=nc - 1)
    cell, order = torch.sort(cxy[:, 1] * nc + cxy[:, 0], stable=True)
    pts, cxy = pts[order], cxy[order]
    first = torch.searchsorted(cell, torch.arange(nc * nc + 1, device=DEV))
    lo, cnt = [], []
    for dy in (-1, 0, 1):
        y = cxy[:, 1] + dy
        ok = (y >= 0) & (y < nc)
        yc = y.clamp(0, nc - 1) * nc
        a = first[yc + (cxy[:, 0] - 1).clamp(min=0)]
        b = first[yc + (cxy[:, 0] + 1).clamp(max=nc - 1) + 1]
        lo.append(a)
        cnt.append(torch.where(ok, b - a, torch.zeros_like(a)))
    lo, cnt = torch.stack(lo, 1).reshape(-1), torch.stack(cnt, 1).reshape(-1)
    seg = torch.repeat_interleave(torch.arange(3 * n, device=DEV), cnt)
    j = lo[seg] + torch.arange(seg.numel(), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[seg]
    i = seg // 3
    keep = (i != j) & ((pts[i] - pts[j]).square().sum(1) < r * r)
    return i[keep], j[keep], None


def _grid(dims):
    n = math.prod(dims)
    idx = torch.arange(n, device=DEV).reshape(dims)
    src, dst = [], []
    for ax, d in enumerate(dims):
        a, b = idx.narrow(ax, 0, d - 1).reshape(-1), idx.narrow(ax, 1, d - 1).reshape(-1)
        src += [a, b]
        dst += [b, a]
    i, j = torch.cat(src), torch.cat(dst)
    key = torch.sort(i * n + j).values
    return key // n, key % n, None


def _ba(n, gen):
    """Preferential attachment, 5 edges per new node, weights uniform in [0.5, 1.5]: the far
    end of an edge is a copy of a uniformly drawn earlier end (resolved by pointer jumping);
    loops and repeated edges are dropped."""
    k, c = 5, 15   # edges per new node; edges of the seed clique on k + 1 nodes
    ci, cj = torch.triu_indices(k + 1, k + 1, 1, device=DEV)
    ne = c + (n - k - 1) * k
    e = torch.arange(ne, device=DEV)
    ptr = torch.arange(2 * ne, device=DEV)
    draw_ = (torch.rand(ne, dtype=torch.float64, device=DEV, generator=gen) * (2 * e)).long()
    ptr[1::2] = torch.where(e < c, ptr[1::2], draw_)
    while bool(((ptr % 2 == 1) & (ptr >= 2 * c)).any()):
        ptr = ptr[ptr]
    owner = torch.where(e < c, torch.zeros_like(e), (e - c) // k + k + 1)   # the edge's new node
    owner[:c] = ci
    end = ptr[1::2]
    dst = torch.where((end < 2 * c) & (end % 2 == 1), cj[(end // 2).clamp(max=c - 1)], owner[end // 2])
    src = owner
    a, b = torch.minimum(src, dst), torch.maximum(src, dst)
    key = torch.unique((a * n + b)[a != b])
    a, b = key // n, key % n
    w = torch.rand(key.numel(), dtype=torch.float32, device=DEV, generator=gen) + 0.5
    full, order = torch.sort(torch.cat([a * n + b, b * n + a]))
    return full // n, full % n, torch.cat([w, w])[order]


def _dims(case):
    n = case["n"]
    if case["graph"] == "grid2":
        a = max(2, int(round(math.sqrt(n))))
        return (a, max(2, n // a))
    a = max(2, int(round(n ** (1 / 3))))
    return (a, a, max(2, n // (a * a)))


class _Inputs:
    """Graph (edges as device tensors), node sets and labels of a case, from the seed alone."""

    def __init__(self, case, seed):
        gen = _gen(seed)
        if case["graph"] == "rgg":
            self.n = case["n"]
            self.i, self.j, self.w = _rgg(self.n, gen)
        elif case["graph"] == "ba":
            self.n = case["n"]
            self.i, self.j, self.w = _ba(self.n, gen)
        else:
            self.n = math.prod(_dims(case))
            self.i, self.j, self.w = _grid(_dims(case))
        self.deg = torch.bincount(self.i, minlength=self.n)
        rng = np.random.default_rng(seed + 17)
        cand = torch.nonzero(self.deg >= 3).reshape(-1).cpu().numpy()
        self.widths = [case["M"]]
        for q in range(1, case["requests"]):
            self.widths.append(max(1, case["M"] * (q + 1) // (case["requests"] + 1)))
        self.nodes = [rng.choice(cand, size=w, replace=False).astype(np.int32) for w in self.widths]
        self.labels = rng.choice([-1.0, 1.0], size=case["M"])

    def diag(self):
        if self.w is None:
            return self.deg.double()
        d = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        d.index_add_(0, self.i, self.w.double())
        return d.float().double()   # the matrix holds its 32-bit rounding

    def handle(self):
        flags = kb.KB_GRAPH_SKIP_SYMMETRY_CHECK
        if self.w is None:
            ptr = torch.zeros(self.n + 1, dtype=torch.int64, device=DEV)
            torch.cumsum(self.deg, 0, out=ptr[1:])
            return kb.kb_graph_create(ptr.int().cpu().numpy(), self.j.int().cpu().numpy(), None, flags)
        v = torch.arange(self.n, device=DEV)
        key, order = torch.sort(torch.cat([self.i * self.n + self.j, v * self.n + v]))
        val = torch.cat([-self.w, self.diag().float()])[order]
        ptr = torch.zeros(self.n + 1, dtype=torch.int64, device=DEV)
        torch.cumsum(self.deg + 1, 0, out=ptr[1:])
        return kb.kb_graph_create(ptr.int().cpu().numpy(), (key % self.n).int().cpu().numpy(),
                                  val.cpu().numpy(), flags)


class _Server:
    """kb.Server closed with the state that holds it."""

    def __init__(self, streams):
        self.sv = kb.Server(streams=streams)

    def __del__(self):
        self.sv.close()


def prepare(case, seed):
    x = _Inputs(case, seed)
    st = {"case": case, "graph": x.handle(), "nodes": x.nodes, "labels": x.labels,
          "params": kb.make_params(t=case["t"], eps=case["eps"] or 0.01, s=case["s"] or 1.0,
                                   reorth=case["reorth"], basis=case["basis"], tol=case["tol"]),
          "Y": [torch.empty(x.n, w, dtype=torch.float32, device=DEV) for w in x.widths]}
    if case["entry"] == "server":
        st["server"] = _Server(case["requests"])
    if case["entry"] == "rls":
        st["Y"] = [torch.empty(x.n, dtype=torch.float32, device=DEV)]
    del x
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------- one pass
GAMMA = 0.01   # regularisation of the predictor


def run(st):
    c, G, p, Y = st["case"], st["graph"], st["params"], st["Y"]
    if c["entry"] == "apply":
        kb.kb_krylov_apply(G, c["method"], c["phi"], p, st["nodes"][0], c["M"], c["m"], Y[0])
        return Y[0]
    if c["entry"] == "fixed":
        kb.kb_cheb_apply_fixed_scratch(G, c["phi"], p, st["nodes"][0], c["M"], c["m"], Y[0])
        return Y[0]
    if c["entry"] == "rls":
        coef = kb.kb_rls_predict(G, c["method"], c["phi"], p, st["nodes"][0], c["m"], st["labels"], GAMMA, Y[0])
        # formed from FP32 kernel columns: it carries 32-bit accuracy and goes on as such
        return {"y": Y[0], "c": coef.astype(np.float32)}
    sv = st["server"].sv
    tickets = [sv.submit(G, c["method"], c["phi"], p, w, c["m"], y) for w, y in zip(st["nodes"], Y)]
    for t in tickets:
        sv.poll(t, -1)
    return Y


# ---------------------------------------------------------------------- the same in 64 bits
def _laplacian64(x):
    v = torch.arange(x.n, device=DEV)
    off = torch.full_like(x.i, -1, dtype=torch.float64) if x.w is None else -x.w.double()
    key, order = torch.sort(torch.cat([x.i * x.n + x.j, v * x.n + v]))
    val = torch.cat([off, x.diag()])[order]
    ptr = torch.zeros(x.n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(x.deg + 1, 0, out=ptr[1:])
    L = torch.sparse_csr_tensor(ptr, key % x.n, val, size=(x.n, x.n))
    lam = torch.zeros(x.n, dtype=torch.float64, device=DEV)
    lam.index_add_(0, key // x.n, val.abs())
    return L, float(lam.max())


def _unit(x, nodes):
    E = torch.zeros(x.n, len(nodes), dtype=torch.float64, device=DEV)
    E[torch.from_numpy(nodes.astype(np.int64)).to(DEV), torch.arange(len(nodes), device=DEV)] = 1.0
    return E


def _phi(case, lam, root=False):
    f = 0.5 if root else 1.0
    return torch.exp(-f * case["t"] * lam) if case["phi"] == "exp" else (case["eps"] + lam) ** (-f * case["s"])


def _cheb64(case, L, lam, B, h, root=False):
    """Lobatto interpolant of degree h of phi on [0, lam], applied to B."""
    j = torch.arange(h + 1, dtype=torch.float64)
    f = _phi(case, 0.5 * lam * (1.0 - torch.cos(math.pi * j / h)), root)
    half = torch.ones(h + 1, dtype=torch.float64)
    half[0] = half[h] = 0.5
    coef = (2.0 / h) * (torch.cos(math.pi * torch.outer(j, j) / h) @ (half * f)) * half
    a, b = B, B - (2.0 / lam) * (L @ B)
    Y = float(coef[0]) * a + float(coef[1]) * b
    for k in range(2, h + 1):
        a, b = b, 2.0 * (b - (2.0 / lam) * (L @ b)) - a
        Y += float(coef[k]) * b
    return Y


def _cbl64(case, L, B):
    """Classical block Lanczos; the reduced QR by two Cholesky passes."""
    m, M = case["m"], B.shape[1]
    Q, H = [B], torch.zeros(m * M, m * M, dtype=torch.float64, device=DEV)
    for k in range(m):
        X = L @ Q[k]
        A = Q[k].T @ X
        H[k * M:(k + 1) * M, k * M:(k + 1) * M] = 0.5 * (A + A.T)
        if k == m - 1:
            break
        X -= Q[k] @ A
        if k:
            X -= Q[k - 1] @ H[(k - 1) * M:k * M, k * M:(k + 1) * M]
        if case["reorth"]:
            for P in Q:
                X -= P @ (P.T @ X)
        R = torch.eye(M, dtype=torch.float64, device=DEV)
        for _ in range(2):
            S = torch.linalg.cholesky(X.T @ X, upper=True)
            X = torch.linalg.solve_triangular(S, X, upper=True, left=False)
            R = S @ R
        Q.append(X)
        H[(k + 1) * M:(k + 2) * M, k * M:(k + 1) * M] = R
        H[k * M:(k + 1) * M, (k + 1) * M:(k + 2) * M] = R.T
    w, V = torch.linalg.eigh(H.cpu())
    U = ((V * _phi(case, w)) @ V[:M].T).to(DEV)
    return sum(Q[k] @ U[k * M:(k + 1) * M] for k in range(m))


def _scalar64(case, L, B):
    """Global or sequential Lanczos: one tridiagonal matrix, or one for each column."""
    m, M = case["m"], B.shape[1]
    glob = case["method"] == "gbl"
    dot = (lambda a, b: (a * b).sum().expand(M)) if glob else (lambda a, b: (a * b).sum(0))
    h0 = torch.sqrt(dot(B, B))
    Q, T = [B / h0], torch.zeros(M, m, m, dtype=torch.float64, device=DEV)
    for k in range(m):
        X = L @ Q[k]
        if k:
            X -= T[:, k - 1, k] * Q[k - 1]
        T[:, k, k] = dot(Q[k], X)
        if k == m - 1:
            break
        X -= T[:, k, k] * Q[k]
        T[:, k, k + 1] = T[:, k + 1, k] = torch.sqrt(dot(X, X))
        Q.append(X / T[:, k, k + 1])
    w, V = torch.linalg.eigh(T.cpu())
    u = (V @ (_phi(case, w) * V[:, 0, :]).unsqueeze(2)).squeeze(2).to(DEV)
    return sum(Q[k] * (h0 * u[:, k]) for k in range(m))


def _limit64(case, L, lam, B):
    """phi(L) B itself, which a solve under the stopping rule approximates: Chebyshev to
    convergence for the diffusion kernel, conjugate gradients for the spline kernel."""
    if case["phi"] == "exp":
        rho = 0.5 * case["t"] * lam
        return _cheb64(case, L, lam, B, int(rho + 12 * math.sqrt(rho) + 40))
    X = B
    for _ in range(int(case["s"])):
        S, R = torch.zeros_like(X), X.clone()
        P, rr = R.clone(), (R * R).sum(0)
        stop = 1e-28 * rr
        for _ in range(5000):
            AP = L @ P + case["eps"] * P
            a = rr / (P * AP).sum(0).clamp(min=1e-300)
            S += a * P
            R -= a * AP
            new = (R * R).sum(0)
            if bool((new <= stop).all()):
                break
            P, rr = R + (new / rr.clamp(min=1e-300)) * P, new
        X = S
    return X


def exact(case, seed):
    x = _Inputs(case, seed)
    L, lam = _laplacian64(x)
    out = []
    for nodes in x.nodes:
        B = _unit(x, nodes)
        if case["tol"] > 0:
            out.append(_limit64(case, L, lam, B))
        elif case["method"] == "cbl":
            out.append(_cbl64(case, L, B))
        elif case["method"] == "cheb":
            out.append(_cheb64(case, L, lam, B, case["m"]))
        elif case["method"] == "cheb2":
            h = case["m"] // 2
            out.append(_cheb64(case, L, lam, _cheb64(case, L, lam, B, h, True), h, True))
        else:
            out.append(_scalar64(case, L, B))
    if case["entry"] == "rls":
        Y, M = out[0], case["M"]
        K = Y[torch.from_numpy(x.nodes[0].astype(np.int64)).to(DEV)]
        A = K + GAMMA * M * torch.eye(M, dtype=torch.float64, device=DEV)
        c = torch.linalg.solve(A.cpu(), torch.from_numpy(x.labels).reshape(-1, 1))
        return {"y": (Y @ c.to(DEV)).reshape(-1), "c": c.reshape(-1).numpy()}
    return out if case["entry"] == "server" else out[0]


# ---------------------------------------------------------------------- the work of a pass
def work(case):
    """The graph read once, the columns written once; the products with L and, for the block
    method, its tall-skinny products, on the rows that the nodes reach."""
    n, m = case["n"], case["m"] if case["tol"] == 0 else 24
    deg = {"rgg": 10.0, "grid2": 4.0, "grid3": 6.0, "ba": 10.0}[case["graph"]]
    size = 8 if case["basis"] == "f64" else 4
    widths = [case["M"]] + [max(1, case["M"] * (q + 1) // (case["requests"] + 1)) for q in range(1, case["requests"])]

    def reach(M, k):   # rows within k hops of M nodes
        per = {"rgg": 4.0 * k * k, "grid2": 2.0 * k * k + 2 * k + 1, "grid3": 4.0 / 3.0 * k ** 3 + 2 * k * k + 1,
               "ba": 10.0 ** min(k, 8)}[case["graph"]] + 1
        return min(float(n), M * per)

    nbytes = 4.0 * n * (1 + deg * (2 if case["graph"] == "ba" else 1))
    flops = 0.0
    for M in widths:
        nbytes += 4.0 * n * (1 if case["entry"] == "rls" else M)
        rows = sum(reach(M, k) for k in range(1, m + 1))
        flops += 3.0 * deg * M * rows
        if case["method"] == "cbl":
            # projection, three-term update (one triangular factor), two triangular products,
            # two symmetric Grams, assembly
            flops += rows * M * M * 11.0
            if case["reorth"] == 1:
                flops += sum(4.0 * k * reach(M, k) for k in range(1, m)) * M * M
            # the stored basis is written once and read once
            nbytes += 2.0 * size * rows * M
        elif case["method"] in ("gbl", "sbl"):
            flops += 6.0 * M * rows
            nbytes += 2.0 * size * rows * M
    return {"bytes": nbytes, "flops": flops}

"""Grid barriers that run out of their polls (none allowed: every CTA gives up at the first one),
through the library's own launchers: the projected series ends the process with KB_ERR_CUDA, the search
reaches every row.  And the stopping
rule on a solution that is not finite."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KB_ERR_CUDA = -4
I32, VP, DBL = ctypes.c_int, ctypes.c_void_p, ctypes.c_double


class Ctrl(ctypes.Structure):
    _fields_ = [("status", I32), ("stop", I32), ("steps", I32), ("breakdown_step", I32), ("est_change", DBL),
                ("from_check", I32), ("reserved", I32)]

    @staticmethod
    def on_device(steps):
        import torch
        c = Ctrl(0, 0, steps, -1, -1.0, -1, 0)
        return torch.frombuffer(bytearray(bytes(c)), dtype=torch.uint8).cuda()

    @staticmethod
    def read(t):
        return Ctrl.from_buffer_copy(t.cpu().numpy().tobytes())


@pytest.fixture(scope="module")
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_06384_gb300 import kb
    kb.lib()
    return ctypes.CDLL(kb.LIB_PATH)


def _tridiagonal(M, m, seed):
    """Blocks of a block tridiagonal matrix (off-diagonal blocks upper triangular), the matrix."""
    rng = np.random.default_rng(seed)
    Hd = rng.standard_normal((m, M, M)) / np.sqrt(M)
    Hd = (0.5 * (Hd + Hd.transpose(0, 2, 1)) + 6 * np.eye(M)).astype(np.float32).astype(np.float64)
    Hs = (np.triu(rng.standard_normal((m, M, M))) / np.sqrt(M)).astype(np.float32).astype(np.float64)
    H = np.zeros((m * M, m * M))
    for k in range(m):
        a = slice(k * M, (k + 1) * M)
        H[a, a] = Hd[k]
        if k + 1 < m:
            b = slice((k + 1) * M, (k + 2) * M)
            H[b, a], H[a, b] = Hs[k], Hs[k].T
    return Hd, Hs, H


@pytest.mark.parametrize("M,m", [(1, 1), (9, 5), (40, 7)])
def test_projected_series_gives_up(lib, M, m):
    import scipy.linalg
    import torch
    from paper_2301_06384_gb300 import kb
    Hd, Hs, H = _tridiagonal(M, m, M)
    lam = float(np.abs(H).sum(1).max())
    d = kb.kb_exp_series_coeffs(1.0, lam)
    vec = (VP * 3)(d.ctypes.data, d.ctypes.data + d.nbytes, d.ctypes.data + d.nbytes)   # a std::vector<double>
    f = lib["_ZN2kb14launch_cheb_btEPKdS1_iidRKSt6vectorIdSaIdEEPdS7_S7_S7_PKNS_4CtrlEP11CUstream_stS7_PiiPS8_i"]
    f.restype, f.argtypes = I32, [VP, VP, I32, I32, DBL, VP, VP, VP, VP, VP, VP, VP, VP, VP, I32, VP, I32]
    hd, hs = [torch.from_numpy(h).cuda() for h in (Hd, Hs)]
    V = [torch.zeros(m * M * M, dtype=torch.float64, device="cuda") for _ in range(3)]
    hdf = torch.zeros(2 * m * M * (M + 1), dtype=torch.float64, device="cuda")
    sync = torch.zeros(2, dtype=torch.int32, device="cuda")
    exact = scipy.linalg.expm(-H)[:, :M]
    for spins in (1 << 22, 0):
        U = torch.zeros(m * M, M, dtype=torch.float64, device="cuda")
        ctrl, proc = Ctrl.on_device(m), Ctrl.on_device(m + 3)
        torch.cuda.synchronize()
        rc = f(hd.data_ptr(), hs.data_ptr(), M, m, lam, ctypes.addressof(vec), *[v.data_ptr() for v in V], U.data_ptr(),
               ctrl.data_ptr(), None, hdf.data_ptr(), sync.data_ptr(), m, proc.data_ptr(), spins)
        torch.cuda.synchronize()
        assert rc == 0
        p, u = Ctrl.read(proc), U.cpu().numpy()
        if spins:
            assert (p.status, p.stop, p.steps) == (0, 0, m + 3)
            # pairs of floats, about 30 terms of a recurrence: 30^2 units of 2^-46
            assert np.abs(u - exact).max() < 900 * 2.0 ** -46
        else:
            assert (p.status, p.stop, p.steps) == (KB_ERR_CUDA, 1, m)
            assert np.isnan(u).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_check_of_unusable_u_does_not_converge(lib, bad):
    """The stopping rule on a U that holds a NaN or an infinity: the process goes on (the test of the
    projected solution reports it), and the change is not a number."""
    import torch
    f = lib["_ZN2kb17launch_conv_checkEPKdS1_iPKNS_4CtrlEPidPS2_P11CUstream_sti"]
    f.restype, f.argtypes = I32, [VP, VP, I32, VP, VP, DBL, VP, VP, I32]
    M, steps, before = 5, 4, 3
    rng = np.random.default_rng(1)
    for value in (None, bad):
        Up = torch.from_numpy(rng.standard_normal(before * M * M)).cuda()
        U = torch.cat([Up, torch.zeros((steps - before) * M * M, dtype=torch.float64, device="cuda")])
        if value is not None:
            U[7] = value
        prev = torch.tensor([before], dtype=torch.int32, device="cuda")
        chk, ctrl = Ctrl.on_device(steps), Ctrl.on_device(20)
        torch.cuda.synchronize()
        assert f(U.data_ptr(), Up.data_ptr(), M, chk.data_ptr(), prev.data_ptr(), 1e-6, ctrl.data_ptr(), None, 1) == 0
        torch.cuda.synchronize()
        c = Ctrl.read(ctrl)
        if value is None:
            assert (c.stop, c.steps, c.from_check, c.est_change) == (1, steps, 1, 0.0)
        else:
            assert (c.stop, c.steps, c.from_check) == (0, 20, -1) and np.isnan(c.est_change)
        assert int(prev) == steps


class GraphDev(ctypes.Structure):
    _fields_ = [("n", ctypes.c_int64), ("nnz", ctypes.c_int64), ("rowptr", VP), ("col", VP), ("w", VP), ("rdiag", VP),
                ("longs", VP), ("nlong", I32), ("long_row", I32)]


class FrontierBufs(ctypes.Structure):
    _fields_ = [(f, VP) for f in ("gen", "tgen", "alist", "acount", "lists", "zeroed")] + [("zero_bytes", ctypes.c_size_t)] + \
               [(f, VP) for f in ("qlev", "tcnt", "queue", "sync", "vis")] + [("levels", I32), ("nt", ctypes.c_int64)]


@pytest.fixture(scope="module")
def layouts(tmp_path_factory):
    """The two structures' layouts by the compiler, before anything is launched with the ones above."""
    from paper_2301_06384_gb300 import build
    d = tmp_path_factory.mktemp("layout")
    lines = []
    for cls in (GraphDev, FrontierBufs):
        name = cls.__name__
        lines.append(f'printf("{name} %zu\\n", sizeof(kb::{name}));')
        lines += [f'printf("{name}.{f[0]} %zu\\n", offsetof(kb::{name}, {f[0]}));' for f in cls._fields_]
    (d / "layout.cu").write_text("#include <cstddef>\n#include <cstdio>\n#include \"kb_internal.cuh\"\n#include "
                                 "\"kb_kernels.cuh\"\nint main() {\n" + "\n".join(lines) + "\n}\n")
    subprocess.run([build.nvcc(), *build._flags(), "-c", str(d / "layout.cu"), "-o", str(d / "layout.o")], check=True)
    subprocess.run([build.nvcc(), build.ARCH, str(d / "layout.o"), "-o", str(d / "layout")], check=True)
    got = dict(x.split() for x in subprocess.run([str(d / "layout")], check=True, capture_output=True, text=True).stdout.splitlines())
    for cls in (GraphDev, FrontierBufs):
        assert int(got[cls.__name__]) == ctypes.sizeof(cls)
        for f in cls._fields_:
            assert int(got[f"{cls.__name__}.{f[0]}"]) == getattr(cls, f[0]).offset, f[0]


@pytest.mark.parametrize("n", [31, 5000])
@pytest.mark.parametrize("levels", [2, 9])
def test_search_that_gives_up_reaches_every_row(lib, layouts, n, levels):
    """Distances and tile lists of the search; without polls every row counts as reached at once, and
    the lists hold every tile."""
    import torch
    # a path with a few chords: rows in hop order of node 0 only near the start
    src = np.concatenate([np.arange(n - 1), np.arange(0, n - 40, 37)])
    dst = np.concatenate([np.arange(1, n), np.arange(0, n - 40, 37) + 29])
    r, c = np.concatenate([src, dst]), np.concatenate([dst, src])
    order = np.argsort(r, kind="stable")
    ptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int32)
    col = c[order].astype(np.int32)
    nodes = np.array([n // 2, 3, n - 1], dtype=np.int32)
    dist = np.full(n, 255)
    dist[nodes] = 0
    for k in range(1, levels + 1):
        near = np.concatenate([col[:0]] + [col[ptr[i]:ptr[i + 1]] for i in np.nonzero(dist == k - 1)[0]])
        near = near[dist[near] == 255]
        dist[near] = k

    plan = lib["_ZN2kb13plan_frontierERNS_12FrontierBufsEliPhPmS2_"]
    plan.restype, plan.argtypes = None, [VP, ctypes.c_int64, I32, VP, VP, VP]
    search = lib["_ZN2kb21frontier_search_bytesEl"]
    search.restype, search.argtypes = ctypes.c_size_t, [ctypes.c_int64]
    launch = lib["_ZN2kb15launch_frontierERKNS_8GraphDevERNS_12FrontierBufsEPKiiP11CUstream_sti"]
    launch.restype, launch.argtypes = I32, [VP, VP, VP, I32, VP, I32]
    dptr, dcol = torch.from_numpy(ptr).cuda(), torch.from_numpy(col).cuda()
    g = GraphDev(n, col.size, dptr.data_ptr(), dcol.data_ptr(), None, None, None, 0, 64)
    fr, size = FrontierBufs(), ctypes.c_size_t()
    plan(ctypes.byref(fr), n, levels, None, ctypes.byref(size), None)
    buf = torch.zeros(size.value, dtype=torch.uint8, device="cuda")
    scratch = torch.zeros(search(n), dtype=torch.uint8, device="cuda")
    plan(ctypes.byref(fr), n, levels, buf.data_ptr(), ctypes.byref(size), scratch.data_ptr())
    nt = (n + 31) // 32
    assert (fr.levels, fr.nt) == (levels, nt)

    def ints(p, count):
        return buf[p - buf.data_ptr():][:4 * count].cpu().numpy().view(np.int32)

    for spins in (1 << 22, 0):
        buf.fill_(0xA5)
        scratch.fill_(0xA5)
        torch.cuda.synchronize()
        assert launch(ctypes.byref(g), ctypes.byref(fr), nodes.ctypes.data, nodes.size, None, spins) == 0
        torch.cuda.synchronize()
        want = dist if spins else np.zeros(n, dtype=int)
        gen = buf[fr.gen - buf.data_ptr():][:n].cpu().numpy()
        assert np.array_equal(gen, want)
        tile = np.array([want[32 * t:32 * t + 32].min() for t in range(nt)])
        tgen = ints(fr.tgen, nt)
        assert np.array_equal(np.where(tgen > levels, 255, tgen), tile)
        assert np.array_equal(ints(fr.alist, nt), np.argsort(tile, kind="stable"))
        count = ints(fr.acount, levels + 1)
        lists = ints(fr.lists, (levels + 1) * nt).reshape(levels + 1, nt)
        for k in range(levels + 1):
            assert count[k] == np.sum(tile <= k)
            assert np.array_equal(lists[k, :count[k]], np.nonzero(tile <= k)[0])

"""Grid barriers that run out of their polls (none allowed: every CTA gives up at the first one),
through the library's own launchers: the projected series ends the process with KB_ERR_CUDA.  And the stopping
rule on a solution that is not finite."""
import ctypes

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

"""The CholeskyQR kernel against extended precision, through the library's own launcher: R1 as the
inverse of the applied inverse on both sides of the width where its form changes, and the
reciprocals of the pivots."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U32, U64 = 2.0 ** -24, 2.0 ** -53
LAUNCH = {"f": "_ZN2kb11launch_cholIfEEiPKdiiiiddPdPT_S3_S5_PNS_4CtrlEP11CUstream_st",
          "d": "_ZN2kb11launch_cholIdEEiPKdiiiiddPdPT_S3_S5_PNS_4CtrlEP11CUstream_st"}


@pytest.fixture(scope="module")
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_06384_gb300 import kb
    kb.lib()
    return ctypes.CDLL(kb.LIB_PATH)


def _pass1(lib, G, kind):
    """(S, R1): the applied inverse and the FP64 inverse of it for the M x M Gram matrix G."""
    import torch
    M = G.shape[0]
    W = next(w for w in (16, 32, 64, 128) if M <= w)
    f = getattr(lib, LAUNCH[kind])
    f.restype = ctypes.c_int
    vp, i32, dbl = ctypes.c_void_p, ctypes.c_int, ctypes.c_double
    f.argtypes = [vp, i32, i32, i32, i32, dbl, dbl] + [vp] * 6
    Gw = torch.zeros(W, W, dtype=torch.float64, device="cuda")
    Gw[:M, :M] = torch.from_numpy(np.ascontiguousarray(G))
    R1, Hs = [torch.zeros(M, M, dtype=torch.float64, device="cuda") for _ in range(2)]
    S, B = [torch.zeros(W, W, dtype=torch.float32 if kind == "f" else torch.float64, device="cuda") for _ in range(2)]
    ctrl = torch.zeros(8, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    rc = f(Gw.data_ptr(), M, W, 1, 1, 0.0, 0.0, R1.data_ptr(), S.data_ptr(), Hs.data_ptr(), B.data_ptr(), ctrl.data_ptr(),
           None)
    torch.cuda.synchronize()
    assert rc == 0 and int(ctrl[1]) == 0
    return S[:M, :M].double().cpu().numpy(), R1.cpu().numpy()


# columns of sizes 1 to 50 (triangular inversion does not depend on the scaling of columns).  FP64
# inversion: sums of M rounding errors, 4 sqrt(M) u; the corrected FP32 factor: E is at most about M u32,
# its corrections are rounded to FP32, so M u32^2 and a third-order term below it
@pytest.mark.parametrize("M,kind", [(1, "f"), (16, "f"), (33, "f"), (64, "f"), (65, "f"), (80, "f"), (113, "f"), (128, "f"),
                                    (1, "d"), (17, "d"), (33, "d"), (64, "d")])
def test_r1_is_the_inverse_of_the_applied_inverse(lib, M, kind):
    rng = np.random.default_rng(M)
    X = rng.standard_normal((6 * M, M)) * np.logspace(0, 1.7, M)[rng.permutation(M)][None, :]
    X = X @ (np.eye(M) + 0.3 * rng.standard_normal((M, M)) / np.sqrt(M))
    S, R1 = _pass1(lib, X.T @ X, kind)
    assert np.all(np.tril(S, -1) == 0) and np.all(np.tril(R1, -1) == 0)
    Q = X @ S
    assert np.linalg.norm(Q.T @ Q - np.eye(M)) < 50 * M * (U32 if kind == "f" else U64)   # 50: the scaling
    ld = np.longdouble
    R = np.linalg.inv(S)
    ref = R.astype(ld) + R.astype(ld) @ (np.eye(M) - S.astype(ld) @ R.astype(ld))
    err = float(np.abs(R1 - ref).max() / np.abs(ref).max())
    assert err < (4 * M ** 0.5 * U64 if kind == "d" or M > 64 else max(8, M) * U32 ** 2 * 8), err


@pytest.mark.parametrize("kind", ["f", "d"])
def test_pivot_reciprocals_are_rounded(lib, kind):
    # diagonal G: S holds the reciprocals of the (correctly rounded) square roots: half a unit in
    # the last place, and in FP64 a term of the squared error before the last Newton step
    rng = np.random.default_rng(3)
    dt, ulp = (np.float32, 2 * U32) if kind == "f" else (np.float64, 2 * U64)
    for rep in range(20):
        d = 10.0 ** rng.uniform(0, 4 if kind == "f" else 200, 64) * (1 if kind == "f" else 1e-100)
        if kind == "f":
            d = d.astype(np.float32).astype(np.float64)
        S, _ = _pass1(lib, np.diag(d), kind)
        rt = np.sqrt(d.astype(dt)).astype(np.longdouble)
        exact = 1 / rt
        unit = np.exp2(np.floor(np.log2(exact.astype(np.float64)))) * ulp
        assert np.all(np.abs(np.diag(S) - exact) <= 0.51 * unit)

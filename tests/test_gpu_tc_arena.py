"""The tensor-core filter for a problem smaller than the handle has served before: only its own
tiles are computed, over the K slices of the larger order and with column tiles of half the width
where few blocks would run. Exact on small integers (BF16 operands, FP32 sums below 2^24), with
nothing of the larger problem (here NaN) left in the padding; the FP32-class form keeps the
tolerance it has on a fresh handle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def T(x, dev):
    return torch.from_numpy(np.ascontiguousarray(x)).to(dev)


def _tc_product(cuda, Cm, Y):
    import ctypes as C
    from paper_1007_4400_gb300 import gevp
    L = gevp.load()
    L.gevp_matmul_tc.argtypes = [C.c_void_p, C.c_int64, C.c_int, C.c_void_p, C.c_int64, C.c_void_p, C.c_int64,
                                 C.c_void_p, C.c_int64]
    L.gevp_matmul_tc.restype = C.c_int
    Ct, Yt = T(Cm, cuda), T(Y, cuda)
    D = torch.empty_like(Yt)
    h = gevp._handle(cuda)
    st = L.gevp_matmul_tc(h, Ct.shape[0], Yt.shape[1], C.c_void_p(Ct.data_ptr()), Ct.stride(0),
                          C.c_void_p(Yt.data_ptr()), Yt.stride(0), C.c_void_p(D.data_ptr()), D.stride(0))
    gevp._check(st, h)
    return D.cpu().numpy()


@pytest.mark.parametrize("n,m", [(64, 1), (129, 65), (300, 140), (777, 200), (1024, 161), (1407, 129)])
def test_product_after_a_larger_problem(cuda, n, m):
    rng = np.random.default_rng(4100 + n + m)
    big = np.full((1500, 1500), np.nan + 0j)
    assert np.isnan(_tc_product(cuda, big, np.ones((1500, 210), complex))).all()
    Cm = rng.integers(-2, 3, (n, n)) + 1j * rng.integers(-2, 3, (n, n))
    Y = rng.integers(-2, 3, (n, m)) + 1j * rng.integers(-2, 3, (n, m))
    D = _tc_product(cuda, Cm.astype(np.complex128), Y.astype(np.complex128))
    assert np.array_equal(D, Cm @ Y)


@pytest.mark.parametrize("n,m", [(384, 40), (500, 130)])
def test_fp32_filter_after_a_larger_problem(cuda, n, m):
    from oracle import pieces
    from paper_1007_4400_gb300 import gevp
    rng = np.random.default_rng(4200 + n)
    _tc_product(cuda, np.full((1500, 1500), np.nan + 0j), np.ones((1500, 210), complex))
    lam = np.sort(rng.uniform(-2, 50, n))
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    Cm = (Q * lam) @ Q.conj().T
    Cm = 0.5 * (Cm + Cm.conj().T)
    Y0 = rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m))
    lo, hi, s = 5.0, 50.5, -2.5
    Yg = gevp.chebyshev_filter(T(Cm, cuda), T(Y0, cuda), 12, lo, hi, s, prec="fp32").cpu().numpy()
    Yr = pieces.chebyshev_filter(Cm, Y0, 12, lo, hi, s)
    assert np.linalg.norm(Yg - Yr) / np.linalg.norm(Yr) < 2e-5

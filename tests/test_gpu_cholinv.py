"""The cluster Cholesky factor and inverse at the edges of its panels (8 columns) and of its rows
per CTA (16 CTAs), through CholQR2, and its short form for matrices near the identity."""
import numpy as np
import pytest
import torch

from tests.conftest import crandn

pytestmark = pytest.mark.gpu


# 1, 7, 8, 9: one panel and its edges; 16, 17: one row per CTA and one more; 129, 257, 288: more rows
@pytest.mark.parametrize("m", [1, 7, 8, 9, 16, 17, 129, 257, 288, 289])
@pytest.mark.parametrize("kind", ["general", "orthonormal", "nearly"])
def test_cholqr2(cuda, m, kind):
    from paper_1007_4400_gb300 import gevp
    n = 700
    rng = np.random.default_rng(8000 + m)
    Y = crandn(rng, n, m)
    if kind != "general":
        # an orthonormal block (the first pass takes the short form), and one whose Gram matrix is
        # about 1e-7 away from the identity (only the second does), columns of different lengths
        Y = np.linalg.qr(Y)[0]
        if kind == "nearly":
            Y = Y + 1e-8 * crandn(rng, n, m)
        Y = Y * np.exp(rng.uniform(-3, 3, m))
    Q, R = np.linalg.qr(Y)
    ph = np.diag(R) / np.abs(np.diag(R))
    Q, R = Q * ph, np.conj(ph)[:, None] * R
    t = torch.empty(Y.shape, dtype=torch.complex128, device=cuda).copy_(torch.from_numpy(Y))
    Qg, Rg = gevp.cholqr2(t, want_R=True)
    Qg, Rg = Qg.cpu().numpy(), Rg.cpu().numpy()
    # CholQR2: orthonormality and residual at FP64 rounding times a modest function of the sizes
    assert np.abs(Qg.conj().T @ Qg - np.eye(m)).max() <= 1e-13
    assert np.abs(Qg @ Rg - Y).max() <= 1e-13 * np.abs(Y).max() * np.sqrt(m)
    # cond(Y) <= about 10 after scaling: the factors themselves agree with Householder QR's
    assert np.abs(Qg - Q).max() <= 1e-12


@pytest.mark.parametrize("n,m", [(700, 40), (2100, 140), (2500, 300)])
def test_columns_over_many_decades(cuda, n, m):
    """Columns whose lengths span sixteen decades (FP64 kernels, emulated products, orders above the
    cluster's): Q does not depend on the lengths, so it has to be as accurate as for unit columns."""
    from paper_1007_4400_gb300 import gevp
    rng = np.random.default_rng(8500 + m)
    Y = crandn(rng, n, m)
    Q, R = np.linalg.qr(Y)
    Q = Q * (np.diag(R) / np.abs(np.diag(R)))
    t = torch.empty(Y.shape, dtype=torch.complex128, device=cuda).copy_(
        torch.from_numpy(Y * 2.0 ** rng.integers(-27, 28, m)))
    Qg = gevp.cholqr2(t).cpu().numpy()
    assert np.abs(Qg - Q).max() <= 1e-13


def test_non_finite_entries_stay_visible(cuda):
    """A NaN or Inf in a large projection is not lost in the emulated products."""
    from paper_1007_4400_gb300 import gevp
    n, m = 1600, 64
    C = torch.eye(n, dtype=torch.complex128, device=cuda)
    Q = torch.linalg.qr(torch.randn((n, m), dtype=torch.complex128, device=cuda))[0].contiguous()
    C[5, 7] = complex(float("nan"), 0.0)
    th, _, W, _ = gevp.rayleigh_ritz(C, Q)
    assert torch.isnan(torch.view_as_real(W)).any() and torch.isnan(th).any()
    X = torch.randn((n, 300), dtype=torch.complex128, device=cuda)
    X[3, 2] = complex(float("inf"), 0.0)
    GA, GB = gevp.energy_backward(X, torch.ones(300, dtype=torch.float64, device=cuda))
    assert not torch.isfinite(torch.view_as_real(GA[3])).all() and not torch.isfinite(torch.view_as_real(GB[3])).all()
    # and it is not held against a later call
    A = torch.randn((300, 300), dtype=torch.complex128, device=cuda)
    assert torch.isfinite(torch.view_as_real(gevp.zgemm_emulated(A, A))).all()

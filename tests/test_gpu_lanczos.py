"""Lanczos bounds at the edges of the row slices, of the cluster sizes and of the order from which the
products run outside the cluster, and after a breakdown. With full re-orthogonalisation in FP32 the
Ritz values lie in the spectrum to n 2^-24 ||A||, whatever was summed in which order; with as many
steps as the order, or as many as there are distinct eigenvalues, the extreme ones are reached
(to 64 n 2^-24 ||A||), and after a breakdown the last residual norm counts as zero."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _matrix(rng, lam):
    n = len(lam)
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    A = (Q * lam) @ Q.conj().T
    return 0.5 * (A + A.conj().T)


@pytest.mark.parametrize("n", [2, 17, 31, 63, 64, 65, 129, 520, 1025, 2304, 2305])
def test_bounds_at_slice_edges(cuda, n):
    from paper_1007_4400_gb300 import gevp
    rng = np.random.default_rng(7000 + n)
    if n <= 600:
        lam = np.sort(rng.uniform(-3, 11, n))
        A = _matrix(rng, lam)
    else:   # the spectrum of a random Hermitian matrix
        A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        A = 0.5 * (A + A.conj().T)
        lam = np.linalg.eigvalsh(A)
    b = [float(x) for x in gevp.spectral_bounds(torch.from_numpy(A).to(cuda), k=32, count=max(1, n // 4))]
    tol = n * 2.0 ** -24 * np.abs(lam).max() + 1e-5 * np.abs(lam).max()
    assert lam[0] - tol <= b[0] <= b[1] <= lam[-1] + tol
    assert b[2] >= b[1] and b[2] >= lam[-1] - tol
    if n <= 32:
        assert abs(b[0] - lam[0]) <= 64 * tol and abs(b[1] - lam[-1]) <= 64 * tol


@pytest.mark.parametrize("n", [60, 300, 2400])
def test_breakdown(cuda, n):
    from paper_1007_4400_gb300 import gevp
    rng = np.random.default_rng(7100 + n)
    u = rng.standard_normal((n, 2)) + 1j * rng.standard_normal((n, 2))
    u, _ = np.linalg.qr(u)
    A = 2.0 * np.eye(n) + u @ np.diag([5.0, -4.0]) @ u.conj().T   # eigenvalues 2, 7, -2
    A = 0.5 * (A + A.conj().T)
    lo, hi, upper, _, beta = [float(x) for x in gevp.spectral_bounds(torch.from_numpy(A).to(cuda), k=32, count=1)]
    tol = 64 * n * 2.0 ** -24 * 7
    assert abs(lo + 2) <= tol and abs(hi - 7) <= tol
    assert upper >= 7 - tol and beta <= 7

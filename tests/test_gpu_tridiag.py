"""The small eigensolver across the forms of its FP32 start (one CTA, clusters of eight and
sixteen, orders above them) and on spectra that make the QL iteration split or deflate."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def unitary(rng, m):
    return np.linalg.qr(rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m)))[0]


def spectrum(kind, rng, m):
    if kind == "random":
        return np.sort(rng.uniform(-2, 5, m))
    if kind == "degenerate":          # three values, each many times
        return np.sort(rng.integers(0, 3, m).astype(float))
    if kind == "graded":              # four decades
        return 10.0 ** np.linspace(-3, 1, m)
    if kind == "cluster":             # a quarter of the values (at most 60) closer than FP32 resolves
        c = min(m // 4, 60)
        return np.sort(np.concatenate([np.linspace(0, 1e-5, c), rng.uniform(0.1, 1, m - c)]))
    return np.zeros(m)


# 1, 2: no and one reflector; 32 | 33, 72 | 73, 160 | 161, 256 | 257, 416 | 417: the forms' edges
@pytest.mark.parametrize("m", [1, 2, 3, 31, 32, 33, 72, 73, 160, 161, 256, 257, 416, 417, 601])
@pytest.mark.parametrize("kind", ["random", "degenerate", "graded", "cluster", "zero"])
def test_eigenpairs(cuda, m, kind):
    from paper_1007_4400_gb300 import gevp
    if m == 601 and kind != "random":
        pytest.skip("one spectrum above the limit")
    rng = np.random.default_rng(9000 + m)
    lam, V = spectrum(kind, rng, m), unitary(rng, m)
    G = (V * lam) @ V.conj().T
    G = (G + G.conj().T) / 2
    th, Z = gevp.heev_small(torch.from_numpy(G).to(cuda))
    th, Z = th.cpu().numpy(), Z.cpu().numpy()
    scale = max(np.abs(lam).max(), 1e-300)
    # FP64 rounding of an order-m product: m u, with room for the constants (as the parity tests)
    tol = 1e-12
    assert np.all(np.diff(th) >= 0)
    assert np.abs(th - lam).max() <= tol * scale
    assert np.abs(G @ Z - Z * th).max() <= tol * scale
    assert np.abs(Z.conj().T @ Z - np.eye(m)).max() <= tol


def test_tridiagonal_and_diagonal_input(cuda):
    """Columns that are already reduced (tau = 0), exact splits, and an unsorted diagonal."""
    from paper_1007_4400_gb300 import gevp
    m = 90
    rng = np.random.default_rng(9500)
    d, e = rng.standard_normal(m), rng.standard_normal(m - 1)
    e[[10, 40, 41]] = 0.0
    for G in (np.diag(d), np.diag(d) + np.diag(e, 1) + np.diag(e, -1)):
        G = G.astype(np.complex128)
        th, Z = gevp.heev_small(torch.from_numpy(G).to(cuda))
        th, Z = th.cpu().numpy(), Z.cpu().numpy()
        assert np.abs(th - np.linalg.eigvalsh(G)).max() <= 1e-12 * np.abs(G).max()
        assert np.abs(G @ Z - Z * th).max() <= 1e-12 * np.abs(G).max()

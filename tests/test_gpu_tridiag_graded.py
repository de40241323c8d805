"""The small eigensolver on matrices whose reduction meets columns far below FP32's resolution of the
whole matrix: rounding residue of low-rank matrices (it shrinks by 1e-8 a step) and entries over
many decades. The results are as exact as any in terms of the matrix's norm; the same matrices as
k-points of a batch whose blocks span the whole space."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def herm(rng, m):
    X = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    return 0.5 * (X + X.conj().T)


def matrix(kind, m):
    rng = np.random.default_rng(9800 + m)
    if kind == "ones":
        return np.ones((m, m), dtype=complex)
    if kind == "rank1":
        u = rng.standard_normal(m) + 1j * rng.standard_normal(m)
        return np.outer(u, u.conj())
    if kind == "graded":              # D M D, D over 40 decades
        d = 10.0 ** -np.linspace(0, 40, m)
        return d[:, None] * herm(rng, m) * d
    G = np.zeros((m, m), dtype=complex)   # two blocks, one 1e-21 of the other
    b = m // 2
    G[:b, :b] = herm(rng, b)
    G[b:, b:] = 1e-21 * herm(rng, m - b)
    return G


# one CTA (up to 72) and clusters of eight
@pytest.mark.parametrize("m", [8, 24, 48, 72, 73, 100])
@pytest.mark.parametrize("kind", ["ones", "rank1", "graded", "blocks"])
def test_eigenpairs(cuda, m, kind):
    from paper_1007_4400_gb300 import gevp
    G = matrix(kind, m)
    th, Z = gevp.heev_small(torch.from_numpy(G).to(cuda))
    th, Z = th.cpu().numpy(), Z.cpu().numpy()
    scale = np.abs(np.linalg.eigvalsh(G)).max()
    # FP64 rounding of an order-m product, as in the other eigensolver tests
    assert np.abs(th - np.linalg.eigvalsh(G)).max() <= 1e-12 * scale
    assert np.abs(G @ Z - Z * th).max() <= 1e-12 * scale
    assert np.abs(Z.conj().T @ Z - np.eye(m)).max() <= 1e-12


def test_batch_of_whole_spaces(cuda):
    from paper_1007_4400_gb300 import gevp
    sizes = [24, 48, 73]
    As = [torch.from_numpy(matrix(kind, m)).to(cuda) for m, kind in zip(sizes, ["ones", "blocks", "rank1"])]
    Bs = [torch.eye(m, dtype=torch.complex128, device=cuda) for m in sizes]
    r = gevp.solve_batched([[A] for A in As], Bs, [m - 2 for m in sizes], nex=2)
    for A, lam, res in zip(As, r.Lambda, r.resid):
        ref = np.linalg.eigvalsh(A.cpu().numpy())
        lam = lam[0].cpu().numpy()
        assert res.max().item() <= 1e-10
        assert np.abs(lam - ref[:len(lam)]).max() <= 1e-12 * np.abs(ref).max()

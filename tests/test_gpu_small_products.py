"""The 4 x 8 tiles of the small FP64 products, at the edges of tiles and of the eight-way split of K,
through the per-step entry points: the FP64 filter (products with both added terms), the
orthonormalisation (Gram matrix, triangular product) and Rayleigh-Ritz (Q^H W). References in
NumPy. Tolerances: a filter step adds n products and two terms, each 2^-53 of the row's absolute sum,
for three steps; the others (n + 8 m) 2^-53 of norms of order one times a factor for the chain."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def T(x, dev):
    return torch.from_numpy(np.ascontiguousarray(x)).to(dev)


@pytest.mark.parametrize("n,m", [(2, 1), (5, 3), (8, 8), (9, 1), (17, 9), (50, 18), (63, 33), (129, 7)])
def test_fp64_filter_of_small_blocks(cuda, n, m):
    from oracle import pieces
    from paper_1007_4400_gb300 import gevp
    rng = np.random.default_rng(6000 + 13 * n + m)
    C = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    C = 0.5 * (C + C.conj().T)
    Y = rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m))
    w = np.abs(np.linalg.eigvalsh(C)).max()
    lo, hi, s = 0.2 * w, 1.1 * w, -1.1 * w
    Yg = gevp.chebyshev_filter(T(C, cuda), T(Y, cuda), 3, lo, hi, s, prec="fp64").cpu().numpy()
    Yr = pieces.chebyshev_filter(C, Y, 3, lo, hi, s)
    # |p_j(t)| <= 1 between s and the damped interval; the chain's factors 2 sn / e * ||C||_F and so on
    # are at most 8 ||C||_F / e, three steps
    bound = 3 * (n + 8) * U * (8 * np.linalg.norm(C) / (0.45 * w)) * np.linalg.norm(Y)
    assert np.linalg.norm(Yg - Yr) <= bound


@pytest.mark.parametrize("n,m", [(5, 3), (9, 8), (50, 18), (64, 33), (130, 9), (257, 17)])
def test_orthonormal_and_ritz_of_small_blocks(cuda, n, m):
    from paper_1007_4400_gb300 import gevp
    rng = np.random.default_rng(6100 + 13 * n + m)
    Y = rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m))
    Q = gevp.cholqr2(T(Y, cuda)).cpu().numpy()
    assert np.linalg.norm(Q.conj().T @ Q - np.eye(m)) <= 8 * (n + 8 * m) * U * m
    assert np.linalg.norm(Q @ (Q.conj().T @ Y) - Y) <= 32 * (n + 8 * m) * U * m * np.linalg.norm(Y)
    C = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    C = 0.5 * (C + C.conj().T)
    th = gevp.rayleigh_ritz(T(C, cuda), T(Q, cuda))[0].cpu().numpy()
    ref = np.linalg.eigvalsh(Q.conj().T @ C @ Q)
    assert np.abs(th - ref).max() <= 8 * (n + 8 * m) * U * np.linalg.norm(C)

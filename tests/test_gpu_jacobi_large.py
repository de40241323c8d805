"""The small eigensolver above the order of its tridiagonal start (600), where FP32 Jacobi runs on all
SMs: even and odd orders up to the largest, well separated values and a multiple one."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,multiple", [(602, 1), (749, 40), (1024, 1)])
def test_eigenpairs(cuda, m, multiple):
    from paper_1007_4400_gb300 import gevp
    g = torch.Generator(device=cuda).manual_seed(m)
    V = torch.linalg.qr(torch.randn(m, m, dtype=torch.complex128, device=cuda, generator=g))[0]
    lam = torch.linspace(-2, 5, m, dtype=torch.float64, device=cuda)
    lam[:multiple] = lam[0].item()
    G = (V * lam) @ V.conj().T
    G = 0.5 * (G + G.conj().T)
    th, Z = gevp.heev_small(G)
    # FP64 rounding of an order-m product, as in the other eigensolver tests
    assert (th[1:] >= th[:-1]).all()
    assert (th - lam).abs().max().item() <= 1e-12 * 5
    assert (G @ Z - Z * th).abs().max().item() <= 1e-12 * 5
    assert (Z.conj().T @ Z - torch.eye(m, dtype=Z.dtype, device=cuda)).abs().max().item() <= 1e-12

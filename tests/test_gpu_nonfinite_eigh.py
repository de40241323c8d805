"""A NaN or Inf in the matrix of the small eigensolver: NaN eigenvalues, every one of them written,
on each side of the orders where the FP32 start changes its form (above 600 its permutation is an
index into memory)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("m", [2, 48, 140, 601])
def test_every_eigenvalue_is_nan(cuda, m, bad):
    from paper_1007_4400_gb300 import gevp
    g = torch.Generator(device=cuda).manual_seed(m)
    G = torch.randn(m, m, dtype=torch.complex128, device=cuda, generator=g)
    G = 0.5 * (G + G.conj().T)
    gevp.heev_small(G)   # finite values in the workspace and in the memory of the results
    G[m - 1, m - 2] = G[m - 2, m - 1] = bad
    th, Z = gevp.heev_small(G)
    assert torch.isnan(th).all()
    # and the next call is not affected
    G[m - 1, m - 2] = G[m - 2, m - 1] = 0.25
    th, Z = gevp.heev_small(G)
    assert (G @ Z - Z * th).abs().max().item() <= 1e-12 * G.abs().max().item() * m

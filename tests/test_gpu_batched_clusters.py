"""K-points with a cluster of eigenvalues that the FP32 start of the small eigensolver cannot resolve,
in blocks that span the whole space: the exact rotations separate them."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,c", [(64, 16), (160, 40), (256, 60)])
def test_unresolved_cluster(cuda, m, c):
    from paper_1007_4400_gb300 import gevp
    rng = np.random.default_rng(m)
    V = np.linalg.qr(rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m)))[0]
    lam = np.sort(np.concatenate([np.linspace(0, 1e-5, c), rng.uniform(0.1, 1, m - c)]))
    A = torch.from_numpy((V * lam) @ V.conj().T).to(cuda)
    A = 0.5 * (A + A.conj().T)
    B = torch.eye(m, dtype=torch.complex128, device=cuda)
    r = gevp.solve_batched([[A], [A.conj().resolve_conj().clone()]], [B, B], m - 2, nex=2, tol=1e-13)
    assert r.status == 0
    for k in range(2):
        assert r.resid[k].max().item() <= 1e-13
        assert np.abs(r.Lambda[k][0].cpu().numpy() - lam[:m - 2]).max() <= 1e-12
        X = r.X[k]
        assert (X.conj().T @ X - torch.eye(m - 2, dtype=X.dtype, device=cuda)).abs().max().item() <= 1e-10

"""Failures that a kernel records in a device word reach the caller of the call in which they
happened, and no other. They are injected on the host: nothing fails on the device."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _herm(m, device):
    g = torch.Generator(device=device).manual_seed(m)
    G = torch.randn(m, m, dtype=torch.complex128, device=device, generator=g)
    return 0.5 * (G + G.conj().T)


def test_small_eigensolver(cuda):
    from paper_1007_4400_gb300 import gevp
    G = _herm(48, cuda)
    gevp.inject_failure(1)
    with pytest.raises(gevp.GevpError) as e:
        gevp.heev_small(G)
    assert e.value.name == "GEVP_ERR_TIMEOUT"
    gevp.heev_small(G)


@pytest.mark.parametrize("n,m", [(64, 8), (800, 64)])   # products on the FP64 pipe, and emulated
def test_rayleigh_ritz(cuda, n, m):
    from paper_1007_4400_gb300 import gevp
    C = _herm(n, cuda)
    Q = torch.linalg.qr(torch.randn(n, m, dtype=torch.complex128, device=cuda))[0].contiguous()
    gevp.inject_failure(1)
    with pytest.raises(gevp.GevpError) as e:
        gevp.rayleigh_ritz(C, Q.clone())
    assert e.value.name == "GEVP_ERR_TIMEOUT"
    gevp.rayleigh_ritz(C, Q.clone())


def test_gradient_products(cuda):
    """The gradient's call does not wait: its own results are NaN, and the failure is not reported by
    the next call that waits."""
    from paper_1007_4400_gb300 import gevp
    n, nev = 1024, 64
    X = torch.randn(n, nev, dtype=torch.complex128, device=cuda)
    lam = torch.linspace(-1, 1, nev, dtype=torch.float64, device=cuda)
    ref = gevp.energy_backward(X, lam)
    gevp.inject_failure(2)
    for G in gevp.energy_backward(X, lam):
        assert torch.isnan(G.real).all()
    gevp.cholqr2(X.clone())
    for G, R in zip(gevp.energy_backward(X, lam), ref):
        assert torch.equal(torch.view_as_real(G), torch.view_as_real(R))


def test_products_that_wait(cuda):
    from paper_1007_4400_gb300 import gevp
    X = torch.randn(2048, 128, dtype=torch.complex128, device=cuda)   # Gram matrix emulated
    for call in (lambda: gevp.cholqr2(X.clone()), lambda: gevp.zgemm_emulated(X, X, opA="C", opB="N")):
        gevp.inject_failure(2)
        with pytest.raises(gevp.GevpError) as e:
            call()
        assert e.value.name == "GEVP_ERR_TIMEOUT"
        call()

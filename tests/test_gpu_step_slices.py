"""Which pipe the products of the per-step calls take: the emulated one by default, the FP64 pipe for
a caller that asks for it, and, in the gradient, for rows whose entries spread over decades (there an
entry far below the rows' largest ones would lose what the FP64 sum keeps)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def emulated(call):
    """(result, number of emulated products in the call)"""
    from paper_1007_4400_gb300 import gevp
    torch.cuda.synchronize()
    gevp.kernel_timing(True)
    r = call()
    torch.cuda.synchronize()
    n = gevp.kernel_timing_read()["oz_gemm_kernel"]["launches"]
    gevp.kernel_timing(False)
    return r, n


def block(kind, n, nev, device):
    g = torch.Generator(device=device).manual_seed(n)
    X = torch.randn(n, nev, dtype=torch.complex128, device=device, generator=g)
    if kind == "halves":       # each row large in one half of the columns, in the other 1e-9 or 1e-12
        X[: n // 2, nev // 2:] *= 1e-9
        X[n // 2:, : nev // 2] *= 1e-12
    if kind == "one row":
        X[n - 1, : nev // 2] *= 1e-11
    if kind == "rows":         # rows of any length are even
        X *= torch.logspace(-8, 3, n, dtype=torch.float64, device=device)[:, None]
    return X


# 1537: not a multiple of any tile; 200 columns: more than a warp's share of a row
@pytest.mark.parametrize("n,nev", [(1024, 64), (1537, 200)])
@pytest.mark.parametrize("kind", ["even", "rows", "halves", "one row"])
def test_gradient_entries(cuda, kind, n, nev):
    from paper_1007_4400_gb300 import gevp
    X = block(kind, n, nev, cuda)
    lam = torch.linspace(-2, 5, nev, dtype=torch.float64, device=cuda)
    (GA, GB), launched = emulated(lambda: gevp.energy_backward(X, lam))
    assert launched > 0
    # reference entries in extended precision, of rows from both halves
    rows = np.r_[0:3, n // 2 - 1:n // 2 + 2, n - 3:n]
    Xs = X[torch.from_numpy(rows).to(cuda)].cpu().numpy()
    re, im = Xs.real.astype(np.longdouble), Xs.imag.astype(np.longdouble)
    l = lam.cpu().numpy().astype(np.longdouble)
    a = np.abs(Xs)
    pick = np.ix_(rows, rows)
    u = 2.0 ** -53
    for G, w in ((GA, np.ones_like(l)), (GB, -l)):
        G = G.cpu().numpy()[pick]
        rr = (re * w) @ re.T + (im * w) @ im.T
        ii = (im * w) @ re.T - (re * w) @ im.T
        # the bound of an FP64 sum of 4 nev products. Even rows are emulated: their 2 nev roundings of
        # 2^-57 of the rows' largest entries m_i m_j, with the factor 4 that gevp.h gives
        bound = 4 * nev * u * ((a * np.abs(w).astype(float)) @ a.T)
        if kind in ("even", "rows"):
            m = a.max(axis=1)
            bound = bound + 2 * nev * 2.0 ** -52 * np.outer(m * np.abs(w).max().astype(float), m)
        assert np.all(np.abs(G.real - rr) <= bound) and np.all(np.abs(G.imag - ii) <= bound)


def test_fp64_on_request(cuda):
    from paper_1007_4400_gb300 import gevp, synth
    s = synth.make_sequence(4, 900, 1, 60, 24, device=cuda)
    X = torch.randn(2048, 160, dtype=torch.complex128, device=cuda)
    C = s.A[0]
    Q0 = torch.linalg.qr(torch.randn(900, 90, dtype=torch.complex128, device=cuda))[0].contiguous()
    lam = torch.linspace(-2, 5, 160, dtype=torch.float64, device=cuda)
    calls = [lambda k: gevp.cholqr2(X.clone(), want_R=True, slices=k),
             lambda k: gevp.rayleigh_ritz(C, Q0.clone(), slices=k),
             lambda k: gevp.energy_backward(X, lam, slices=k)]
    for call in calls:
        r8, n8 = emulated(lambda: call(8))
        r0, n0 = emulated(lambda: call(0))
        assert n8 > 0 and n0 == 0
        # columns of Q and W agree up to a phase: their moduli
        for a, b in zip(r8, r0):
            assert (a.abs() - b.abs()).abs().max().item() <= 1e-10 * b.abs().max().item()
    with pytest.raises(gevp.GevpError):
        call(7)


@pytest.mark.parametrize("slices", [0, 8])
def test_gradient_follows_the_solve(cuda, slices):
    from paper_1007_4400_gb300 import gevp, synth
    s = synth.make_sequence(4, 700, 1, 50, 20, device=cuda)
    A = s.A[0].clone().requires_grad_(True)
    B = s.B.clone().requires_grad_(True)
    E = gevp.band_energy(A, B, s.nev, nex=s.nex, reduce_slices=slices)
    _, launched = emulated(lambda: E.backward())
    assert (launched > 0) == (slices > 0)
    assert abs(float(torch.real(torch.sum(A.grad * s.B.T))) - s.nev) <= 1e-9 * s.nev

"""The work that a user of this library has it do, as cases that can be timed and compared.

Whole calls: an SCF-like sequence (`solve_sequence`), a batch of k-points
(`solve_batched`), the band energy with its gradients (`band_energy`, forward and
backward). Single steps, each through its own entry point: the reduction to standard form,
the emulated FP64 product, the Chebyshev filter in its two tensor-core modes, CholQR2, the
Rayleigh-Ritz projection, the small eigensolver.

Eigenvectors are fixed only up to a phase, so the solver cases return what an SCF program
forms from them next: the density matrix X X^H and the energy-weighted one, X diag(lambda)
X^H (`energy_backward`), which do not depend on the phases; the two projection cases return
the moduli of the vectors' entries (the amplitudes behind a state's density) for the same
reason. The tensor-core filter modes return complex128 that carries single or half
precision; the cases keep the result in a type of that precision.
"""
import math

import torch

from paper_1007_4400_gb300 import gevp

DEV = "cuda"


# ----------------------------------------------------------------------------- the cases
def listed():
    return [
        # bulk Cu in the paper: pencils of order about 50, where launches and host
        # synchronisations are the cost; the plain FP64 filter (the library's default)
        dict(name="seq_cu_n50", kind="seq", n=50, nev=12, nex=6, nprob=8, prec="fp64"),
        # the benchmark's SCF sequence (n 2048, nev 100, nex 40, FP32-class filter): a cold
        # problem and the warm ones after it
        dict(name="seq_scf_n2048", kind="seq", n=2048, nev=100, nex=40, nprob=6, prec="fp32"),
        # ragged k-points in lock step, as many SCF steps as the batch's graph needs to settle
        dict(name="kpoints_8x3", kind="batch", nk=8, lo=800, hi=1900, nsteps=3, prec="fp32"),
        # the differentiable band energy of one large problem, forward and backward
        dict(name="grad_n4096", kind="grad", n=4096, nev=200, nex=50, prec="fp32"),
        # the reduction to standard form at the precision workload's order (largest)
        dict(name="reduce_n6144", kind="reduce", n=6144, slices=8),
        # the same at an odd order, near the Fe multilayer's and the k-points' sizes
        dict(name="reduce_n777", kind="reduce", n=777, slices=8),
        # a block product with an n x n operand (C Q, A X, B X in every round): odd sizes
        dict(name="product_3001x181", kind="product", M=3001, N=181, K=3001, opA="N", opB="N", slices=8),
        # the Chebyshev filter of the benchmark's block, FP32-class
        dict(name="filter_fp32_n2048", kind="filter", n=2048, m=140, degree=16, prec="fp32"),
        # and in BF16, at an odd order and a block wider than one column tile
        dict(name="filter_bf16_n4100", kind="filter", n=4100, m=211, degree=8, prec="bf16"),
        # orthonormalisation of the benchmark's block
        dict(name="cholqr2_n2048", kind="cholqr", n=2048, m=140),
        # the projection of a block of a k-point's size
        dict(name="ritz_n1500", kind="ritz", n=1500, m=100),
        # the small eigensolver alone on the projection of the smallest workload
        # (n 512, nev 32, nex 16)
        dict(name="heev_m48", kind="heev", m=48),
    ]


def _logint(rng, lo, hi):
    """Log-uniform whole number, odd more often than not."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, v | 1) if rng.random() < 0.6 else v


def draw(rng):
    kind = rng.choice(["seq", "seq", "batch", "grad", "reduce", "reduce", "product", "product", "filter", "filter",
                       "cholqr", "ritz", "heev"])
    if kind == "seq":
        n = _logint(rng, 50, 2048)
        nev = max(4, int(n * rng.uniform(0.04, 0.2 if n < 400 else 0.07)))
        return dict(kind=kind, n=n, nev=nev, nex=max(3, int(nev * rng.uniform(0.25, 0.5))), nprob=rng.randint(2, 6),
                    prec=rng.choice(["fp64", "fp32"]) if n < 300 else rng.choice(["fp32", "fp32", "bf16"]))
    if kind == "batch":
        lo = _logint(rng, 300, 900)
        return dict(kind=kind, nk=rng.randint(2, 8), lo=lo, hi=lo + rng.randint(50, 900), nsteps=rng.randint(1, 3),
                    prec=rng.choice(["fp32", "fp32", "fp64"]) if lo < 400 else "fp32")
    if kind == "grad":
        n = _logint(rng, 400, 3500)
        nev = max(8, int(n * rng.uniform(0.03, 0.06)))
        return dict(kind=kind, n=n, nev=nev, nex=max(4, int(0.3 * nev)), prec="fp32")
    if kind == "reduce":
        n = _logint(rng, 60, 4500)
        return dict(kind=kind, n=n, slices=rng.choice([0, 8]) if n < 900 else 8)
    if kind == "product":
        K = _logint(rng, 100, 4000)
        thin = rng.random() < 0.6
        return dict(kind=kind, M=_logint(rng, 100, 4000), N=_logint(rng, 16, 400) if thin else _logint(rng, 200, 4000),
                    K=K, opA=rng.choice(["N", "C"]), opB=rng.choice(["N", "C"]), slices=8)
    if kind == "filter":
        n = _logint(rng, 300, 5000)
        return dict(kind=kind, n=n, m=min(n // 2, _logint(rng, 20, 360)), degree=rng.randint(4, 24),
                    prec=rng.choice(["fp32", "bf16"]))
    if kind == "cholqr":
        n = _logint(rng, 200, 5000)
        return dict(kind=kind, n=n, m=min(n // 4, _logint(rng, 16, 360)))
    if kind == "ritz":
        n = _logint(rng, 200, 2500)
        return dict(kind=kind, n=n, m=min(n // 6, _logint(rng, 12, 200)))
    return dict(kind="heev", m=_logint(rng, 8, 360))


# ----------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _cn(g, *shape):
    """Standard complex normal entries, E|z|^2 = 1."""
    return torch.randn(*shape, dtype=torch.complex128, device=DEV, generator=g)


def _unitary(g, n):
    """A dense random unitary as a map on the rows of a matrix and its inverse: diagonal
    phases around unitary Fourier transforms (a dense Haar draw by QR would cost more than
    the calls that are timed)."""
    ph = [torch.polar(torch.ones(n, dtype=torch.float64, device=DEV),
                      2 * math.pi * torch.rand(n, dtype=torch.float64, device=DEV, generator=g))[:, None]
          for _ in range(3)]

    def fwd(M):
        M = torch.fft.fft(ph[2] * M, dim=0, norm="ortho")
        return ph[0] * torch.fft.fft(ph[1] * M, dim=0, norm="ortho")

    return fwd


def _herm(M):
    return 0.5 * (M + M.conj().T)


def _factor(g, n):
    """The factor L of an overlap B = L L^H: diagonal in [0.5, 2], off-diagonal entries 0.3 / sqrt(n)."""
    L = torch.tril(_cn(g, n, n), -1) * (0.3 / math.sqrt(n))
    return L + torch.diag(0.5 + 1.5 * torch.rand(n, dtype=torch.float64, device=DEV, generator=g)).to(L.dtype)


def _spectrum(g, n, nocc):
    """Sorted levels in [-2, 50] with a gap of 0.05 above the occupied ones."""
    lam = -2 + 52 * torch.sort(torch.rand(n, dtype=torch.float64, device=DEV, generator=g)).values
    lam[nocc:] += 0.05
    return lam


def _pencil(g, n, nev):
    """(A, B, L, Q, lam) with A = L Q diag(lam) Q^H L^H, B = L L^H."""
    L, lam = _factor(g, n), _spectrum(g, n, nev)
    Q = _unitary(g, n)(torch.eye(n, dtype=torch.complex128, device=DEV))
    LQ = L @ Q
    A = _herm((LQ * lam.to(LQ.dtype)) @ LQ.conj().T).contiguous()
    return A, _herm(L @ L.conj().T).contiguous(), L, Q, lam


def _sequence(g, n, nev, nprob):
    """The slowly drifting problems of an SCF cycle: A_{l+1} = A_l + 0.1 0.6^l P_l, P_l Hermitian of norm about 1."""
    A, B, L, Q, lam = _pencil(g, n, nev)
    As = [A]
    for l in range(nprob - 1):
        As.append((As[-1] + (0.1 * 0.6 ** l / math.sqrt(2.0 * n)) * _herm(_cn(g, n, n))).contiguous())
    return As, B, L, Q, lam


def _kpoint_sizes(case):
    """Ragged orders spread over [lo, hi], nev = 0.06 n, nex = 0.4 nev."""
    out = []
    for k in range(case["nk"]):
        n = case["lo"] + int((case["hi"] - case["lo"]) * ((0.38 + 0.618034 * k) % 1.0))
        nev = max(4, round(0.06 * n))
        out.append((n, nev, math.ceil(0.4 * nev)))
    return out


def _block(g, n, m):
    """A filtered block: columns of different lengths, moderately dependent."""
    Y = _cn(g, n, m) @ (torch.eye(m, dtype=torch.complex128, device=DEV) + 0.2 * _cn(g, m, m) / math.sqrt(m))
    return (Y * torch.logspace(-1.5, 1.5, m, dtype=torch.float64, device=DEV)).contiguous()


def _make(case, seed):
    """Everything that a case's inputs are made of, the parts that only exact() needs among them."""
    g = _gen(seed)
    kind = case["kind"]
    if kind == "seq":
        return _sequence(g, case["n"], case["nev"], case["nprob"])
    if kind == "batch":
        return [_sequence(g, n, nev, case["nsteps"]) for n, nev, _ in _kpoint_sizes(case)]
    if kind == "grad":
        return _pencil(g, case["n"], case["nev"])
    if kind == "reduce":
        n = case["n"]
        # an overlap near the identity (eigenvalues in about [0.4, 1.6]) with scaled functions
        d = 0.5 + 1.5 * torch.rand(n, dtype=torch.float64, device=DEV, generator=g)
        S = _herm(_cn(g, n, n)) * (0.6 / math.sqrt(2.0 * n))
        S.diagonal().fill_(1.0)
        return _herm(_cn(g, n, n)).contiguous(), (d[:, None] * S * d).contiguous()
    if kind == "product":
        a = (case["M"], case["K"]) if case["opA"] == "N" else (case["K"], case["M"])
        b = (case["K"], case["N"]) if case["opB"] == "N" else (case["N"], case["K"])
        return _cn(g, *a), _cn(g, *b)
    if kind in ("filter", "ritz"):
        n, m = case["n"], case["m"]
        fwd = _unitary(g, n)
        lam = _spectrum(g, n, m)
        if kind == "ritz":  # levels apart from each other: the vectors are then well defined
            lam[:m] = torch.linspace(-2, 5, m, dtype=torch.float64, device=DEV)
            lam[m:] = lam[m:].clamp(min=5.05)
        V = fwd(torch.eye(n, dtype=torch.complex128, device=DEV))
        C = _herm((V * lam.to(V.dtype)) @ V.conj().T).contiguous()
        if kind == "filter":
            return C, _cn(g, n, m), lam
        # an orthonormal block close to the lowest eigenvectors, mixed among itself
        mix = torch.linalg.qr(_cn(g, m, m))[0]
        return C, torch.linalg.qr(V[:, :m] @ mix + 0.02 * _cn(g, n, m) / math.sqrt(n))[0].contiguous(), lam
    if kind == "cholqr":
        return (_block(g, case["n"], case["m"]),)
    m = case["m"]
    V = torch.linalg.qr(_cn(g, m, m))[0]
    lam = torch.linspace(-2, 5, m, dtype=torch.float64, device=DEV)
    lam = lam + (2.0 / max(m, 2)) * (torch.rand(m, dtype=torch.float64, device=DEV, generator=g) - 0.5)
    return (_herm((V * lam.to(V.dtype)) @ V.conj().T).contiguous(),)


def prepare(case, seed):
    x = _make(case, seed)
    kind = case["kind"]
    if kind == "seq":
        return dict(case=case, A=x[0], B=x[1])
    if kind == "batch":
        sizes = _kpoint_sizes(case)
        return dict(case=case, A=[s[0] for s in x], B=[s[1] for s in x], nev=[s[1] for s in sizes],
                    nex=[s[2] for s in sizes])
    if kind == "grad":
        return dict(case=case, A=x[0].requires_grad_(True), B=x[1].requires_grad_(True))
    if kind == "filter":
        return dict(case=case, C=x[0], Y=x[1], interval=_interval(case, x[2]))
    return dict(case=case, x=x)


def _interval(case, lam):
    """(lo, hi, s) of the filter: damp everything above the block's own levels."""
    m = case["m"]
    return float(0.5 * (lam[m - 1] + lam[m])), float(lam[-1]) + 0.1, float(lam[0])


# ----------------------------------------------------------------------------- the passes
_LOW = {"fp32": lambda Y: Y.to(torch.complex64), "bf16": lambda Y: torch.view_as_real(Y).to(torch.bfloat16)}


def _tight(case):
    """The residual that an SCF program near its end asks for."""
    return dict(tol=1e-12, filter_prec=case["prec"])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "seq":
        r = gevp.solve_sequence(state["A"], state["B"], case["nev"], nex=case["nex"], **_tight(case))
        P, W = gevp.energy_backward(r.X, r.Lambda[-1])
        return dict(Lambda=list(r.Lambda), P=P, W=W)
    if kind == "batch":
        r = gevp.solve_batched(state["A"], state["B"], state["nev"], nex=state["nex"], **_tight(case))
        return [dict(Lambda=list(lam), P=gevp.energy_backward(X, lam[-1])[0]) for lam, X in zip(r.Lambda, r.X)]
    if kind == "grad":
        A, B = state["A"], state["B"]
        A.grad = B.grad = None
        E = gevp.band_energy(A, B, case["nev"], nex=case["nex"], **_tight(case))
        E.backward()
        return dict(E=E.detach(), GA=A.grad, GB=B.grad)
    if kind == "filter":
        # the filter works in place: the program keeps its block and filters a copy
        return _LOW[case["prec"]](gevp.chebyshev_filter(state["C"], state["Y"].clone(), case["degree"],
                                                        *state["interval"], prec=case["prec"]))
    x = state["x"]
    if kind == "reduce":
        return list(gevp.reduce(x[0], x[1], slices=case["slices"]))
    if kind == "product":
        return gevp.zgemm_emulated(x[0], x[1], slices=case["slices"], opA=case["opA"], opB=case["opB"])
    if kind == "cholqr":
        return list(gevp.cholqr2(x[0].clone(), want_R=True))
    if kind == "ritz":
        th, Q, W, res = gevp.rayleigh_ritz(x[0], x[1].clone())
        return [th, Q.abs(), W.abs(), res]
    th, Z = gevp.heev_small(x[0])
    return [th, Z.abs()]


# ----------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    """16-byte entries, 8 flop per complex multiply-add. The solver's count is one reduction,
    three filter steps of degree 16, projections and the final check per problem."""
    kind = case["kind"]

    def solve(n, nev, nex, nprob):
        m = nev + nex
        fl = nprob * (4.0 * n ** 3 + 8.0 * n * n * (20.0 * m + 2.5 * nev)) + 8.0 / 3 * n ** 3
        return 16.0 * n * n * (nprob + 1) + 8.0 * nprob * nev, fl

    if kind == "seq":
        n, nev = case["n"], case["nev"]
        b, f = solve(n, nev, case["nex"], case["nprob"])
        return dict(bytes=b + 32.0 * n * n, flops=f + 8.0 * n * n * nev)
    if kind == "batch":
        b = f = 0.0
        for n, nev, nex in _kpoint_sizes(case):
            p, q = solve(n, nev, nex, case["nsteps"])
            b, f = b + p + 16.0 * n * n, f + q + 4.0 * n * n * nev
        return dict(bytes=b, flops=f)
    if kind == "grad":
        n, nev = case["n"], case["nev"]
        b, f = solve(n, nev, case["nex"], 1)
        return dict(bytes=b + 32.0 * n * n, flops=f + 8.0 * n * n * nev)
    if kind == "reduce":
        n = case["n"]
        return dict(bytes=64.0 * n * n, flops=(4.0 + 8.0 / 3) * n ** 3)
    if kind == "product":
        M, N, K = case["M"], case["N"], case["K"]
        return dict(bytes=16.0 * (M * K + K * N + M * N), flops=8.0 * M * N * K)
    if kind == "filter":
        n, m = case["n"], case["m"]
        out = 8.0 if case["prec"] == "fp32" else 4.0
        return dict(bytes=16.0 * n * n + (16.0 + out) * n * m, flops=8.0 * n * n * m * case["degree"])
    if kind == "cholqr":
        n, m = case["n"], case["m"]
        return dict(bytes=32.0 * n * m + 16.0 * m * m, flops=16.0 * n * m * m)
    if kind == "ritz":
        n, m = case["n"], case["m"]
        return dict(bytes=16.0 * n * n + 32.0 * n * m, flops=8.0 * n * n * m + 24.0 * n * m * m)
    m = case["m"]
    return dict(bytes=24.0 * m * m, flops=36.0 * m ** 3)


# ----------------------------------------------------------------------------- the same in plain 64-bit torch
def _occupied(A, B, nev):
    """(lambda, X) of the lowest nev pairs of A x = lambda B x."""
    L = torch.linalg.cholesky(B)
    T = torch.linalg.solve_triangular(L, A, upper=False)
    C = torch.linalg.solve_triangular(L, T.conj().T.contiguous(), upper=False)
    lam, V = torch.linalg.eigh(_herm(C))
    return lam[:nev], torch.linalg.solve_triangular(L.conj().T, V[:, :nev], upper=True)


def _solved(As, B, L, Q, lam, nev):
    """Rows of eigenvalues (problem 0 by construction, the last one solved, the rest None) and the last X."""
    if len(As) == 1:
        last, X = lam[:nev], torch.linalg.solve_triangular(L.conj().T, Q[:, :nev], upper=True)
        return [last], X
    last, X = _occupied(As[-1], B, nev)
    return [lam[:nev]] + [None] * (len(As) - 2) + [last], X


def _density(X, w=None):
    return ((X if w is None else X * w.to(X.dtype)) @ X.conj().T)


def exact(case, seed):
    x = _make(case, seed)
    kind = case["kind"]
    if kind == "seq":
        rows, X = _solved(*x, case["nev"])
        return dict(Lambda=rows, P=_density(X), W=-_density(X, rows[-1]))
    if kind == "batch":
        out = []
        for s, (_, nev, _) in zip(x, _kpoint_sizes(case)):
            rows, X = _solved(*s, nev)
            out.append(dict(Lambda=rows, P=_density(X)))
        return out
    if kind == "grad":
        A, B, L, Q, lam = x
        nev = case["nev"]
        X = torch.linalg.solve_triangular(L.conj().T, Q[:, :nev], upper=True)
        return dict(E=lam[:nev].sum(), GA=_density(X), GB=-_density(X, lam[:nev]))
    if kind == "reduce":
        L = torch.linalg.cholesky(x[1])
        T = torch.linalg.solve_triangular(L, x[0], upper=False)
        return [L, _herm(torch.linalg.solve_triangular(L, T.conj().T.contiguous(), upper=False))]
    if kind == "product":
        a = x[0] if case["opA"] == "N" else x[0].conj().T
        b = x[1] if case["opB"] == "N" else x[1].conj().T
        return a @ b
    if kind == "filter":
        C, Y, lam = x
        lo, hi, s = _interval(case, lam)
        c, e = 0.5 * (hi + lo), 0.5 * (hi - lo)
        sigma1 = e / (s - c)
        sigma, prev, cur = sigma1, Y, (C @ Y - c * Y) * (sigma1 / e)
        for _ in range(case["degree"] - 1):
            new = 1.0 / (2.0 / sigma1 - sigma)
            prev, cur = cur, (C @ cur - c * cur) * (2.0 * new / e) - (sigma * new) * prev
            sigma = new
        return cur if case["prec"] == "fp32" else torch.view_as_real(cur)
    if kind == "cholqr":
        Q, R = torch.linalg.qr(x[0])
        ph = R.diagonal() / R.diagonal().abs()
        return [Q * ph, R * ph.conj()[:, None]]
    if kind == "ritz":
        C, Q, _ = x
        W = C @ Q
        th, Z = torch.linalg.eigh(_herm(Q.conj().T @ W))
        Q, W = Q @ Z, W @ Z
        return [th, Q.abs(), W.abs(), torch.linalg.vector_norm(W - Q * th.to(Q.dtype), dim=0)]
    th, Z = torch.linalg.eigh(x[0])
    return [th, Z.abs()]

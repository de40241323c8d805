"""The emulated FP64 product at the edges of its tiles and K chunks, its K slices, and the form
that keeps one group of moduli at a time, against exact integers and each other."""
import ctypes as C

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def ints(rng, bits, *shape):
    """Complex whole numbers below 2^bits."""
    return rng.integers(-2 ** bits, 2 ** bits + 1, shape) + 1j * rng.integers(-2 ** bits, 2 ** bits + 1, shape)


# 128 / 256: the rows of one CTA and of a pair; 32, 256: column tiles; 64: one K block; 512: one
# accumulation chunk; (64, 64, 1100): K slices; (9, 700, 24): three column tiles. 21-bit
# whole numbers: 43 + log2(2K) < 53 bits, so the FP64 result is exact and has to be equal.
@pytest.mark.parametrize("M,N,K", [(128, 32, 64), (129, 33, 65), (256, 256, 8), (257, 257, 511), (255, 31, 512),
                                   (1, 1, 513), (64, 64, 1100), (9, 700, 24), (300, 96, 1537)])
@pytest.mark.parametrize("opA,opB", [("N", "C"), ("C", "N")])
def test_integers_are_exact(cuda, M, N, K, opA, opB):
    from paper_1007_4400_gb300 import gevp
    rng = np.random.default_rng(M + 7 * N + 13 * K)
    a, b = ints(rng, 20, M, K), ints(rng, 20, K, N)
    A = a if opA == "N" else a.conj().T
    B = b if opB == "N" else b.conj().T
    # (a fresh tensor: numpy gives a matrix of one row any row stride)
    dev = lambda x: torch.empty(x.shape, dtype=torch.complex128, device=cuda).copy_(torch.from_numpy(x.copy()))
    D = gevp.zgemm_emulated(dev(A), dev(B), slices=8, opA=opA, opB=opB).cpu().numpy()
    assert np.array_equal(D, a @ b)


def test_groups_of_moduli_give_the_same_bits(cuda):
    """With device memory short, the operands' residues are kept a group of moduli at a time;
    the arithmetic is the same, so the results are equal bit for bit."""
    from paper_1007_4400_gb300 import gevp
    L = gevp.load()
    n, K = 2500, 2600
    A = torch.randn((n, K), dtype=torch.complex128, device=cuda)
    B = torch.randn((n, K), dtype=torch.complex128, device=cuda)
    full = gevp.zgemm_emulated(A, B)
    out = torch.empty_like(full)
    h = C.c_void_p()
    assert L.gevp_create(C.byref(h), 0, C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    # the residues of all 16 moduli take 2 * 64 n K = 830 MB next to at most 250 MB for the
    # result's; leave about 700 MB
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - 700 * 2 ** 20, dtype=torch.uint8, device=cuda)
    st = L.gevp_zgemm_emulated(h, 0, 1, n, n, K, C.c_void_p(A.data_ptr()), K, C.c_void_p(B.data_ptr()), K,
                               C.c_void_p(out.data_ptr()), n, 8)
    del hog
    torch.cuda.empty_cache()
    assert L.gevp_destroy(h) == 0
    assert st == 0
    assert torch.equal(out, full)

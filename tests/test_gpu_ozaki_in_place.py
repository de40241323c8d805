"""The emulated product with its result over an operand's memory, with all residues made first and in
groups of moduli over several panels of rows (where the operands are read again for each)."""
import ctypes as C

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("groups", [False, True])
@pytest.mark.parametrize("over", ["A", "B"])
def test_result_over_an_operand(cuda, over, groups):
    from paper_1007_4400_gb300 import gevp
    # 2 x 16 bytes of residues an entry and at most 1 GiB of them: two panels
    M, N, K = (6400, 6400, 300) if over == "A" else (6400, 6400, 6400)
    if over == "A":
        N = K          # D (M x K) over A
        M = 130000
    g = torch.Generator(device=cuda).manual_seed(5)
    A = torch.randn(M, K, dtype=torch.complex128, device=cuda, generator=g)
    B = torch.randn(K, N, dtype=torch.complex128, device=cuda, generator=g)
    ref = gevp.zgemm_emulated(A, B, opA="N", opB="N")
    for h in gevp._HANDLES.values():
        gevp.load().gevp_destroy(h)
    gevp._HANDLES.clear()
    if groups:
        gevp.inject_failure(4)
    h = gevp._handle(cuda)
    D = A if over == "A" else B
    st = gevp.load().gevp_zgemm_emulated(h, 0, 0, M, N, K, C.c_void_p(A.data_ptr()), K, C.c_void_p(B.data_ptr()), N,
                                         C.c_void_p(D.data_ptr()), N, 8)
    assert st == 0
    assert torch.equal(torch.view_as_real(D), torch.view_as_real(ref))

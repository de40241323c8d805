"""A non-finite A in one k-point with the products on the FP64 pipe (reduce_slices = 0), where the
final check runs as grouped products whose item lists the plan holds: over two steps and two calls
on one plan, the other k-points converge and the bad one's next step does too."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_nonfinite_matrix_fp64_products(cuda, prec, bad):
    from paper_1007_4400_gb300 import gevp, synth
    seqs = synth.kpoint_batch(3, 2, device=cuda, sizes=[(150, 9, 4), (203, 12, 5), (261, 16, 7)])
    opts = dict(nex=[s.nex for s in seqs], filter_prec=prec, reduce_slices=0)
    args = ([s.A for s in seqs], [s.B for s in seqs], [s.nev for s in seqs])
    lam0 = [s.lam0[:s.nev] for s in seqs]
    seqs[2].A[0][5, 5] = bad
    for _ in range(2):
        r = gevp.solve_batched(*args, **opts)
        assert r.status == 3
        for k in range(3):
            res = r.resid[k].cpu().numpy()
            assert res[1].max() <= 1e-10
            if k < 2:
                assert res[0].max() <= 1e-10
                assert np.abs(r.Lambda[k][0].cpu().numpy() - lam0[k]).max() <= 2e-12 * np.abs(seqs[k].lam0).max()
        assert not np.isfinite(r.resid[2][0].cpu().numpy()).any()

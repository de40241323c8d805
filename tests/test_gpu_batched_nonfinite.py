"""A k-point whose A holds a NaN or Inf ends as not converged without holding up the batch: the other
k-points converge, and so does its own next step (finite again) after one restart of its block."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_nonfinite_matrix_of_one_kpoint(cuda, bad):
    from paper_1007_4400_gb300 import gevp, synth
    seqs = synth.kpoint_batch(3, 2, device=cuda, sizes=[(150, 9, 4), (203, 12, 5), (261, 16, 7)])

    def solve():
        return gevp.solve_batched([s.A for s in seqs], [s.B for s in seqs], [s.nev for s in seqs],
                                  nex=[s.nex for s in seqs], filter_prec="fp32")

    lam0 = [x[1].cpu().numpy() for x in solve().Lambda]
    seqs[1].A[0][5, 5] = bad
    r = solve()
    assert r.status == 3
    assert r.stats["orth_fallbacks"] <= 4
    for k in range(3):
        lam, res = r.Lambda[k].cpu().numpy(), r.resid[k].cpu().numpy()
        assert res[1].max() <= 1e-10 and np.abs(lam[1] - lam0[k]).max() <= 2e-12 * np.abs(lam0[k]).max()
        if k != 1:
            assert res[0].max() <= 1e-10
    assert not np.isfinite(r.resid[1][0].cpu().numpy()).any()

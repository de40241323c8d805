"""The k-point batch with its emulated products spread over streams: one k-point, as many as there are
streams, one more, and orders on both sides of the rule that chooses between the grouped FP64
products and the emulated ones. Against the same batch on the FP64 pipe (reduce_slices 0): both
converge to tol, so the eigenvalues agree to the sum of their bounds (2 * 1e-12 of the largest)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _solve(seqs, **kw):
    from paper_1007_4400_gb300 import gevp
    return gevp.solve_batched([s.A for s in seqs], [s.B for s in seqs], [s.nev for s in seqs],
                              nex=[s.nex for s in seqs], filter_prec="fp32", **kw)


@pytest.mark.parametrize("sizes", [[(139, 9, 4)], [(50, 5, 3)] * 2, [(300, 20, 12), (64, 5, 3), (131, 30, 17), (257, 6, 2)],
                                   [(97 + 7 * k, 6 + k, 3) for k in range(5)], [(200, 8, 4)] * 9])
def test_lanes_agree_with_the_fp64_pipe(cuda, sizes):
    from paper_1007_4400_gb300 import synth
    seqs = synth.kpoint_batch(len(sizes), 3, device=cuda, sizes=sizes)
    r0 = _solve(seqs, reduce_slices=0)
    r8 = _solve(seqs, reduce_slices=8)
    r8b = _solve(seqs, reduce_slices=8)   # the captured round again
    for r in (r0, r8, r8b):
        assert r.status == 0 and r.stats["max_resid"] <= 1e-10
    for k in range(len(sizes)):
        a = r0.Lambda[k].cpu().numpy()
        for r in (r8, r8b):
            assert np.abs(a - r.Lambda[k].cpu().numpy()).max() <= 2e-12 * np.abs(a).max()

"""Scratch of the emulated products that cannot be had for all moduli at once (injected on the host):
the results are the same, whichever of the two streams it concerns, and the next call tries again."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def new_handle():
    """The next call makes a handle without scratch."""
    from paper_1007_4400_gb300 import gevp
    for h in gevp._HANDLES.values():
        gevp.load().gevp_destroy(h)
    gevp._HANDLES.clear()


@pytest.mark.parametrize("what", [3, 4])
def test_sequence_in_groups_of_moduli(cuda, what):
    """Four problems with one B: the later ones' standard forms are built on the second stream from the
    residues of L^-1 that the first stream's scratch holds."""
    from paper_1007_4400_gb300 import gevp, synth
    s = synth.make_sequence(1, 601, 4, 30, 12, device=cuda)
    new_handle()
    gevp.inject_failure(what)
    r = gevp.solve_sequence(s.A, s.B, s.nev, nex=s.nex, filter_prec="fp32")
    ref = gevp.solve_sequence(s.A, s.B, s.nev, nex=s.nex, filter_prec="fp32")
    assert r.status == 0 and ref.status == 0
    assert r.resid.max().item() <= 1e-10
    assert [x["outer_iters"] for x in r.stats] == [x["outer_iters"] for x in ref.stats]
    scale = np.abs(s.lam0).max()
    assert np.abs(r.Lambda[0].cpu().numpy() - s.lam0[:s.nev]).max() <= 1e-12 * scale
    assert (r.Lambda - ref.Lambda).abs().max().item() <= 1e-12 * scale


def test_next_call_tries_again(cuda):
    from paper_1007_4400_gb300 import gevp, synth
    n = 1500
    s = synth.make_sequence(1, n, 1, 20, 8, device=cuda)

    def kept():
        gevp.solve_sequence(s.A, s.B, s.nev, nex=s.nex, filter_prec="fp32")
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    new_handle()
    gevp.inject_failure(3)
    free_lean = kept()
    free_full = kept()
    # six operands of 64 bytes an entry against 16
    assert free_lean - free_full >= 0.9 * 6 * 48 * n * n
    assert abs(kept() - free_full) <= 64 << 20

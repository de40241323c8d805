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


def test_sequence_and_batch_give_each_other_up(cuda):
    from paper_1007_4400_gb300 import gevp, synth
    s = synth.make_sequence(1, 400, 3, 20, 8, device=cuda)
    ks = synth.kpoint_batch(2, 2, device=cuda, sizes=[(200, 12, 5), (261, 16, 7)])

    def sequence():
        r = gevp.solve_sequence(s.A, s.B, s.nev, nex=s.nex, filter_prec="fp32")
        assert r.status == 0 and r.resid.max().item() <= 1e-10
        assert np.abs(r.Lambda[0].cpu().numpy() - s.lam0[:s.nev]).max() <= 1e-12 * np.abs(s.lam0).max()

    def batch():
        r = gevp.solve_batched([x.A for x in ks], [x.B for x in ks], [x.nev for x in ks],
                               nex=[x.nex for x in ks], filter_prec="fp32")
        assert r.status == 0
        for x, lam, res in zip(ks, r.Lambda, r.resid):
            assert res.max().item() <= 1e-10
            assert np.abs(lam[0].cpu().numpy() - x.lam0[:x.nev]).max() <= 1e-12 * np.abs(x.lam0).max()
        return r.stats["graph_replays"]

    new_handle()
    batch()
    gevp.inject_failure(5)
    sequence()              # the plan is given up
    batch()
    assert batch() > 0      # and made again, its round captured
    new_handle()
    sequence()
    gevp.inject_failure(5)
    batch()                 # the sequence's scratch is given up
    sequence()
    # nothing to give up: the error, and the handle works on
    new_handle()
    gevp.inject_failure(5)
    with pytest.raises(gevp.GevpError) as e:
        sequence()
    assert e.value.name == "GEVP_ERR_OOM"
    sequence()
    batch()

"""A batch of another shape replaces the handle's plan: all of the old one's memory comes back."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_plans_do_not_pile_up(cuda):
    from paper_1007_4400_gb300 import gevp, synth
    # 96 k-points have item lists of more than a megabyte, which no other allocation absorbs
    seqs = synth.kpoint_batch(96, 1, device=cuda, sizes=[(24, 3, 2)] * 96)

    def free_after(nev):
        gevp.solve_batched([s.A for s in seqs], [s.B for s in seqs], nev, nex=2)
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    free_after(3)
    first = free_after(4)
    for nev in (3, 4) * 12:
        last = free_after(nev)
    assert first - last <= 8 << 20

"""Which grouped products of a batch take tiles of 4 x 8, whose sums have another order than the larger
ones', follows from the shapes: the same in every plan, whatever the tuning runs measured."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,slices", [("fp64", 8), ("fp64", 0), ("fp32", 8)])
@pytest.mark.parametrize("sizes", [[(30, 4, 3)] * 6, [(150 + 9 * i, 12, 5) for i in range(16)],
                                   [(500 + 60 * i, 34, 13) for i in range(3)]])
def test_small_tiles_do_not_depend_on_timing(cuda, sizes, prec, slices):
    from paper_1007_4400_gb300 import gevp, synth
    seqs = synth.kpoint_batch(len(sizes), 1, device=cuda, sizes=sizes)
    seen = set()
    for _ in range(3):
        for h in gevp._HANDLES.values():   # a new handle makes and tunes a new plan
            gevp.load().gevp_destroy(h)
        gevp._HANDLES.clear()
        r = gevp.solve_batched([s.A for s in seqs], [s.B for s in seqs], [s.nev for s in seqs],
                               nex=[s.nex for s in seqs], filter_prec=prec, reduce_slices=slices)
        assert r.status == 0
        seen.add(tuple(t == 0 for t in r.stats["tile"]))
    assert len(seen) == 1

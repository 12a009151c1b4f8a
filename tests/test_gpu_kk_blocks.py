"""Kramers-Kronig stage: batches that take each number of blocks per problem."""
import pytest

from paper_2407_20469_gb300 import apic, learn, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile,sizes", [(128, (1, 5, 10)), (256, (1, 2, 5, 10, 38)), (512, (1, 2, 5, 10, 19))])
def test_each_number_of_blocks_per_problem(tile, sizes):
    """With 8 problems a tile and 152, 76, 36 and 15 at once, the sizes take 8, 4, 2 and 1 blocks
    per problem (4, 2, 1 at 128 pixels) by the fewest rounds times the time of one, the last at 256
    two rounds of one; all give the spectra of the largest batch."""
    n = max(sizes)
    plan = apic.Plan.from_illumination(tile, synth.illumination(), max_tiles=n)
    _, zern, blank = learn.draw_tiles(n, 3, learn.field_table())
    I = learn.simulate(plan, zern, blank, 3)
    shape = (plan.info.n_bf, plan.info.n_pupil, 2)
    ref = torch.empty((n,) + shape, device="cuda")
    plan.kk_spectra(n, I, ref)
    assert bool(torch.isfinite(ref).all()) and float(ref.abs().max()) > 0
    for k in sizes:
        x = torch.zeros((k,) + shape, device="cuda")
        plan.kk_spectra(k, I[:k].contiguous(), x)
        assert torch.equal(x, ref[:k]), k

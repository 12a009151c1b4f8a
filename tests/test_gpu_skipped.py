"""Darkfield batches above one wave of blocks, with tiles to skip: full waves and the rounds
of clusters behind them take the tiles to solve from a list, or one launch takes them all
from a counter."""
import numpy as np
import pytest

from paper_2407_20469_gb300 import apic, learn, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

UNIQUE = 7


def _stage(tile, extra):
    """Plan, inputs of the darkfield stage for a wave and `extra` tiles (UNIQUE different ones in
    turn), and the solved spectra of the different ones, from a batch of their own."""
    ill = synth.illumination_8_24() if tile == 512 else synth.illumination()
    n = apic.Plan.from_illumination(tile, ill, max_tiles=1).info.df_wave + extra
    plan = apic.Plan.from_illumination(tile, ill, max_tiles=n)
    info = plan.info
    _, zern, _ = learn.draw_tiles(UNIQUE, 3, learn.field_table())
    I = learn.simulate(plan, zern, np.zeros(UNIQUE, dtype=bool), 3)
    x = torch.empty((UNIQUE, info.n_bf, info.n_pupil, 2), device="cuda")
    z = torch.empty((UNIQUE, 15), device="cuda")
    spec = torch.empty((UNIQUE, info.n_aperture, 2), device="cuda")
    plan.kk_spectra(UNIQUE, I, x)
    plan.aberration(UNIQUE, x, z)
    plan.stitch(UNIQUE, x, z, spec)
    ref = spec.clone()
    plan.darkfield(UNIQUE, I, z, ref)
    pick = torch.arange(n, device="cuda") % UNIQUE
    return plan, n, I[pick].contiguous(), z[pick].contiguous(), spec[pick].contiguous(), ref[pick]


@pytest.mark.parametrize("tile,extra", [(128, 20), (128, 100), (256, 1), (256, 30), (256, 60), (256, 120), (512, 20),
                                        (512, 140)])
@pytest.mark.parametrize("share", [None, 0.0, 0.3, 0.97, 1.0])
def test_waves_and_rounds_solve_the_tiles_that_are_not_skipped(tile, extra, share):
    """Each tile that is not skipped is solved as in a batch of UNIQUE tiles, bit for bit; the
    spectrum of a skipped one and every status stay as they were. share: of skipped tiles, None:
    no status given."""
    plan, n, I, z, spec, ref = _stage(tile, extra)
    skip = torch.as_tensor(np.random.default_rng(n).random(n) < (share or 0.0), device="cuda")
    st0 = torch.where(skip, torch.where(torch.arange(n, device="cuda") % 2 == 0, apic.APIC_TILE_BACKGROUND,
                                        apic.APIC_TILE_BADINPUT), 0).to(torch.int32)
    st = None if share is None else st0.clone()
    out = spec.clone()
    plan.darkfield(n, I, z, out, st)
    torch.cuda.synchronize()
    assert torch.equal(out, torch.where(skip[:, None, None], spec, ref))
    assert st is None or torch.equal(st, st0)


@pytest.mark.parametrize("tile", [128, 256])
def test_skipped_tiles_take_no_round(tile):
    """A wave and 88 tiles with two fifths skipped, fewer to solve than one wave, take the time of
    those alone, not that of two rounds (twice as much)."""
    plan, n, I, z, spec, _ = _stage(tile, 88)
    skip = torch.arange(n, device="cuda") % 5 < 2
    keep = torch.nonzero(~skip)[:, 0]
    assert len(keep) < n - 88

    def ms(n, I, z, spec, st0):
        best = float("inf")
        for _ in range(4):
            s, st = spec.clone(), st0.clone()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            plan.darkfield(n, I, z, s, st)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    flags = skip.to(torch.int32) * apic.APIC_TILE_BACKGROUND
    mixed = ms(n, I, z, spec, flags)
    alone = ms(len(keep), I[keep].contiguous(), z[keep].contiguous(), spec[keep].contiguous(), flags[keep])
    assert mixed < 1.3 * alone, (mixed, alone)


def test_list_of_tiles_replays_from_a_graph():
    """The list is made on the device, so a replay follows the status it finds."""
    plan, n, I, z, spec, ref = _stage(128, 20)
    out, st = spec.clone(), torch.zeros(n, dtype=torch.int32, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        plan.darkfield(n, I, z, out, st)
    for step in (3, 5):
        skip = torch.arange(n, device="cuda") % step == 0
        out.copy_(spec)
        st.copy_(skip.to(torch.int32) * apic.APIC_TILE_BACKGROUND)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, torch.where(skip[:, None, None], spec, ref))

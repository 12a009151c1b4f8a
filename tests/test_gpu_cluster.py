"""Small batches: the darkfield solves of a tile spread over a cluster of blocks.

A batch below a full wave is solved in rounds of several blocks per tile, the number
chosen by the batch size. Covered here: every choice at each tile size, rounds of
different kinds within one batch and graph replay.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2407_20469_gb300 import apic, learn, synth  # noqa: E402

pytestmark = pytest.mark.gpu

def _run(plan, I, n):
    H = plan.info.out_h
    f = torch.full((n, H, 2 * H), 7.0, dtype=torch.float32, device="cuda")
    z = torch.empty((n, 15), dtype=torch.float32, device="cuda")
    st = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    plan.reconstruct_batch(n, I[:n].contiguous(), f, z, None, st)
    torch.cuda.synchronize()
    return f, z, st


def _tiles(tile, ill, n, up=2):
    plan = apic.Plan.from_illumination(tile, ill, max_tiles=n, upsample=up)
    uv, zern, blank = learn.draw_tiles(n, 3, learn.field_table())
    if up == 2:
        return plan, learn.simulate(plan, zern, blank, 3)
    p2 = apic.Plan.from_illumination(tile, ill, max_tiles=1)
    return plan, learn.simulate(p2, zern, blank, 3)


@pytest.mark.parametrize("tile,ill,up,sizes", [
    (64, "8+16", 2, (1, 40, 100)),
    (128, "8+16", 2, (1, 7, 20, 37, 60, 100)),
    (256, "8+16", 2, (1, 9, 20, 33, 45, 60, 100)),
    (256, "12+22", 3, (2, 30)),
    (512, "8+24", 2, (1, 9, 24, 30, 50)),
])
def test_batch_size_does_not_change_a_tile(tile, ill, up, sizes):
    """The tiles of a small batch (clusters of every size in use, rounds of different sizes)
    are bit for bit those of a full wave (one block per tile)."""
    il = {"8+16": synth.illumination, "8+24": synth.illumination_8_24, "12+22": synth.illumination_12_22}[ill]()
    W = apic.Plan.from_illumination(tile, il, max_tiles=1).info.df_wave
    plan, I = _tiles(tile, il, W, up)
    f_ref, z_ref, s_ref = _run(plan, I, W)
    assert int(s_ref.max()) == 0
    for n in sizes:
        f, z, st = _run(plan, I, n)
        assert torch.equal(z, z_ref[:n]) and torch.equal(st, s_ref[:n]), n
        assert torch.equal(f, f_ref[:n]), n


@pytest.mark.parametrize("mx,my", [(192, 192), (192, 144), (192, 128), (192, 96), (160, 128), (160, 96), (144, 144)])
def test_every_solve_grid_in_a_cluster(mx, my):
    """Each (row, column) grid of the 256-pixel solve, forced on every image it is exact for:
    one tile (a cluster) against the same tile in a full wave."""
    ill = synth.illumination()
    W = apic.Plan.from_illumination(256, ill, max_tiles=1).info.df_wave
    plan, I = _tiles(256, ill, W)
    for i in range(plan.info.n_df):
        try:
            plan.set_df_grid(i, mx, my)
        except apic.ApicError:
            pass
    assert any(plan.df_grid(i)[1:] == (mx, my) for i in range(plan.info.n_df))
    f_ref, _, _ = _run(plan, I, W)
    f, _, _ = _run(plan, I, 1)
    assert torch.equal(f[0], f_ref[0])


def test_skipped_tiles_in_a_cluster_round():
    """Background tiles leave their cluster at once; the others are what they are alone."""
    ill = synth.illumination()
    T = 11
    zern = learn.coefficients(learn.field_table(), np.zeros((T, 2), np.float32))
    blank = np.zeros(T, dtype=bool)
    blank[::3] = True
    plan = apic.Plan.from_illumination(256, ill, max_tiles=T, bg_contrast=0.02, flags=apic.APIC_SKIP_BACKGROUND)
    I = learn.simulate(plan, zern, blank, 5)
    f, z, st = _run(plan, I, T)
    keep = torch.as_tensor(np.nonzero(~blank)[0], device="cuda")
    f1, z1, _ = _run(plan, I[keep], len(keep))
    assert torch.count_nonzero(f[torch.as_tensor(np.nonzero(blank)[0], device="cuda")]) == 0
    assert torch.equal(f[keep], f1) and torch.equal(z[keep], z1)


def test_cluster_round_replays_from_a_graph():
    ill = synth.illumination()
    plan, I = _tiles(128, ill, 3)
    f0, z0, _ = _run(plan, I, 3)
    f, z = torch.zeros_like(f0), torch.zeros_like(z0)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        plan.reconstruct_batch(3, I, f, z)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(f, f0) and torch.equal(z, z0)


@pytest.mark.parametrize("tile,sizes", [(64, (1, 30)), (128, (1, 3, 30)), (256, (1, 2, 4, 9, 30)), (512, (1, 4, 9, 20))])
def test_kramers_kronig_does_not_depend_on_the_blocks_per_problem(tile, sizes):
    """Batches of every size class (8 to 1 blocks per problem) and the allocation-free entry
    point (few grids, many blocks each) give the same spectra bit for bit."""
    ill = synth.illumination()
    n = max(sizes)
    plan, I = _tiles(tile, ill, n)
    shape = (plan.info.n_bf, plan.info.n_pupil, 2)
    ref = torch.empty((n,) + shape, device="cuda")
    plan.kk_spectra(n, I, ref)
    for k in sizes:
        x = torch.zeros((k,) + shape, device="cuda")
        plan.kk_spectra(k, I[:k].contiguous(), x)
        assert torch.equal(x, ref[:k]), k
        x.zero_()
        plan.kk_spectra_noalloc(k, I[:k].contiguous(), x)
        assert torch.equal(x, ref[:k]), k


@pytest.mark.parametrize("tile,ill", [(64, "8+16"), (256, "8+16"), (256, "12+22"), (512, "8+24")])
def test_background_does_not_depend_on_the_blocks_per_tile(tile, ill):
    """Eight blocks per tile (up to 64 tiles) and four: the same values and flags, a bad pixel
    found wherever it is, and the contrast of float64 sums. A thread sums q = npix / 2048 groups
    of four pixels in FP32: both means are within (q + 2) 2^-24 of exact, so the contrast c is
    within 3 (q + 2) 2^-24 (1 + c)."""
    il = {"8+16": synth.illumination, "8+24": synth.illumination_8_24, "12+22": synth.illumination_12_22}[ill]()
    n = 70
    plan, I = _tiles(tile, il, n)
    n_img, n_bf = plan.info.n_bf + plan.info.n_df, plan.info.n_bf
    I = I.reshape(n, n_img, tile, tile).clone()
    for t in range(n_img):
        I[t, t, -1, -1] = float("nan") if t % 2 else -1.0
    out = {}
    for k in (1, 9, 64, 65, n):
        c2 = torch.full((k,), -1.0, device="cuda")
        st = torch.full((k,), -1, dtype=torch.int32, device="cuda")
        plan.background(k, I[:k].contiguous(), c2, st)
        out[k] = c2, st
    for k in (1, 9, 64, 65):
        assert torch.equal(out[k][1], out[n][1][:k]), k
        assert torch.equal(out[k][0].view(torch.int32), out[n][0][:k].view(torch.int32)), k
    bad = (out[n][1] & apic.APIC_TILE_BADINPUT) != 0
    assert bad[:n_img].all() and not bad[n_img:].any()
    x = I[n_img:, :n_bf].double()
    m = x.mean((2, 3))
    c = (((x * x).mean((2, 3)) - m * m) / (m * m)).mean(1)
    q = max(1, tile * tile // 2048)
    assert ((out[n][0][n_img:].double() - c).abs() <= 3 * (q + 2) * 2.0 ** -24 * (1 + c)).all()


@pytest.mark.parametrize("tile,up,sizes", [(256, 2, (1, 16, 30, 60, 152, 200)), (512, 2, (1, 16, 30, 60, 152, 200)),
                                           (128, 2, (1, 3))])
def test_synthesis_does_not_depend_on_the_blocks_per_tile(tile, up, sizes):
    """Eight blocks per tile down to one: the same fields."""
    ill = synth.illumination()
    n = max(sizes)
    plan = apic.Plan.from_illumination(tile, ill, max_tiles=n, upsample=up)
    H, nap = plan.info.out_h, plan.info.n_aperture
    g = torch.Generator(device="cuda").manual_seed(1)
    spec = torch.randn((n, nap, 2), generator=g, device="cuda")
    ref = torch.empty((n, H, 2 * H), device="cuda")
    plan.synthesize(n, spec, ref)
    for k in sizes:
        f = torch.full((k, H, 2 * H), 7.0, device="cuda")
        plan.synthesize(k, spec[:k].contiguous(), f)
        assert torch.equal(f, ref[:k]), k
    # Parseval: the field's energy is the spectrum's, up to the transform's scale, for every tile alike
    e = ref.double().square().sum((1, 2)) / spec.double().square().sum((1, 2))
    assert float((e / e[0] - 1).abs().max()) < 1e-5


@pytest.mark.parametrize("tile,ill", [(64, "8+16"), (128, "12+22"), (256, "8+16")])
def test_aberration_does_not_depend_on_the_blocks_per_tile(tile, ill):
    """Two blocks per tile (up to a tile per SM) and one, a batch beyond the resident blocks:
    the same coefficients."""
    il = synth.illumination_12_22() if ill == "12+22" else synth.illumination()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 2 * sms + 3
    plan, I = _tiles(tile, il, n)
    x = torch.empty((n, plan.info.n_bf, plan.info.n_pupil, 2), device="cuda")
    plan.kk_spectra(n, I, x)
    ref = torch.empty((n, 15), device="cuda")
    plan.aberration(n, x, ref)
    assert bool(torch.isfinite(ref).all()) and float(ref[:, 3:].abs().max()) > 0.01
    for k in (1, 20, sms, sms + 1):
        z = torch.full((k, 15), 7.0, device="cuda")
        plan.aberration(k, x[:k].contiguous(), z)
        assert torch.equal(z, ref[:k]), k

"""512-pixel darkfield kernel: plans at the limit of its shared memory, intensities up to the limit of
FP32, autotuning on a few tiles."""
import ctypes as C

import numpy as np
import pytest

from helpers import as_complex, rel_l2
from paper_2407_20469_gb300 import apic, learn, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FIELD_TOL = 1e-3               # the workload's bar


@pytest.mark.parametrize("ill", [synth.illumination(8, ((0.29, 8, 0.0), (0.376, 8, 22.5))),
                                 synth.illumination(8, ((0.31, 8, 0.0), (0.392, 8, 22.5))),
                                 synth.illumination_12_22()])
def test_most_unknowns_that_fit_a_block(ill):
    """Images of up to 3933, 3940 and 3954 unknowns: their CG vectors leave no 2 KB of a block's
    shared memory beside the transforms, and the register kernel still takes them; its field is
    that of the shared-memory kernels."""
    plan = apic.Plan.from_illumination(512, ill, max_tiles=1)
    unknowns = max(int(plan.df_set(i, 0)[1][2]) for i in range(plan.info.n_df))
    assert 3902 < unknowns <= 3967
    I = learn.simulate(plan, learn.coefficients(learn.field_table(), np.zeros((1, 2), np.float32)),
                       np.zeros(1, dtype=bool), 5)
    assert plan.autotune(1, I)["darkfield_register"] > 0
    out = []
    for flags in (0, apic.APIC_LEGACY_KERNELS):
        plan = apic.Plan.from_illumination(512, ill, max_tiles=1, flags=flags)
        H = plan.info.out_h
        f = torch.zeros((1, H, 2 * H), device="cuda")
        z = torch.zeros((1, 15), device="cuda")
        st = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        plan.reconstruct_batch(1, I, f, z, None, st)
        torch.cuda.synchronize()
        assert int(st) == 0
        out.append(as_complex(f)[0])
    assert rel_l2(out[0], out[1]) < FIELD_TOL


def _stitched(tile, ill, n):
    """Plan, intensities, coefficients and stitched spectrum: the darkfield stage's inputs."""
    plan = apic.Plan.from_illumination(tile, ill, max_tiles=n)
    zern = learn.coefficients(learn.field_table(), np.zeros((n, 2), np.float32))
    I = learn.simulate(plan, zern, np.zeros(n, dtype=bool), 5)
    info = plan.info
    x = torch.empty((n, info.n_bf, info.n_pupil, 2), device="cuda")
    z = torch.empty((n, 15), device="cuda")
    spec = torch.empty((n, info.n_aperture, 2), device="cuda")
    plan.kk_spectra(n, I, x)
    plan.aberration(n, x, z)
    plan.stitch(n, x, z, spec)
    return plan, I, z, spec


def test_intensity_scale():
    """Intensities times 2^t with a spectrum times 2^(t/2): every FP32 operation of the solve then
    scales by a power of two, so the result does too, bit for bit, while no product or sum of a
    row leaves FP32's range (the sums over all rows do before: at 2^41). Beyond, a tile's solve
    may end early, but never unflagged."""
    plan, I, z, spec = _stitched(512, synth.illumination_8_24(), 1)

    def solve(t):
        s = spec * 2.0 ** (t % 2 / 2) * 2.0 ** (t // 2)
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        plan.darkfield(1, I * 2.0 ** t, z, s, st)
        torch.cuda.synchronize()
        return s, int(st)

    base = [solve(t) for t in (0, 1)]
    assert all(st == 0 for _, st in base)
    for t in (-10, 2, 20, 35, 38, 40, 41):
        s, st = solve(t)
        assert st == 0 and torch.equal(s, base[t % 2][0] * 2.0 ** (t // 2)), t
    for t in range(42, 75):
        s, st = solve(t)
        assert st == apic.APIC_TILE_NOTCONV or torch.equal(s, base[t % 2][0] * 2.0 ** (t // 2)), t


def _wave(plan):
    info = apic.apic_plan_info()
    assert apic.load().apic_plan_query(plan.handle, C.byref(info)) == apic.APIC_OK
    return info.df_wave


def test_autotune_on_a_few_tiles_keeps_the_rounds():
    """A sample below a wave leaves the plan at one block per tile by default, so that batches
    below a wave still go in rounds; results and waves are those of an untuned plan."""
    plan, I, z, spec = _stitched(512, synth.illumination_8_24(), 4)
    wave = _wave(plan)
    a, b = spec.clone(), spec.clone()
    plan.darkfield(4, I, z, a)
    ms = plan.autotune(4, I)
    assert all(ms[k] > 0 for k in ms)
    assert _wave(plan) == wave
    plan.darkfield(4, I, z, b)
    assert torch.equal(a, b)

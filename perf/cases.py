"""The work this library is timed on: whole-tile reconstruction from one tile to large batches, the
brightfield stages alone, whole slides, and the aberration network (training step and inference).

Inputs follow the synthetic recipe of the test suite and the benchmark (10x / 0.25 NA, 0.52 um, smooth
random samples, Noll 4..15 aberrations that vary over the slide, Poisson noise at 1e4 photons), made on
the GPU by plain torch from the seed alone. `exact` restates the method in float64 torch / numpy.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2407_20469_gb300 import apic, learn, slide, synth

PHOTONS = 1e4
# Illumination sets: number of NA-matching LEDs and the darkfield rings (NA, LEDs, turn in degrees).
SETS = {
    "8+16": (8, ((0.30, 8, 0.0), (0.38, 8, 22.5))),
    "8+24": (8, ((0.29, 8, 0.0), (0.34, 8, 22.5), (0.40, 8, 11.25))),
    "12+22": (12, ((0.31, 6, 0.0), (0.375, 8, 22.5), (0.44, 8, 0.0))),
}


def listed():
    return [
        # a single 128-pixel tile: the smallest reconstruction, where latency is everything
        {"name": "one_128", "kind": "batch", "n": 1, "tile": 128, "set": "8+16", "up": 2},
        # a few 256-pixel tiles: an interactive look at a region
        {"name": "few_256", "kind": "batch", "n": 5, "tile": 256, "set": "8+16", "up": 2},
        # one field of view of the paper's scanner: 25 patches of 512 pixels
        {"name": "view_512", "kind": "batch", "n": 25, "tile": 512, "set": "8+24", "up": 2},
        # the batched workload of 256-pixel tiles (16 x 32 grid)
        {"name": "batch_256", "kind": "batch", "n": 512, "tile": 256, "set": "8+16", "up": 2},
        # a large batch of the paper's patch size, not a whole number of GPU-wide waves
        {"name": "batch_512", "kind": "batch", "n": 400, "tile": 512, "set": "8+24", "up": 2},
        # the paper's set-up size: 12 + 22 LEDs and an output three times the camera sampling
        {"name": "setup_256x3", "kind": "batch", "n": 60, "tile": 256, "set": "12+22", "up": 3},
        # learned warm start, near-blank tiles taken over by the network (30 % of them)
        {"name": "learned_256", "kind": "learned", "n": 300, "tile": 256, "set": "8+16", "up": 2},
        # a ragged slide cut into overlapping windows, background skipped, overlaps blended
        {"name": "slide_256", "kind": "slide", "sh": 1300, "sw": 1900, "tile": 256, "stride": 241, "set": "8+16",
         "up": 2, "batch": 32},
        # the brightfield part alone (Kramers-Kronig, aberration, stitch, inverse transform): a preview
        {"name": "preview_512", "kind": "stages", "n": 96, "tile": 512, "set": "8+24", "up": 2},
        # one training step of the aberration network at the training loop's batch size
        {"name": "train_64", "kind": "train", "n": 64},
        # network inputs and coefficients of a batch of tiles
        {"name": "infer_256", "kind": "infer", "n": 512, "tile": 256},
        # joining the overlapping fields of a 16 x 32 window grid
        {"name": "blend_16x32", "kind": "blend", "rows": 16, "cols": 32, "tile": 256, "stride": 241, "up": 2},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["batch", "batch", "batch", "batch", "learned", "slide", "stages", "train", "infer", "blend"])
    if kind == "batch":
        tile = rng.choice([128, 256, 256, 512])
        s = rng.choice(["8+16", "8+24", "12+22"]) if tile < 512 else rng.choice(["8+16", "8+24"])
        n = _log(rng, 1, {128: 1024, 256: 600, 512: 350}[tile])
        return {"kind": kind, "n": n, "tile": tile, "set": s, "up": 3 if s == "12+22" and rng.random() < 0.5 else 2}
    if kind == "learned":
        tile = rng.choice([128, 256])
        return {"kind": kind, "n": _log(rng, 2, 500), "tile": tile, "set": "8+16", "up": 2}
    if kind == "slide":
        tile = rng.choice([128, 256])
        return {"kind": kind, "sh": rng.randint(2 * tile, 1800), "sw": rng.randint(2 * tile, 2400), "tile": tile,
                "stride": tile - rng.randint(0, tile // 8), "set": "8+16", "up": 2, "batch": rng.randint(16, 100)}
    if kind == "stages":
        tile = rng.choice([128, 256, 512])
        return {"kind": kind, "n": _log(rng, 1, {128: 1000, 256: 500, 512: 200}[tile]), "tile": tile,
                "set": rng.choice(["8+16", "8+24"]), "up": 2}
    if kind == "train":
        return {"kind": kind, "n": _log(rng, 8, 256)}
    if kind == "infer":
        return {"kind": kind, "n": _log(rng, 1, 1000), "tile": rng.choice([128, 256])}
    tile = rng.choice([128, 256])
    return {"kind": kind, "rows": rng.randint(2, 20), "cols": rng.randint(2, 30), "tile": tile,
            "stride": tile - rng.randint(1, tile // 8), "up": 2}


# ------------------------------------------------------------------ geometry (float64 restatement)

def _in_pupil(kx, ky, R):
    return (kx * kx + ky * ky) / (R * R) <= 1.0 + 1e-9


@functools.lru_cache(maxsize=8)
def _illumination(name):
    n_bf, rings = SETS[name]
    kx, ky = [], []
    for na, count, turn in ((0.25, n_bf, 0.0),) + rings:     # NA-matching ring first
        a = np.deg2rad(turn + 360.0 * np.arange(count) / count)
        r = na / float(synth.WAVELENGTH_UM)
        kx.append(r * np.cos(a))
        ky.append(r * np.sin(a))
    return np.concatenate(kx).astype(np.float32), np.concatenate(ky).astype(np.float32), n_bf


@functools.lru_cache(maxsize=8)
def _geometry(tile, name):
    """(pupil radius R, pupil points [n, 2], LED grid points [n_img, 2]) of a tile size and LED set."""
    kx, ky, n_bf = _illumination(name)
    R = float(np.float32(0.25)) * tile * float(np.float32(0.345)) / float(np.float32(0.52))
    a = math.ceil(R) + 1
    y, x = np.meshgrid(np.arange(-a, a + 1), np.arange(-a, a + 1), indexing="ij")
    m = _in_pupil(x, y, R)
    pupil = np.stack([x[m], y[m]], 1)
    leds = []
    win = 2 + int(0.2 * R)
    for i in range(len(kx)):
        px, py = (float(v) * tile * float(np.float32(0.345)) for v in (kx[i], ky[i]))
        if i >= n_bf:
            leds.append((math.floor(px + 0.5), math.floor(py + 0.5)))
            continue
        # NA-matching LEDs: the nearest pupil point whose shifted pupil keeps the DC term on its edge
        best = None
        for cy in range(math.floor(py) - win, math.floor(py) + win + 1):
            for cx in range(math.floor(px) - win, math.floor(px) + win + 1):
                key = ((cx - px) ** 2 + (cy - py) ** 2, cy, cx)
                if not _in_pupil(cx, cy, R) or (best is not None and key >= best):
                    continue
                K = pupil - (cx, cy)
                if np.any((K @ np.array([cx, cy]) >= 0) & np.any(K != 0, 1)):
                    continue
                best = key
        leds.append((best[2], best[1]))
    return R, pupil, np.array(leds)


def _zernike(x, y):
    """Noll 4..15, unit RMS on the disc, at unit-pupil coordinates (torch float64): [..., 12]."""
    r2 = x * x + y * y
    c2, s2 = x * x - y * y, 2 * x * y
    c3, s3 = x * c2 - y * s2, x * s2 + y * c2
    c4, s4 = c2 * c2 - s2 * s2, 2 * c2 * s2
    q, t = math.sqrt(6), math.sqrt(8)
    return torch.stack([
        math.sqrt(3) * (2 * r2 - 1), q * s2, q * c2, t * (3 * r2 - 2) * y, t * (3 * r2 - 2) * x, t * s3, t * c3,
        math.sqrt(5) * (6 * r2 * r2 - 6 * r2 + 1), math.sqrt(10) * (4 * r2 - 3) * c2, math.sqrt(10) * (4 * r2 - 3) * s2,
        math.sqrt(10) * c4, math.sqrt(10) * s4], -1)


# ------------------------------------------------------------------ inputs

def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _table(seed):
    return synth.quadratic_field(np.random.default_rng(seed + 77))


def _coefficients(seed, uv):
    """Noll 4..15 of tiles at uv: the microscope's quadratic field plus a focus offset per tile, [n, 12]."""
    rng = np.random.default_rng(seed)
    u, v = uv[:, 0].astype(np.float64), uv[:, 1].astype(np.float64)
    c = np.stack([np.ones_like(u), u, v, u * u, u * v, v * v], 1) @ _table(seed)
    c[:, 3] += rng.uniform(-0.2, 0.2, len(u))
    return torch.tensor(c[:, 3:], device="cuda")


def _objects(n, H, g, blank=None):
    """Smooth random transmissions [n, H, H] complex64; blank tiles with under 2 % contrast."""
    f = torch.fft.fftfreq(H, device="cuda")
    gauss = torch.exp(-2.0 * (math.pi * 4.0) ** 2 * (f[:, None] ** 2 + f[None, :] ** 2))
    z = torch.randn((2, n, H, H), device="cuda", generator=g)
    s = torch.fft.ifft2(torch.fft.fft2(z) * gauss).real
    lo, hi = s.amin((-2, -1), keepdim=True), s.amax((-2, -1), keepdim=True)
    s = (s - lo) / (hi - lo)
    amp, ph = torch.full((n, 1, 1), 0.2, device="cuda"), torch.full((n, 1, 1), math.pi, device="cuda")
    if blank is not None:
        amp[blank], ph[blank] = 0.01, 0.02
    return torch.polar(1 - amp + amp * s[0], ph * s[1])


def _stack(case, seed, n, uv, blank=None):
    """Noisy intensity stacks [n, n_img, tile, tile] of n tiles (forward model on the 2x grid)."""
    t = case["tile"]
    H = 2 * t
    R, pupil, leds = _geometry(t, case["set"])
    coef = _coefficients(seed, uv)
    pk = torch.tensor(pupil, device="cuda")
    phase = (_zernike(pk[:, 0].double() / R, pk[:, 1].double() / R) @ coef.T).T                     # [n, npup]
    ctf = torch.polar(torch.ones_like(phase), phase).to(torch.complex64)
    out = torch.empty((n, len(leds), t, t), device="cuda")
    step = max(1, (1 << 25) // (H * H))
    g = _gen(seed, 1)
    for a in range(0, n, step):
        b = min(n, a + step)
        O = torch.fft.fft2(_objects(b - a, H, g, None if blank is None else blank[a:b])) / (H * H)
        for i, (lx, ly) in enumerate(leds):
            S = torch.zeros((b - a, t, t), dtype=torch.complex64, device="cuda")
            S[:, pk[:, 1] % t, pk[:, 0] % t] = O[:, (pk[:, 1] - int(ly)) % H, (pk[:, 0] - int(lx)) % H] * ctf[a:b]
            I = (torch.fft.ifft2(S) * (t * t)).abs() ** 2
            out[a:b, i] = torch.poisson(I * PHOTONS, generator=g) / PHOTONS
    return out


def _uv(seed, n):
    return np.random.default_rng(seed + 5).uniform(-1, 1, (n, 2)).astype(np.float32)


def _blank(seed, n, share):
    return torch.tensor(np.random.default_rng(seed + 9).random(n) < share, device="cuda")


def _plan(case, n, flags=0):
    kx, ky, n_bf = _illumination(case["set"])
    return apic.Plan(case["tile"], kx, ky, n_bf, upsample=case["up"], max_tiles=n, flags=flags)


def _weights(seed):
    """Parameters with nonzero biases, as a network in training has them."""
    p = apic.unpack_params(learn.init_params(seed))
    rng = np.random.default_rng(seed + 3)
    for l in range(6):
        p[f"b{l}"] = 0.02 * rng.standard_normal(p[f"b{l}"].shape)
    return apic.pack_params(p)


def _features(seed, n):
    """Network inputs with the falling log spectra of real stacks, [n, 64, 64, 8] float32."""
    k = torch.arange(-32, 32, device="cuda", dtype=torch.float32)
    r = torch.sqrt(k[:, None] ** 2 + k[None, :] ** 2)
    f = -2.0 - 0.12 * r[None, :, :, None] + 0.8 * torch.randn((n, 64, 64, 8), device="cuda", generator=_gen(seed, 2))
    f = torch.maximum(f, torch.full_like(f, math.log(1e-4)))
    f[:, 32, 32] = 0.0
    return f


def _slide_blank(case, seed):
    """Tissue / background cells (128 pixels) of a slide: 40 % background in blobs."""
    h, w = -(-case["sh"] // 128), -(-case["sw"] // 128)
    rng = np.random.default_rng(seed + 13)
    z = rng.standard_normal((h + 2, w + 2))
    z = sum(z[dy:dy + h, dx:dx + w] for dy in range(3) for dx in range(3))
    return z < np.quantile(z, 0.4)


def _slide_stack(case, seed):
    """A slide's raw images [n_img, sh, sw]: cells of the tile size, each simulated on its own grid."""
    t, sh, sw = case["tile"], case["sh"], case["sw"]
    cells = [(y, x) for y in range(0, sh, t) for x in range(0, sw, t)]
    mask = _slide_blank(case, seed)
    blank = torch.tensor([bool(mask[min(y // 128, mask.shape[0] - 1), min(x // 128, mask.shape[1] - 1)])
                          for y, x in cells], device="cuda")
    uv = np.array([[2 * (x + t / 2) / sw - 1, 2 * (y + t / 2) / sh - 1] for y, x in cells], dtype=np.float32)
    I = _stack(case, seed, len(cells), uv, blank)
    out = torch.empty((I.shape[1], sh, sw), device="cuda")
    for k, (y, x) in enumerate(cells):
        out[:, y:y + t, x:x + t] = I[k][:, :min(t, sh - y), :min(t, sw - x)]
    return out


def _windows(length, t, stride):
    s = list(range(0, length - t + 1, stride))
    return s + [length - t] if s[-1] + t < length else s


def _blend_fields(case, seed):
    """Overlapping crops of one smooth field, each with its own global phase: [n, L, L] complex64, starts."""
    t, u, st = case["tile"], case["up"], case["stride"]
    sh, sw = t + (case["rows"] - 1) * st, t + (case["cols"] - 1) * st
    g = _gen(seed, 4)
    low = torch.randn((1, 4, u * sh // 16 + 2, u * sw // 16 + 2), device="cuda", generator=g)
    f = torch.nn.functional.interpolate(low, size=(u * sh, u * sw), mode="bilinear")[0]
    F = torch.polar(0.8 + 0.05 * f[0], 0.8 * f[1])
    ph = torch.rand(case["rows"] * case["cols"], device="cuda", generator=g) * 2 * math.pi
    ys, xs = _windows(sh, t, st), _windows(sw, t, st)
    out = torch.empty((len(ys) * len(xs), u * t, u * t), dtype=torch.complex64, device="cuda")
    for k, (y, x) in enumerate((y, x) for y in ys for x in xs):
        out[k] = F[u * y:u * (y + t), u * x:u * (x + t)] * torch.polar(torch.ones_like(ph[k]), ph[k])
    out += 0.01 * torch.view_as_complex(torch.randn(out.shape + (2,), device="cuda", generator=g))
    return out, ys, xs, sh, sw


# ------------------------------------------------------------------ the measured calls

def prepare(case, seed):
    k = case["kind"]
    s = {"case": case}
    if k in ("batch", "learned", "stages"):
        n, t = case["n"], case["tile"]
        H = case["up"] * t
        uv = _uv(seed, n)
        s["plan"] = _plan(case, n)
        s["I"] = _stack(case, seed, n, uv, _blank(seed, n, 0.3) if k == "learned" else None)
        s["uv"] = torch.tensor(uv, device="cuda")
        s["field"] = torch.empty((n, H, 2 * H), device="cuda")
        s["zern"] = torch.empty((n, 15), device="cuda")
        s["status"] = torch.empty(n, dtype=torch.int32, device="cuda")
        if k == "learned":
            s["net"] = apic.Net(256)
            s["net"].set_params(_weights(2407))
        if k == "stages":
            info = s["plan"].info
            s["xdisc"] = torch.empty((n, info.n_bf, info.n_pupil, 2), device="cuda")
            s["spec"] = torch.empty((n, info.n_aperture, 2), device="cuda")
    elif k == "slide":
        s["plan"] = _plan(case, case["batch"], apic.APIC_SKIP_BACKGROUND)
        s["slide"] = _slide_stack(case, seed)
    elif k == "train":
        s["net"] = apic.Net(case["n"])
        s["net"].set_params(_weights(seed))
        s["feat"] = _features(seed, case["n"])
        s["uv"] = torch.tensor(_uv(seed, case["n"]), device="cuda")
        s["target"] = torch.zeros((case["n"], 15), device="cuda")
        s["target"][:, 3:] = _coefficients(seed, _uv(seed, case["n"])).float()
        s["out"] = torch.empty((case["n"], 15), device="cuda")
        s["loss"] = torch.empty(1, device="cuda")
        s["step"] = 0
    elif k == "infer":
        n = case["n"]
        c = dict(case, set="8+16", up=2)
        uv = _uv(seed, n)
        s["plan"] = _plan(c, n)
        s["net"] = apic.Net(min(n, 512))
        s["net"].set_params(_weights(2407))
        s["I"] = _stack(c, seed, n, uv, _blank(seed, n, 0.3))
        s["uv"] = torch.tensor(uv, device="cuda")
        s["feat"] = torch.empty((n, 64, 64, 8), device="cuda")
    else:
        f, _, _, sh, sw = _blend_fields(case, seed)
        s["plan"] = _plan(dict(case, set="8+16"), 1)
        s["field"] = torch.view_as_real(f).reshape(len(f), f.shape[1], -1)
        s["size"] = (sh, sw)
        s["windows"] = apic.slide_windows(sh, sw, case["tile"], case["stride"])
    return s


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "batch":
        s["plan"].reconstruct_batch(case["n"], s["I"], s["field"], s["zern"], None, s["status"])
        return [s["field"], s["zern"], s["status"]]
    if k == "learned":
        s["plan"].reconstruct_learned(s["net"], apic.APIC_NET_WARM | apic.APIC_NET_REPLACE, case["n"], s["I"], s["uv"],
                                      s["field"], s["zern"], None, s["status"])
        return [s["field"], s["zern"], s["status"]]
    if k == "stages":
        p, n = s["plan"], case["n"]
        p.kk_spectra(n, s["I"], s["xdisc"])
        p.aberration(n, s["xdisc"], s["zern"])
        p.stitch(n, s["xdisc"], s["zern"], s["spec"])
        p.synthesize(n, s["spec"], s["field"])
        return [s["xdisc"], s["zern"], s["spec"], s["field"]]
    if k == "slide":
        field, zern, status, _ = slide.reconstruct_slide(s["plan"], s["slide"], case["sh"], case["sw"], case["stride"],
                                                         blend=True)
        return [field, zern, status]
    if k == "train":
        # the schedule's warm-up rate; one step, with its gradients as a data-parallel trainer reads them
        s["step"] += 1
        s["net"].forward(case["n"], s["feat"], s["uv"], s["out"])
        s["net"].backward(s["target"], s["loss"])
        grads = s["net"].get_grads()
        s["net"].adamw(1e-6, s["step"])
        return [s["out"], s["loss"], grads]
    if k == "infer":
        s["plan"].features(case["n"], s["I"], s["feat"])
        return [s["feat"], learn.predict(s["net"], s["feat"], s["uv"])]
    return list(slide.blend_slide(s["plan"], s["field"], s["windows"], *s["size"]))


# ------------------------------------------------------------------ the least work of a pass

def _fft(n, m=None):
    m = m or n
    return 5.0 * n * m * math.log2(n * m)


NET_MACS = 64 * 64 * 32 * 72 + 32 * 32 * 64 * 288 + 16 * 16 * 128 * 576 + 64 * 256 * 1152 + 258 * 256 + 256 * 12


def _tile_flops(case, darkfield=True):
    """Transforms of one tile (the bulk of its FP32 work): three per NA-matching image; the image's and
    the known field's, then four per conjugate-gradient step (about 17) on the darkfield solve's grid,
    which is about 0.55 of the camera's; the output's."""
    t = case["tile"]
    n_bf, rings = SETS[case["set"]]
    f = 3 * n_bf * _fft(t) + _fft(case["up"] * t)
    if darkfield:
        f += sum(r[1] for r in rings) * (2 * _fft(t) + 17 * 4 * _fft(0.55 * t))
    return f


def work(case):
    k = case["kind"]
    if k in ("batch", "learned", "stages"):
        n, t, H = case["n"], case["tile"], case["up"] * case["tile"]
        n_bf, rings = SETS[case["set"]]
        n_img = n_bf + sum(r[1] for r in rings)
        if k == "stages":
            R, pupil, _ = _geometry(t, case["set"])
            out = 8 * H * H + 8 * len(pupil) * (n_bf + 6)
            return {"bytes": n * (4.0 * n_bf * t * t + out), "flops": n * _tile_flops(case, False)}
        return {"bytes": n * (4.0 * n_img * t * t + 8 * H * H + 64),
                "flops": n * (_tile_flops(case) + (2.0 * NET_MACS + 8 * _fft(t) if k == "learned" else 0.0))}
    if k == "slide":
        n_img = SETS[case["set"]][0] + sum(r[1] for r in SETS[case["set"]][1])
        px = case["sh"] * case["sw"]
        tiles = 0.6 * len(_windows(case["sh"], case["tile"], case["stride"])) * \
            len(_windows(case["sw"], case["tile"], case["stride"]))
        return {"bytes": 4.0 * n_img * px + 8 * case["up"] ** 2 * px, "flops": tiles * _tile_flops(case)}
    if k == "train":
        return {"bytes": case["n"] * 4.0 * 64 * 64 * 8 + 5 * 4 * 459244, "flops": 6.0 * NET_MACS * case["n"]}
    if k == "infer":
        return {"bytes": case["n"] * (8 * 4.0 * case["tile"] ** 2 + 4 * 64 * 64 * 8) + 2 * 459244,
                "flops": case["n"] * (2.0 * NET_MACS + 8 * _fft(case["tile"]))}
    L = case["up"] * case["tile"]
    sh, sw = (case["tile"] + (case[a] - 1) * case["stride"] for a in ("rows", "cols"))
    return {"bytes": 8.0 * (case["rows"] * case["cols"] * L * L + case["up"] ** 2 * sh * sw),
            "flops": 16.0 * case["rows"] * case["cols"] * L * L}


# ------------------------------------------------------------------ exact values (float64)

def _wrap(a):
    return math.pi - torch.remainder(math.pi - a, 2 * math.pi)


def _exact_kk(I, leds, R, pupil):
    """Kramers-Kronig spectra of NA-matching images I [n, n_bf, t, t] float64 at the pupil points."""
    n, n_bf, t, _ = I.shape
    k = torch.fft.fftfreq(t, 1.0 / t, device="cuda", dtype=torch.float64)
    pk = torch.tensor(pupil, device="cuda")
    X = torch.empty((n, n_bf, len(pupil)), dtype=torch.complex128, device="cuda")
    for i in range(n_bf):
        lx, ly = (int(v) for v in leds[i])
        dot = k[None, :] * lx + k[:, None] * ly
        mask = torch.where(dot < 0, 1.0, torch.where(dot == 0, 0.5, 0.0))
        a = I[:, i]
        L = torch.log(torch.maximum(a, 1e-6 * a.mean((-2, -1), keepdim=True)))
        S = torch.fft.fft2(torch.exp(torch.fft.ifft2(torch.fft.fft2(L) * mask))) / (t * t)
        X[:, i] = S[:, (pk[:, 1] - ly) % t, (pk[:, 0] - lx) % t]
    return X


def _normal(A, y):
    """Least squares through the normal equations: A [r, 12], y [n, r] -> [n, 12]."""
    return torch.cholesky_solve((y @ A).T, torch.linalg.cholesky(A.T @ A)).T


def _exact_zern(X, leds, R, pupil, start=None):
    """Noll 4..15 [n, 12] from the phase differences on every overlap (neighbour fit, two refinements).
    start: refine from these as well and keep the smaller residual."""
    a = int(np.abs(pupil).max()) + 1
    lut = np.full((2 * a + 1, 2 * a + 1), -1)
    lut[pupil[:, 1] + a, pupil[:, 0] + a] = np.arange(len(pupil))

    def at(x, y):
        ok = (np.abs(x) <= a) & (np.abs(y) <= a)
        return np.where(ok, lut[np.clip(y, -a, a) + a, np.clip(x, -a, a) + a], -1)

    Z = _zernike(*(torch.tensor(pupil[:, c] / R, device="cuda") for c in (0, 1)))
    A, beta, dA, db = [], [], [], []
    for i in range(X.shape[1]):
        for l in range(i + 1, X.shape[1]):
            ql = at(*(pupil - leds[i] + leds[l]).T)
            pi, pl = np.nonzero(ql >= 0)[0], ql[ql >= 0]
            rows = Z[pi] - Z[pl] - Z[at(*leds[i])] + Z[at(*leds[l])]
            b = torch.angle(X[:, i, pi] * X[:, l, pl].conj())
            where = np.full(len(pupil) + 1, -1)
            where[pi] = np.arange(len(pi))
            for d in ((1, 0), (0, 1)):
                nb = where[at(*(pupil[pi] + d).T)]
                r0 = np.nonzero(nb >= 0)[0]
                dA.append(rows[nb[r0]] - rows[r0])
                db.append(_wrap(b[:, nb[r0]] - b[:, r0]))
            A.append(rows)
            beta.append(b)
    A, beta = torch.cat(A), torch.cat(beta, 1)
    c = _normal(torch.cat(dA), torch.cat(db, 1))
    del dA, db

    def refine(c):
        for _ in range(2):
            c = c + _normal(A, _wrap(beta - c @ A.T))
        return c, _wrap(beta - c @ A.T).square().sum(1, keepdim=True)

    c, res = refine(c)
    if start is not None:
        c2, res2 = refine(start)
        c = torch.where(res2 < res, c2, c)
    return c


def _exact_spectrum(case, I, coef, X, darkfield=True):
    """Object spectrum [n, H, H] complex128 (series coefficients) and its known mask [H, H]."""
    t, u = case["tile"], case["up"]
    H = u * t
    R, pupil, leds = _geometry(t, case["set"])
    n, n_bf = len(I), SETS[case["set"]][0]
    pk = torch.tensor(pupil, device="cuda")
    phi = (_zernike(pk[:, 0].double() / R, pk[:, 1].double() / R) @ coef.T).T
    spec = torch.zeros((n, H, H), dtype=torch.complex128, device="cuda")
    count = torch.zeros((H, H), dtype=torch.float64, device="cuda")
    for i in range(n_bf):
        y, x = (pk[:, 1] - int(leds[i][1])) % H, (pk[:, 0] - int(leds[i][0])) % H
        c = phi - phi[:, int(np.nonzero((pupil == leds[i]).all(1))[0][0])][:, None]
        spec[:, y, x] += X[:, i] * torch.polar(torch.ones_like(c), -c)
        count[y, x] += 1
    known = (count > 0).cpu().numpy()
    spec /= count.clamp(min=1)
    if not darkfield:
        return spec, known
    k_df = leds[n_bf:]
    order = np.lexsort((np.arange(len(k_df)), np.arctan2(*k_df.T[::-1].astype(float)), (k_df ** 2).sum(1)))
    m = 2 * t                                    # set algebra: lags up to two diameters
    for j in order:
        lx, ly = (int(v) for v in k_df[j])
        oy, ox = (pupil[:, 1] - ly) % H, (pupil[:, 0] - lx) % H
        isk = known[oy, ox]
        U, P = pupil[~isk], pupil[isk]
        fu, fp = np.zeros((m, m)), np.zeros((m, m))
        fu[U[:, 1] % m, U[:, 0] % m] = 1
        fp[P[:, 1] % m, P[:, 0] % m] = 1
        Fu, Fp = np.fft.fft2(fu), np.fft.fft2(fp)
        up = np.fft.ifft2(Fu * Fp.conj()).real > 0.5
        pu = np.fft.ifft2(Fp * Fu.conj()).real > 0.5
        uu = np.fft.ifft2(Fu * Fu.conj()).real > 0.5
        qy, qx = np.nonzero(up & ~pu & ~uu)
        if not (len(U) and len(qx) >= len(U) and len(U) <= 0.42 * len(pupil)):
            continue
        qy, qx = np.where(qy < m // 2, qy, qy - m), np.where(qx < m // 2, qx, qx - m)
        known[oy[~isk], ox[~isk]] = True
        Q = torch.zeros((t, t), dtype=torch.float64, device="cuda")
        Q[qy % t, qx % t] = 1                    # lags reach two radii, under half the camera grid
        Um = torch.zeros((t, t), dtype=torch.float64, device="cuda")
        Um[U[:, 1] % t, U[:, 0] % t] = 1
        rot = torch.polar(torch.ones_like(phi), phi)
        Pv = torch.zeros((n, t, t), dtype=torch.complex128, device="cuda")
        Pv[:, P[:, 1] % t, P[:, 0] % t] = spec[:, oy[isk], ox[isk]] * rot[:, isk]
        p = torch.fft.ifft2(Pv) * (t * t)
        # (P*U)(k) = sum_q U(q) conj P(q - k): the series coefficients of u conj p
        b = torch.fft.fft2(I[:, n_bf + j] - p.abs() ** 2) / (t * t) * Q
        fwd = lambda d: torch.fft.fft2(torch.fft.ifft2(d) * p.conj()) * Q  # noqa: E731
        adj = lambda r: torch.fft.fft2(torch.fft.ifft2(r) * p) * Um        # noqa: E731
        dot = lambda v: (v.real ** 2 + v.imag ** 2).sum((1, 2), keepdim=True)  # noqa: E731
        x, r = torch.zeros_like(b), b
        s = adj(r)
        d, gam = s, dot(s)
        end = 1e-18 * gam
        for it in range(120):
            q = fwd(d)
            al = gam / dot(q).clamp(min=1e-300)
            x, r = x + al * d, r - al * q
            s = adj(r)
            g2 = dot(s)
            d, gam = s + g2 / gam.clamp(min=1e-300) * d, g2
            if it % 8 == 7 and bool((g2 <= end).all()):
                break
        spec[:, oy[~isk], ox[~isk]] = x[:, U[:, 1] % t, U[:, 0] % t] * rot[:, ~isk].conj()
    return spec, known


def _chunks(case, n):
    c = max(1, (1 << 22) // case["tile"] ** 2)
    return [(a, min(n, a + c)) for a in range(0, n, c)]


def _exact_tiles(case, I, start=None, take=None):
    """(field [n, H, 2 H] float32, Noll coefficients [n, 15]); start: the network's coefficients, taken as
    they are by the tiles in `take`. The field is computed in 64 bits and rounded once."""
    R, pupil, leds = _geometry(case["tile"], case["set"])
    n_bf = SETS[case["set"]][0]
    H = case["up"] * case["tile"]
    field, zern = torch.empty((len(I), H, 2 * H), device="cuda"), []
    for a, b in _chunks(case, len(I)):
        J = I[a:b].double()
        X = _exact_kk(J[:, :n_bf], leds, R, pupil)
        coef = _exact_zern(X, leds, R, pupil, None if start is None else start[a:b])
        if take is not None:
            coef = torch.where(take[a:b, None], start[a:b], coef)
        spec, _ = _exact_spectrum(case, J, coef, X)
        field[a:b] = torch.view_as_real(torch.fft.ifft2(spec) * (H * H)).reshape(b - a, H, 2 * H).float()
        zern.append(coef)
    z = torch.cat(zern)
    return field, torch.cat([torch.zeros((len(z), 3), device="cuda", dtype=z.dtype), z], 1)


def _exact_features(I):
    t = I.shape[-1]
    out = []
    for a in range(0, len(I), 64):
        F = torch.fft.fft2(I[a:a + 64, :8].double()).abs()
        F = F / F[..., :1, :1]
        k = torch.arange(-32, 32, device="cuda") % t
        out.append(torch.log(F[..., k[:, None], k[None, :]] + 1e-4).permute(0, 2, 3, 1))
    return torch.cat(out)


def _exact_net(weights, feat, uv):
    p = {k: torch.tensor(v, device="cuda").requires_grad_() for k, v in _unpack(weights).items()}
    x = feat.double().permute(0, 3, 1, 2)
    for l in range(4):
        x = torch.relu(torch.nn.functional.conv2d(x, p[f"w{l}"], p[f"b{l}"], padding=1))
        x = torch.nn.functional.max_pool2d(x, 2) if l < 3 else x.mean((2, 3))
    x = torch.relu(torch.cat([x, uv.double()], 1) @ p["w4"].T + p["b4"])
    return x @ p["w5"].T + p["b5"], p


def _unpack(v):
    """The flat parameter vector (rows of taps (dy, dx, c_in) and a bias) as conv / dense arrays."""
    v, p, o = np.asarray(v, dtype=np.float64), {}, 0
    for l, (co, ci) in enumerate(((32, 8), (64, 32), (128, 64), (256, 128), (256, 258), (12, 256))):
        taps = 9 * ci if l < 4 else ci
        m = v[o:o + co * (taps + 1)].reshape(co, taps + 1)
        o += co * (taps + 1)
        w = m[:, :-1]
        p[f"w{l}"] = w.reshape(co, 3, 3, ci).transpose(0, 3, 1, 2).copy() if l < 4 else w.copy()
        p[f"b{l}"] = m[:, -1].copy()
    return p


def _exact_blend(f, ys, xs, t, u, sh, sw):
    """(joined field, correlations with the left / upper neighbour, phases) of fields [n, L, L] complex128."""
    rows, cols, L = len(ys), len(xs), u * t
    ys, xs = [u * y for y in ys], [u * x for x in xs]
    corr = torch.zeros((rows * cols, 2), dtype=torch.complex128, device="cuda")
    for k in range(rows * cols):
        i, j = divmod(k, cols)
        if j:
            o = xs[j - 1] + L - xs[j]
            if o > 0:
                corr[k, 0] = (f[k][:, :o] * f[k - 1][:, L - o:].conj()).sum()
        if i:
            o = ys[i - 1] + L - ys[i]
            if o > 0:
                corr[k, 1] = (f[k][:o] * f[k - cols][L - o:].conj()).sum()
    c = corr.cpu().numpy()
    z = np.ones(rows * cols, dtype=np.complex128)
    for k in range(1, rows * cols):
        v, s = (c[k, 0], k - 1) if k < cols else (c[k, 1], k - cols)
        z[k] = z[s] * (np.conj(v) / abs(v) if abs(v) > 0 else 1.0)

    def ramp(st, j):
        p = np.arange(L) + 0.5
        w = np.ones(L)
        if j > 0 and st[j - 1] + L > st[j]:
            o = st[j - 1] + L - st[j]
            w[:o] *= p[:o] / o
        if j + 1 < len(st) and st[j] + L > st[j + 1]:
            o = st[j] + L - st[j + 1]
            w[L - o:] *= (L - p[L - o:]) / o
        return torch.tensor(w, device="cuda")

    acc = torch.zeros((u * sh, u * sw), dtype=torch.complex128, device="cuda")
    ws = torch.zeros((u * sh, u * sw), dtype=torch.float64, device="cuda")
    zt = torch.tensor(z, device="cuda")
    for k in range(rows * cols):
        i, j = divmod(k, cols)
        w = ramp(ys, i)[:, None] * ramp(xs, j)[None, :]
        acc[ys[i]:ys[i] + L, xs[j]:xs[j] + L] += w * zt[k] * f[k]
        ws[ys[i]:ys[i] + L, xs[j]:xs[j] + L] += w
    return acc / ws, corr, zt


def _real(z, width):
    return torch.view_as_real(z).reshape(len(z), width)


def exact(case, seed):
    k = case["kind"]
    if k in ("batch", "learned"):
        # the darkfield solves in 64 bits: under about 20 seconds up to these sizes
        n, t = case["n"], case["tile"]
        if n * t * t * sum(r[1] for r in SETS[case["set"]][1]) > 24 * 25 * 512 * 512:
            return None
        I = _stack(case, seed, n, _uv(seed, n), _blank(seed, n, 0.3) if k == "learned" else None)
        if k == "batch":
            field, zern = _exact_tiles(case, I)
        else:
            with torch.no_grad():
                c0 = _exact_net(_weights(2407), _exact_features(I), torch.tensor(_uv(seed, n), device="cuda"))[0]
            B = I[:, :8].double()
            mean = B.mean((-2, -1))
            c2 = (((B - mean[..., None, None]) ** 2).mean((-2, -1)) / mean ** 2).mean(1)
            field, zern = _exact_tiles(case, I, c0, c2 < 0.02 ** 2)
        return [field, zern, None]
    if k == "stages":
        n = case["n"]
        R, pupil, leds = _geometry(case["tile"], case["set"])
        n_bf, H = SETS[case["set"]][0], case["up"] * case["tile"]
        I = _stack(case, seed, n, _uv(seed, n))
        out = [torch.empty((n, n_bf, len(pupil), 2), device="cuda"), torch.zeros((n, 15), device="cuda"), None,
               torch.empty((n, H, 2 * H), device="cuda")]
        for a, b in _chunks(case, n):
            J = I[a:b].double()
            X = _exact_kk(J[:, :n_bf], leds, R, pupil)
            coef = _exact_zern(X, leds, R, pupil)
            spec, _ = _exact_spectrum(case, J, coef, X, False)
            out[0][a:b] = torch.view_as_real(X).float()
            out[1][a:b, 3:] = coef.float()
            out[3][a:b] = torch.view_as_real(torch.fft.ifft2(spec) * (H * H)).reshape(b - a, H, 2 * H).float()
        return out
    if k == "slide":
        t, u = case["tile"], case["up"]
        S = _slide_stack(case, seed)
        ys, xs = _windows(case["sh"], t, case["stride"]), _windows(case["sw"], t, case["stride"])
        I = torch.stack([S[:, y:y + t, x:x + t] for y in ys for x in xs])
        B = I[:, :SETS[case["set"]][0]].double()
        mean = B.mean((-2, -1))
        c2 = (((B - mean[..., None, None]) ** 2).mean((-2, -1)) / mean ** 2).mean(1)
        use = c2 >= 0.02 ** 2
        H = u * t
        f = torch.zeros((len(I), H, 2 * H), device="cuda")
        zern = torch.zeros((len(I), 15), dtype=torch.float64, device="cuda")
        if bool(use.any()):
            f[use], zern[use] = _exact_tiles(case, I[use])
        z = torch.view_as_complex(f.reshape(len(f), H, H, 2)).to(torch.complex128)
        return [_real(_exact_blend(z, ys, xs, t, u, case["sh"], case["sw"])[0], 2 * u * case["sw"]), zern, None]
    if k == "train":
        uv = _uv(seed, case["n"])
        y, p = _exact_net(_weights(seed), _features(seed, case["n"]), torch.tensor(uv, device="cuda"))
        loss = ((y - _coefficients(seed, uv).float().double()) ** 2).mean()
        loss.backward()
        g = []
        for l in range(6):
            w, b = p[f"w{l}"].grad, p[f"b{l}"].grad
            w = w.permute(0, 2, 3, 1).reshape(len(w), -1) if l < 4 else w
            g.append(torch.cat([w, b[:, None]], 1).reshape(-1))
        out = torch.cat([torch.zeros((len(y), 3), device="cuda", dtype=y.dtype), y.detach()], 1)
        return [out, loss.detach().reshape(1), torch.cat(g)]
    if k == "infer":
        c = dict(case, set="8+16", up=2)
        uv = _uv(seed, case["n"])
        feat = _exact_features(_stack(c, seed, case["n"], uv, _blank(seed, case["n"], 0.3)))
        with torch.no_grad():
            w = _weights(2407)
            y = torch.cat([_exact_net(w, feat[a:a + 64], torch.tensor(uv[a:a + 64], device="cuda"))[0]
                           for a in range(0, case["n"], 64)])
        return [feat, torch.cat([torch.zeros((len(y), 3), device="cuda", dtype=y.dtype), y], 1)]
    f, ys, xs, sh, sw = _blend_fields(case, seed)
    joined, corr, z = _exact_blend(f.to(torch.complex128), ys, xs, case["tile"], case["up"], sh, sw)
    return [_real(joined, 2 * case["up"] * sw), _real(corr, 4), _real(z, 2)]

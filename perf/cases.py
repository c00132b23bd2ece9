"""What this framework is used for, as cases that can be timed and compared.

Each case is one pass through the public calls, on inputs made from a seed:
whole pyramid frames and a closed-loop step as captured CUDA graphs (the way
a simulation replays them), single stages (the pyramid image, Shack-Hartmann
spots and slopes, the batched reconstructor), a multi-sensor frame, the
training-pair generator, training steps and inference of the learned
reconstructor.  Sizes are those of the repository's workloads; ``draw`` gives
others of the same ranges.

``exact`` restates each pass in float64 with plain torch, from the formulas
that include/specula_gb300.h documents.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2602_06688_gb300 as sp

DEV = "cuda"
ARCSEC = math.pi / (180.0 * 3600.0)

# ---- the cases ---------------------------------------------------------------

# pyramid geometries: pupil side, padding, subapertures, image separation,
# modulation points and radius, obscuration
PYR_8M = dict(n_pix=160, pad=2, n_sub=40, pup_dist=160, n_mod=24, mod_amp=3.0, obsc=0.11)
PYR_39M = dict(n_pix=480, pad=2, n_sub=96, pup_dist=480, n_mod=48, mod_amp=4.0, obsc=0.28)
PYR_SOUL = dict(n_pix=220, pad=3, n_sub=40, pup_dist=264, n_mod=24, mod_amp=3.0, obsc=0.11)
PYR_ANDES = dict(n_pix=400, pad=4, n_sub=100, pup_dist=480, n_mod=24, mod_amp=3.0, obsc=0.28)


def listed():
    return [
        # the 8 m pyramid frame (three layers, 500 modes), replayed once per
        # time step: the smallest pass, where launches and gaps count
        dict(name="frame_8m", kind="frame", layers=3, side=1024, n_modes=500, **PYR_8M),
        # the ELT pyramid frame: 35 layers, 960^2 grid, 48 points, 4000 modes
        dict(name="frame_39m", kind="frame", layers=35, side=2048, n_modes=4000, **PYR_39M),
        # one step of the 8 m closed loop: extraction, mirror, residual and
        # its statistics, image, slopes, modes, integrator
        dict(name="loop_8m", kind="loop", layers=3, side=1024, n_modes=500, **PYR_8M),
        # the pyramid image alone: SOUL's 660^2 grid with 5.5 px detector
        # pixels, and ANDES' 1600^2 grid
        dict(name="image_soul", kind="image", batch=1, **PYR_SOUL),
        dict(name="image_andes", kind="image", batch=1, **PYR_ANDES),
        # one 68 x 68 laser-star Shack-Hartmann sensor: spots and centres of gravity
        dict(name="sh_39m", kind="sh", n_sub=68, sub_pix=12, fft_n=24, batch=1, obsc=0.28),
        # six Shack-Hartmann sensors and three pyramids in one launch, with
        # the 4000-mode product on all slopes
        dict(name="system_39m", kind="system", n_sh=6, n_sub_sh=68, n_pyr=3, n_pix=120,
             n_sub=40, n_mod=16, layers=10, side=2048, n_modes=4000),
        # 256 training pairs of the 8 m pyramid: screens, phases, images,
        # slopes, and the labels by the float32 modal projection
        dict(name="pairs_8m", kind="pairs", n=256, side=256, n_modes=500, **PYR_8M),
        # the ELT reconstructor on 8 frames at once in float32, and on 2048
        # in split bf16
        dict(name="recon_fp32_b8", kind="recon", precision="fp32", n_modes=4000,
             n_slopes=13344, batch=8),
        dict(name="recon_split_b2048", kind="recon", precision="bf16x2", n_modes=4000,
             n_slopes=13344, batch=2048),
        # 16 training steps of the 8 m network (forward, backward, Adam) and
        # the weights read back, as a program does that saves or evaluates it
        dict(name="train_8m", kind="train", n_in=2512, h1=1024, h2=1024, n_out=500, batch=256,
             steps=16),
        # the ELT network on one frame's slopes
        dict(name="infer_39m", kind="infer", n_in=13344, h1=2048, h2=2048, n_out=4000, batch=1),
    ]


# padded grids that have a compiled transform: pupil side, padding, and the
# subaperture counts drawn with them
_GRIDS = [(32, 2, (8, 16)), (32, 4, (8, 16)), (64, 2, (16, 32)), (120, 2, (24, 40)),
          (80, 3, (20, 40)), (60, 4, (15, 30)), (160, 2, (32, 40, 80)), (80, 4, (20, 40)),
          (220, 3, (40, 44, 110)), (165, 4, (33, 55)), (480, 2, (80, 96, 120)),
          (320, 3, (64, 80)), (240, 4, (48, 60)), (400, 4, (80, 100))]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_pyr(rng, maps):
    """A pyramid geometry; with maps, one whose four images fall on whole
    detector pixels (what a slope computer needs)."""
    n, pad, subs = rng.choice(_GRIDS)
    n_sub = rng.choice(subs)
    if maps and (pad * n_sub) % 2:
        n_sub = [s for s in subs if (pad * s) % 2 == 0][0]
    if pad == 2:
        dist = n
    else:
        dist = rng.randint(n, (pad - 1) * n)
        if maps:   # 2 d = dist n_sub / n whole, of n_sub's parity
            two_d = n_sub + 2 * rng.randint(0, (pad - 2) * n_sub // 2)
            while (two_d * n) % n_sub:
                two_d += 2
            dist = two_d * n // n_sub
            if dist + n > pad * n:
                dist = n
    big = n * pad >= 960
    n_mod = rng.randint(3, 24 if n * pad > 960 else 48) if big else _log_int(rng, 4, 48)
    return dict(n_pix=n, pad=pad, n_sub=n_sub, pup_dist=dist, n_mod=n_mod,
                mod_amp=round(rng.uniform(1.0, 6.0), 2), obsc=rng.choice([0.0, 0.11, 0.28]))


def draw(rng):
    kind = rng.choice(["frame", "loop", "image", "image", "sh", "system", "pairs", "recon",
                       "recon", "train", "infer"])
    if kind == "frame":
        g = _draw_pyr(rng, True)
        return dict(kind=kind, layers=rng.randint(1, 35), side=rng.choice([512, 1000, 1024, 2048]),
                    n_modes=_log_int(rng, 50, 4000), **g)
    if kind == "loop":
        n, pad, subs = rng.choice([c for c in _GRIDS if c[1] == 2 and c[0] <= 160])
        return dict(kind=kind, layers=rng.randint(1, 10), side=rng.choice([512, 1000, 1024]),
                    n_modes=_log_int(rng, 20, 500), n_pix=n, pad=pad, n_sub=rng.choice(subs),
                    pup_dist=n, n_mod=_log_int(rng, 4, 24), mod_amp=3.0,
                    obsc=rng.choice([0.0, 0.11]))
    if kind == "image":
        g = _draw_pyr(rng, False)
        n_grid = g["n_pix"] * g["pad"]
        cap = max(1, int(24 * 1600 ** 2 / (g["n_mod"] * n_grid ** 2)))
        return dict(kind=kind, batch=_log_int(rng, 1, min(cap, 64)), **g)
    if kind == "sh":
        sub_pix, fft_n = rng.choice([(12, 24), (8, 16), (8, 56), (4, 68)])
        n_sub = _log_int(rng, 8, 68)
        cap = max(1, int(68 * 68 * 24 ** 2 / (n_sub ** 2 * fft_n ** 2)))
        return dict(kind=kind, n_sub=n_sub, sub_pix=sub_pix, fft_n=fft_n,
                    batch=_log_int(rng, 1, min(cap, 16)), obsc=rng.choice([0.0, 0.11, 0.28]))
    if kind == "system":
        n_pix, subs = rng.choice([(64, (16, 32)), (120, (24, 40))])
        return dict(kind=kind, n_sh=rng.randint(1, 6), n_sub_sh=_log_int(rng, 8, 68),
                    n_pyr=rng.randint(1, 3), n_pix=n_pix, n_sub=rng.choice(subs),
                    n_mod=rng.randint(4, 16), layers=rng.randint(1, 10), side=2048,
                    n_modes=_log_int(rng, 50, 4000))
    if kind == "pairs":
        n, pad, subs = rng.choice([c for c in _GRIDS if c[1] == 2 and 64 <= c[0] <= 160])
        return dict(kind=kind, n=_log_int(rng, 16, 256), side=256, n_modes=_log_int(rng, 50, 500),
                    n_pix=n, pad=pad, n_sub=rng.choice(subs), pup_dist=n,
                    n_mod=_log_int(rng, 4, 24), mod_amp=3.0, obsc=rng.choice([0.0, 0.11]))
    if kind == "recon":
        precision = rng.choice(["fp32", "fp32", "bf16x2", "bf16"])
        n_modes, n_slopes = _log_int(rng, 64, 4000), _log_int(rng, 200, 13344)
        if precision != "fp32":
            n_slopes = n_slopes // 8 * 8     # what the bf16 forms take
        elif rng.random() < 0.75:
            n_slopes = n_slopes // 2 * 2     # x and y slopes: even counts
        return dict(kind=kind, precision=precision, n_modes=n_modes, n_slopes=n_slopes,
                    batch=_log_int(rng, 1, 512 if precision == "fp32" else 2048))
    h1, h2 = 128 * rng.randint(1, 8), 128 * rng.randint(1, 8)
    if kind == "train":
        return dict(kind=kind, n_in=_log_int(rng, 200, 2512), h1=h1, h2=h2,
                    n_out=_log_int(rng, 20, 500), batch=rng.choice([64, 100, 128, 200, 256]),
                    steps=rng.randint(4, 16))
    return dict(kind="infer", n_in=_log_int(rng, 200, 13344), h1=h1, h2=h2,
                n_out=_log_int(rng, 20, 4000),
                batch=rng.choice([1, 1, 2, 3, 4, 16, 100, 512, 1024]))


def work(case):
    """Bytes: each input read and each output written once.  Flops: for the
    pyramid, its separable form, each distinct filter once, 5 N log2 N per
    transform; a product's 2 M N K."""
    c = SimpleNamespace(**case)
    if c.kind in ("frame", "loop", "image", "pairs"):
        batch = getattr(c, "batch", getattr(c, "n", 1))
        n, N, nd = c.n_pix, c.pad * c.n_pix, c.pad * c.n_sub
        fft = 5.0 * N * math.log2(N)
        flops = batch * fft * 2 * (n * (c.n_mod // 2 + 1) + N * c.n_mod)
        px = n * n
        nbytes = 4.0 * (px + batch * (px + nd * nd))          # amp, phase, detector
        if c.kind == "image":
            return dict(bytes=nbytes, flops=flops)
        n_slopes = 2 * len(_valid(n, c.obsc, c.n_sub))
        flops += 2.0 * batch * c.n_modes * (px if c.kind == "pairs" else n_slopes)
        nbytes += 4.0 * batch * (n_slopes + c.n_modes)
        if c.kind == "pairs":
            s2 = float(c.side) ** 2
            flops += batch * 5 * s2 * math.log2(s2)
            nbytes += 4.0 * c.n_modes * px
        else:
            flops += 8.0 * c.layers * px
            nbytes += 4.0 * (c.layers * px + c.n_modes * n_slopes)
        if c.kind == "loop":
            flops += 2.0 * c.n_modes * px
            nbytes += 4.0 * (c.n_modes * px + 2 * px + c.n_modes)
        return dict(bytes=nbytes, flops=flops)
    if c.kind == "sh":
        nv = len(_valid(c.n_sub * c.sub_pix, c.obsc, c.n_sub))
        return dict(bytes=4.0 * ((c.batch + 1) * nv * c.sub_pix ** 2
                                 + c.batch * nv * (c.fft_n ** 2 + 2)),
                    flops=c.batch * nv * 5.0 * c.fft_n * math.log2(c.fft_n)
                    * (c.sub_pix + c.fft_n))
    if c.kind == "system":
        nv = len(_valid(12 * c.n_sub_sh, 0.28, c.n_sub_sh))
        nvp = len(_valid(c.n_pix, 0.28, c.n_sub))
        n_slopes = 2 * (c.n_sh * nv + c.n_pyr * nvp)
        N = 2 * c.n_pix
        px = c.n_sh * nv * 144 + c.n_pyr * c.n_pix ** 2
        flops = (8.0 * c.layers * px + c.n_sh * nv * 5.0 * 24 * math.log2(24) * 36
                 + c.n_pyr * 10.0 * N * math.log2(N)
                 * (c.n_pix * (c.n_mod // 2 + 1) + N * c.n_mod)
                 + 2.0 * c.n_modes * n_slopes)
        return dict(bytes=4.0 * (c.layers * px + c.n_modes * n_slopes + n_slopes + c.n_modes),
                    flops=flops)
    if c.kind == "recon":
        return dict(bytes=4.0 * (c.n_modes * c.n_slopes * (0.5 if c.precision == "bf16" else 1.0)
                                 + c.batch * (c.n_slopes + c.n_modes)),
                    flops=2.0 * c.batch * c.n_modes * c.n_slopes)
    w = c.n_in * c.h1 + c.h1 * c.h2 + c.h2 * c.n_out
    if c.kind == "train":   # per step: weights and two moments read and written, data read
        return dict(bytes=c.steps * (24.0 * w + 4.0 * c.batch * (c.n_in + c.n_out)) + 4.0 * w,
                    flops=c.steps * c.batch * 2.0 * (3 * w - c.n_in * c.h1))
    return dict(bytes=2.0 * w + 4.0 * c.batch * (c.n_in + c.n_out), flops=2.0 * c.batch * w)


# ---- inputs -------------------------------------------------------------------

_CTX = []


def _ctx():
    """One library context per process, as a program keeps it."""
    if not _CTX:
        _CTX.append(sp.Context(0))
    return _CTX[0]


def _gen(seed, k=0):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1009 + 7919 * k + 13)


def _randn(shape, seed, k=0):
    return torch.randn(shape, generator=_gen(seed, k), device=DEV)


def _screen(side, rms, g):
    """A smooth random screen with a Kolmogorov-like slope, zero mean, the
    given RMS [rad at 500 nm]."""
    f = torch.fft.fftfreq(side, device=DEV) * side
    f2 = f[:, None] ** 2 + f[None, : side // 2 + 1] ** 2
    f2[0, 0] = 1.0
    a = f2 ** (-11.0 / 12.0)
    a[0, 0] = 0.0
    s = torch.fft.irfft2(torch.fft.rfft2(torch.randn(side, side, generator=g, device=DEV)) * a,
                         s=(side, side))
    return (s * (rms / s.std())).contiguous()


def _atmosphere(c, seed, pitch):
    """(layers, screens, time): ground-heavy layers up to 20 km, winds up to
    40 m/s, the screens and the frame's time from the seed."""
    n = c.layers
    w = np.exp(-np.linspace(0.0, 6.0, n)) if n > 1 else np.ones(1)
    w = w / w.sum()
    ang = np.linspace(0.3, 5.7, n)
    speed = np.linspace(5.0, 40.0, n)
    layers = [sp.LayerDesc(c.side, pitch, 20e3 * k / max(n - 1, 1), float(speed[k] * np.cos(ang[k])),
                           float(speed[k] * np.sin(ang[k]))) for k in range(n)]
    g = _gen(seed, 1)
    screens = [_screen(c.side, 12.0 * math.sqrt(float(w[k])), g) for k in range(n)]
    return layers, screens, 1.0 + (int(seed) * 0.0137) % 50.0


def _phases(n, batch, rms, seed):
    """(batch, n, n) pupil phases cut from smooth screens."""
    side = 1 << max(6, (2 * n - 1).bit_length())
    g = _gen(seed, 2)
    return torch.stack([_screen(side, rms, g)[:n, :n] for _ in range(batch)]).contiguous()


def _pyramid(c, diameter=8.4):
    pu = sp.PupilDesc(c.n_pix, diameter / c.n_pix, c.obsc)
    return pu, sp.PwfsDesc(c.pad, c.n_mod, c.n_sub, c.pup_dist, c.mod_amp)


def _amp(pu):
    a = torch.empty(pu.n_pix, pu.n_pix, device=DEV)
    sp.specula_pupil_mask(_ctx(), pu, a)
    return a


def _sensor(c, s):
    """Plan, pupil, slope computer and flat-wavefront reference of a pyramid."""
    ctx = _ctx()
    s.pu, s.pw = _pyramid(c, getattr(s, "diameter", 8.4))
    sp.specula_pwfs_plan(ctx, s.pu, s.pw)
    s.amp = _amp(s.pu)
    n, nd = c.n_pix, c.pad * c.n_sub
    if c.pad == 2 and c.pup_dist == n:
        idx = torch.from_numpy(sp.specula_valid_subaps_host(s.pu, c.n_sub)).to(DEV)
        s.slopec = sp.slopec_desc(sp.SLOPES_PYR, c.n_sub, idx)
    else:
        m = sp.specula_pyr_image_index_host(s.pu, c.pad, c.pup_dist, c.n_sub)
        s.slopec = sp.slopec_desc(sp.SLOPES_PYR_MAPS, nd, torch.from_numpy(m.ravel()).to(DEV))
    s.n_slopes = 2 * s.slopec.n_valid
    s.ref = torch.empty(s.n_slopes, device=DEV)
    flat, det = torch.zeros(n, n, device=DEV), torch.empty(nd, nd, device=DEV)
    sp.specula_pwfs_image(ctx, s.pu, s.pw, s.amp, flat, det)
    sp.specula_slopes(ctx, s.slopec, det, None, s.ref)


def _capture(call):
    """`call(stream)` as a CUDA graph."""
    ctx, st = _ctx(), torch.cuda.Stream()
    torch.cuda.synchronize()
    sp.specula_graph_begin(ctx, st)
    try:
        call(st)
    finally:
        g = sp.specula_graph_end(ctx, st)
    return g


def _prepare_frame(c, seed, s):
    n, nd = c.n_pix, c.pad * c.n_sub
    s.diameter = 39.0 if n > 220 else 8.4
    _sensor(c, s)
    s.layers, s.screens, s.t = _atmosphere(c, seed, s.diameter / n)
    s.src = sp.SourceDesc(0.0, 0.0, math.inf, 750.0)
    s.R = _randn((c.n_modes, s.n_slopes), seed, 3) / math.sqrt(s.n_slopes)
    s.rec = sp.recon_desc(c.n_modes, s.n_slopes, sp.PREC_FP32, s.R)
    s.t_dev = torch.zeros(1, dtype=torch.float64, device=DEV)
    s.phase, s.det = torch.empty(n, n, device=DEV), torch.empty(nd, nd, device=DEV)
    s.slopes, s.modes = torch.empty(s.n_slopes, device=DEV), torch.empty(c.n_modes, device=DEV)
    ctx = _ctx()

    def frame(st):
        sp.specula_atmo_extract(ctx, s.layers, s.screens, s.src, s.pu, 0.0, s.phase,
                                t_dev=s.t_dev, stream=st)
        sp.specula_pwfs_image(ctx, s.pu, s.pw, s.amp, s.phase, s.det, stream=st)
        sp.specula_slopes(ctx, s.slopec, s.det, s.ref, s.slopes, stream=st)
        sp.specula_recon(ctx, s.rec, s.slopes, s.modes, stream=st)

    s.graph = _capture(frame)


def _run_frame(s):
    s.t_dev.fill_(s.t)
    s.graph.launch()
    return dict(phase=s.phase, det=s.det, slopes=s.slopes, modes=s.modes)


GAIN, LEAK, WFS_OVER_SCI = 0.4, 0.01, 750.0 / 1650.0


def _basis(c, seed):
    """Smooth mirror modes of unit RMS over the grid."""
    b = _phases(c.n_pix, c.n_modes, 1.0, seed + 17)
    return b / b.std(dim=(1, 2), keepdim=True)


def _loop_inputs(c, seed, n_slopes):
    # a reconstructor of small norm: the integrator stays bounded on it
    R = _randn((c.n_modes, n_slopes), seed, 3) * (0.01 / math.sqrt(n_slopes))
    cmd = _randn((c.n_modes,), seed, 4) * 0.05
    return R, cmd


def _prepare_loop(c, seed, s):
    n, nd = c.n_pix, c.pad * c.n_sub
    s.diameter = 8.4
    _sensor(c, s)
    s.layers, s.screens, s.t = _atmosphere(c, seed, s.diameter / n)
    s.src = sp.SourceDesc(0.0, 0.0, math.inf, 750.0)
    s.basis = _basis(c, seed)
    s.R, s.cmd = _loop_inputs(c, seed, s.n_slopes)
    s.rec = sp.recon_desc(c.n_modes, s.n_slopes, sp.PREC_FP32, s.R)
    s.t_dev = torch.zeros(1, dtype=torch.float64, device=DEV)
    s.phase, s.dm, s.resid = (torch.empty(n, n, device=DEV) for _ in range(3))
    s.det = torch.empty(nd, nd, device=DEV)
    s.slopes, s.modes = torch.empty(s.n_slopes, device=DEV), torch.empty(c.n_modes, device=DEV)
    s.stats = torch.zeros(2, dtype=torch.float64, device=DEV)
    s.history = torch.zeros(2, device=DEV)      # RMS and Strehl of the step, float32
    ctx = _ctx()

    def step(st):
        sp.specula_atmo_extract(ctx, s.layers, s.screens, s.src, s.pu, 0.0, s.phase,
                                t_dev=s.t_dev, stream=st)
        sp.specula_dm_shape(ctx, s.basis, s.cmd, s.dm, stream=st)
        sp.specula_loop_residual(ctx, s.amp, s.phase, s.dm, WFS_OVER_SCI, s.resid, s.stats,
                                 stream=st)
        sp.specula_pwfs_image(ctx, s.pu, s.pw, s.amp, s.resid, s.det, stream=st)
        sp.specula_slopes(ctx, s.slopec, s.det, s.ref, s.slopes, stream=st)
        sp.specula_recon(ctx, s.rec, s.slopes, s.modes, stream=st)
        sp.specula_loop_integrate(ctx, GAIN, LEAK, s.modes, s.cmd, stream=st)

    s.graph = _capture(step)


def _run_loop(s):
    s.t_dev.fill_(s.t)
    s.graph.launch()
    s.history.copy_(s.stats)
    return dict(dm=s.dm, resid=s.resid, det=s.det, slopes=s.slopes, modes=s.modes, cmd=s.cmd,
                history=s.history)


def _prepare_image(c, seed, s):
    s.pu, s.pw = _pyramid(c)
    sp.specula_pwfs_plan(_ctx(), s.pu, s.pw)
    s.amp = _amp(s.pu)
    s.phase = _phases(c.n_pix, c.batch, 1.0, seed)
    nd = c.pad * c.n_sub
    s.det = torch.empty(c.batch, nd, nd, device=DEV)


def _run_image(s):
    sp.specula_pwfs_image(_ctx(), s.pu, s.pw, s.amp, s.phase, s.det)
    return s.det


def _prepare_sh(c, seed, s):
    n = c.n_sub * c.sub_pix
    s.pu = sp.PupilDesc(n, 39.0 / n, c.obsc)
    s.sh = sp.ShDesc(c.n_sub, c.sub_pix, c.fft_n)
    s.nv = sp.specula_sh_plan(_ctx(), s.pu, s.sh)
    s.amp = _amp(s.pu)
    s.phase = _phases(n, c.batch, 6.0, seed)
    idx = torch.from_numpy(sp.specula_valid_subaps_host(s.pu, c.n_sub)).to(DEV)
    s.slopec = sp.slopec_desc(sp.SLOPES_SH, c.n_sub, idx, c.fft_n)
    s.spots = torch.empty(c.batch, s.nv, c.fft_n, c.fft_n, device=DEV)
    s.slopes = torch.empty(c.batch, 2 * s.nv, device=DEV)


def _run_sh(s):
    sp.specula_sh_image(_ctx(), s.pu, s.sh, s.amp, s.phase, s.spots, s.nv)
    sp.specula_slopes(_ctx(), s.slopec, s.spots, None, s.slopes)
    return dict(spots=s.spots, slopes=s.slopes)


def _system_sensors(c):
    """Laser stars on a 45" circle (Shack-Hartmann), natural ones on 55"."""
    out = []
    n = 12 * c.n_sub_sh
    pitch_sh = 39.0 * c.n_sub_sh / 68 / n
    for k in range(c.n_sh):
        a = 2 * math.pi * k / c.n_sh
        out.append(SimpleNamespace(kind="sh", n_pix=n, pitch=pitch_sh, n_sub=c.n_sub_sh,
                                   src=sp.SourceDesc(45 * ARCSEC * math.cos(a),
                                                     45 * ARCSEC * math.sin(a), 90e3, 589.0)))
    for k in range(c.n_pyr):
        a = 0.5 + 2 * math.pi * k / c.n_pyr
        out.append(SimpleNamespace(kind="pyr", n_pix=c.n_pix, pitch=39.0 * c.n_sub_sh / 68 / c.n_pix,
                                   n_sub=c.n_sub,
                                   src=sp.SourceDesc(55 * ARCSEC * math.cos(a),
                                                     55 * ARCSEC * math.sin(a), math.inf, 750.0)))
    return out, pitch_sh


def _prepare_system(c, seed, s):
    sensors, pitch = _system_sensors(c)
    s.layers, s.screens, s.t = _atmosphere(c, seed, pitch)
    descs, n_slopes = [], 0
    for q in sensors:
        d = sp.WfsDesc()
        d.pupil, d.source = sp.PupilDesc(q.n_pix, q.pitch, 0.28), q.src
        if q.kind == "sh":
            d.kind, d.sh = sp.WFS_SH, sp.ShDesc(q.n_sub, 12, 24)
        else:
            d.kind, d.pwfs = sp.WFS_PYR, sp.PwfsDesc(2, c.n_mod, q.n_sub, q.n_pix, 3.0)
        n_slopes += 2 * len(sp.specula_valid_subaps_host(d.pupil, q.n_sub))
        descs.append(d)
    s.R = _randn((c.n_modes, n_slopes), seed, 3) / math.sqrt(n_slopes)
    s.m = sp.Mwfs(_ctx(), descs, s.layers, s.screens, s.R)
    s.ref, s.slopes = torch.empty(n_slopes, device=DEV), torch.empty(n_slopes, device=DEV)
    s.modes = torch.empty(c.n_modes, device=DEV)
    s.m.reference(s.ref, s.modes)


def _run_system(s):
    s.m.frame(s.t, s.slopes, s.modes, ref=s.ref)
    return dict(slopes=s.slopes, modes=s.modes)


def _pair_inputs(c, seed):
    """The Philox seed, the per-sample phase scale (r0 in 6-20 cm, 500 nm
    screens seen at 750 nm) and the projection of the phase on the modes."""
    r0 = 0.06 + 0.14 * torch.rand(c.n, generator=_gen(seed, 5), device=DEV)
    P = _randn((c.n_modes, c.n_pix ** 2), seed, 6) / c.n_pix ** 2
    return 1000 + int(seed) % 100000, (r0 ** (-5.0 / 6.0) * (500.0 / 750.0)).contiguous(), P


def _prepare_pairs(c, seed, s):
    _sensor(c, s)
    n, nd = c.n_pix, c.pad * c.n_sub
    s.rng_seed, s.scale, s.P = _pair_inputs(c, seed)
    s.proj = sp.recon_desc(c.n_modes, n * n, sp.PREC_FP32, s.P)
    s.scr = torch.empty(c.n, c.side, c.side, device=DEV)
    s.phase = torch.empty(c.n, n, n, device=DEV)
    s.det = torch.empty(c.n, nd, nd, device=DEV)
    s.slopes = torch.empty(c.n, s.n_slopes, device=DEV)
    s.labels = torch.empty(c.n, c.n_modes, device=DEV)


def _run_pairs(s):
    ctx, c = _ctx(), s.c
    sp.specula_screen_generate_batch(ctx, c.n, c.side, s.pu.pitch_m, 1.0, 40.0, s.rng_seed, 0,
                                     s.scr)
    sp.specula_random_phase(ctx, s.scr, c.n, c.side, c.n_pix, s.scale, s.phase)
    sp.specula_pwfs_image(ctx, s.pu, s.pw, s.amp, s.phase, s.det)
    sp.specula_slopes(ctx, s.slopec, s.det, s.ref, s.slopes)
    sp.specula_recon(ctx, s.proj, s.phase.view(c.n, -1), s.labels)
    return dict(phase=s.phase, slopes=s.slopes, labels=s.labels)


_PREC = {"fp32": sp.PREC_FP32, "bf16": sp.PREC_BF16, "bf16x2": sp.PREC_BF16X2}


def _recon_inputs(c, seed):
    R = _randn((c.n_modes, c.n_slopes), seed, 3) / math.sqrt(c.n_slopes)
    return R, _randn((c.batch, c.n_slopes), seed, 7) * 0.1


def _prepare_recon(c, seed, s):
    s.R, s.slopes = _recon_inputs(c, seed)
    prec = _PREC[c.precision]
    if prec != sp.PREC_FP32:
        hi = torch.empty(s.R.shape, dtype=torch.int16, device=DEV)
        lo = torch.empty_like(hi)
        sp.specula_recon_convert(_ctx(), s.R, sp.PREC_BF16X2, hi, lo)
        s.rec = sp.recon_desc(c.n_modes, c.n_slopes, prec, hi,
                              lo if prec == sp.PREC_BF16X2 else None)
        sp.specula_recon_reserve(_ctx(), s.rec, c.batch)
    else:
        s.rec = sp.recon_desc(c.n_modes, c.n_slopes, prec, s.R)
    s.modes = torch.empty(c.batch, c.n_modes, device=DEV)


def _run_recon(s):
    sp.specula_recon(_ctx(), s.rec, s.slopes, s.modes)
    return s.modes


def _net_weights(c, seed):
    """Uniform starting weights within 1 / sqrt(fan-in), per layer (W, b)."""
    dims = [c.n_in, c.h1, c.h2, c.n_out]
    out = []
    for l in range(3):
        g, bound = _gen(seed, 20 + l), 1.0 / math.sqrt(dims[l])
        W = (torch.rand(dims[l + 1], dims[l], generator=g, device=DEV) * 2 - 1) * bound
        b = (torch.rand(dims[l + 1], generator=g, device=DEV) * 2 - 1) * bound
        out.append((W, b))
    return out


def _network(c, seed):
    m = sp.MLP(_ctx(), (c.n_in, c.h1, c.h2, c.n_out), c.batch)
    for l, (W, b) in enumerate(_net_weights(c, seed)):
        m.set_layer(l, W.cpu().numpy(), b.cpu().numpy())
    return m


def _train_data(c, seed):
    """Standardised slopes and modes: a smooth function of the slopes plus noise."""
    X = _randn((c.steps * c.batch, c.n_in), seed, 8)
    A = _randn((c.n_in, c.n_out), seed, 9) / math.sqrt(c.n_in)
    T = torch.tanh(X @ A) + 0.1 * _randn((c.steps * c.batch, c.n_out), seed, 10)
    return X, T.contiguous()


LR, BETA1, BETA2, EPS = 1e-3, 0.9, 0.999, 1e-8


def _prepare_train(c, seed, s):
    s.mlp = _network(c, seed)
    s.X, s.T = _train_data(c, seed)
    s.loss = torch.empty(c.steps, device=DEV)


def _run_train(s):
    c, m = s.c, s.mlp
    for k in range(c.steps):
        rows = slice(k * c.batch, (k + 1) * c.batch)
        m.forward(s.X[rows])
        m.backward(s.T[rows], s.loss[k:k + 1])
        m.adam(LR, BETA1, BETA2, EPS)
    return dict(loss=s.loss, layers=[list(m.get_layer(l)) for l in range(3)])


def _prepare_infer(c, seed, s):
    s.mlp = _network(c, seed)
    s.X = _randn((c.batch, c.n_in), seed, 8)
    s.Y = torch.empty(c.batch, c.n_out, device=DEV)


def _run_infer(s):
    s.mlp.infer(s.X, s.Y)
    return s.Y


_PREPARE = dict(frame=_prepare_frame, loop=_prepare_loop, image=_prepare_image, sh=_prepare_sh,
                system=_prepare_system, pairs=_prepare_pairs, recon=_prepare_recon,
                train=_prepare_train, infer=_prepare_infer)
_RUN = dict(frame=_run_frame, loop=_run_loop, image=_run_image, sh=_run_sh, system=_run_system,
            pairs=_run_pairs, recon=_run_recon, train=_run_train, infer=_run_infer)


def prepare(case, seed):
    s = SimpleNamespace(c=SimpleNamespace(**case))
    _PREPARE[s.c.kind](s.c, seed, s)
    return s


def run(state):
    return _RUN[state.c.kind](state)


# ---- the same in 64 bits, in plain torch ----------------------------------------

def _mask(n, obsc):
    i = 2 * np.arange(n, dtype=np.int64) - n + 1
    r4 = i[None, :] ** 2 + i[:, None] ** 2
    e = float(obsc) * n
    return (r4 <= n * n) & (r4.astype(np.float64) > e * e)


def _overlap(n, n_sub):
    """Overlap of pixel i with subaperture A, in units of 1 / n_sub pixel."""
    i, A = np.arange(n)[None, :], np.arange(n_sub)[:, None]
    return np.maximum(np.minimum((i + 1) * n_sub, (A + 1) * n)
                      - np.maximum(i * n_sub, A * n), 0).astype(np.int64)


def _valid(n, obsc, n_sub):
    ov = _overlap(n, n_sub)
    return np.flatnonzero((2 * (ov @ _mask(n, obsc).astype(np.int64) @ ov.T) >= n * n).ravel())


def _amp64(n, obsc):
    return torch.from_numpy(_mask(n, obsc)).to(DEV).double()


def _extract64(layers, screens, src, n, pitch, t):
    phi = torch.zeros(n, n, dtype=torch.float64, device=DEV)
    x = (torch.arange(n, dtype=torch.float64, device=DEV) - (n - 1) / 2.0) * pitch
    for L, S in zip(layers, screens):
        cone = 1.0 - L.height_m / src.height_m

        def axis(theta, v):
            u = (x * cone + (L.height_m * theta - v * t)) / L.pitch_m + L.side / 2.0
            k = torch.floor(u)
            i0 = k.long() % L.side
            return i0, (i0 + 1) % L.side, u - k

        x0, x1, fx = axis(src.theta_x_rad, L.vx_mps)
        y0, y1, fy = axis(src.theta_y_rad, L.vy_mps)
        S = S.double()
        a = S[y0][:, x0] * (1 - fx) + S[y0][:, x1] * fx
        b = S[y1][:, x0] * (1 - fx) + S[y1][:, x1] * fx
        phi += a * (1 - fy)[:, None] + b * fy[:, None]
    return phi * (500.0 / src.wavelength_nm)


def _half_phase(n):
    """exp(i pi (n - 1) k / n): centred transforms from plain ones."""
    k = torch.arange(n, dtype=torch.float64, device=DEV)
    return torch.polar(torch.ones_like(k), math.pi * (((n - 1) * k) % (2 * n)) / n)


def _image64(c, amp, phase):
    """The modulated pyramid's detector image of one phase."""
    n, N = c.n_pix, c.pad * c.n_pix
    off, nd = (N - n) // 2, c.pad * c.n_sub
    p = _half_phase(N)
    u = (2 * torch.arange(N, dtype=torch.float64, device=DEV) - N + 1).abs()
    mk = torch.polar(torch.ones_like(u), -math.pi * c.pup_dist * u / (2 * N))
    x = torch.arange(n, dtype=torch.float64, device=DEV) - (n - 1) / 2.0
    E = amp * torch.polar(torch.ones_like(phase), phase)
    I = torch.zeros(N, N, dtype=torch.float64, device=DEV)
    for m in range(c.n_mod):
        th = 2 * math.pi * m / c.n_mod
        ph = 2 * math.pi * c.mod_amp / n * (x[None, :] * math.cos(th) + x[:, None] * math.sin(th))
        P = torch.zeros(N, N, dtype=torch.complex128, device=DEV)
        P[off:off + n, off:off + n] = E * torch.polar(torch.ones_like(ph), ph)
        F = torch.fft.fft2(P * p[:, None] * p[None, :])
        O = torch.fft.ifft2(F * mk[:, None] * mk[None, :])
        I += O.real ** 2 + O.imag ** 2
    W = torch.from_numpy(_overlap(N, nd)).to(DEV).double() / nd
    return W @ (I / c.n_mod) @ W.T


def _image_maps(c):
    """(4, n_valid) detector indices of the four pupil images."""
    valid = torch.from_numpy(_valid(c.n_pix, c.obsc, c.n_sub)).to(DEV)
    nd, two_d = c.pad * c.n_sub, c.pup_dist * c.n_sub // c.n_pix
    a, b = valid // c.n_sub, valid % c.n_sub
    maps = []
    for sx, sy in ((1, 1), (-1, 1), (-1, -1), (1, -1)):
        r0, c0 = (nd + sy * two_d - c.n_sub) // 2, (nd + sx * two_d - c.n_sub) // 2
        maps.append((r0 + a) * nd + (c0 + b))
    return torch.stack(maps)


def _slopes64(maps, det):
    q1, q2, q3, q4 = det.reshape(-1)[maps]
    T = (q1 + q2 + q3 + q4).mean()
    return torch.cat([((q1 + q4) - (q2 + q3)) / T, ((q1 + q2) - (q3 + q4)) / T])


def _sense64(c, phases):
    """Detector images and referenced slopes of (batch, n, n) phases."""
    amp, maps = _amp64(c.n_pix, c.obsc), _image_maps(c)
    ref = _slopes64(maps, _image64(c, amp, torch.zeros_like(amp)))
    dets = torch.stack([_image64(c, amp, p) for p in phases])
    return dets, torch.stack([_slopes64(maps, d) - ref for d in dets])


def _exact_frame(c, seed):
    D = 39.0 if c.n_pix > 220 else 8.4
    layers, screens, t = _atmosphere(c, seed, D / c.n_pix)
    phase = _extract64(layers, screens, sp.SourceDesc(0.0, 0.0, math.inf, 750.0), c.n_pix,
                       D / c.n_pix, t)
    det, sl = _sense64(c, phase[None])
    n_slopes = sl.shape[1]
    R = (_randn((c.n_modes, n_slopes), seed, 3) / math.sqrt(n_slopes)).double()
    return dict(phase=phase, det=det[0], slopes=sl[0], modes=R @ sl[0])


def _exact_loop(c, seed):
    layers, screens, t = _atmosphere(c, seed, 8.4 / c.n_pix)
    phase = _extract64(layers, screens, sp.SourceDesc(0.0, 0.0, math.inf, 750.0), c.n_pix,
                       8.4 / c.n_pix, t)
    R, cmd = _loop_inputs(c, seed, _image_maps(c).shape[1] * 2)
    cmd = cmd.double()
    dm = torch.einsum("k,kyx->yx", cmd, _basis(c, seed).double())
    resid = phase - dm
    det, sl = _sense64(c, resid[None])
    modes = R.double() @ sl[0]
    amp = _amp64(c.n_pix, c.obsc)
    w = amp.sum()
    mean = (amp * resid).sum() / w
    rms = torch.sqrt((amp * resid ** 2).sum() / w - mean ** 2)
    z = (amp * torch.polar(torch.ones_like(resid), resid * WFS_OVER_SCI)).sum() / w
    return dict(dm=dm, resid=resid, det=det[0], slopes=sl[0], modes=modes,
                cmd=(1 - LEAK) * cmd + GAIN * modes,
                history=torch.stack([rms, z.real ** 2 + z.imag ** 2]))


def _exact_image(c, seed):
    amp = _amp64(c.n_pix, c.obsc)
    return torch.stack([_image64(c, amp, p.double())
                        for p in _phases(c.n_pix, c.batch, 1.0, seed)])


def _spots64(n_sub, s, nf, obsc, phase):
    """(n_valid, nf, nf) spots and their centre-of-gravity slopes."""
    n = n_sub * s
    valid = torch.from_numpy(_valid(n, obsc, n_sub)).to(DEV)
    E = _amp64(n, obsc) * torch.polar(torch.ones_like(phase), phase)
    blocks = E.reshape(n_sub, s, n_sub, s).permute(0, 2, 1, 3).reshape(-1, s, s)[valid]
    P = torch.zeros(len(valid), nf, nf, dtype=torch.complex128, device=DEV)
    off = (nf - s) // 2
    P[:, off:off + s, off:off + s] = blocks
    p = _half_phase(nf)
    F = torch.fft.fft2(P * p[:, None] * p[None, :])
    I = (F.real ** 2 + F.imag ** 2) / nf ** 2
    x = torch.arange(nf, dtype=torch.float64, device=DEV) - (nf - 1) / 2.0
    tot = I.sum((1, 2))
    return I, torch.cat([(I * x).sum((1, 2)) / tot, (I * x[:, None]).sum((1, 2)) / tot])


def _exact_sh(c, seed):
    both = [_spots64(c.n_sub, c.sub_pix, c.fft_n, c.obsc, p.double())
            for p in _phases(c.n_sub * c.sub_pix, c.batch, 6.0, seed)]
    return dict(spots=torch.stack([b[0] for b in both]), slopes=torch.stack([b[1] for b in both]))


def _exact_system(c, seed):
    sensors, pitch = _system_sensors(c)
    layers, screens, t = _atmosphere(c, seed, pitch)
    parts = []
    for q in sensors:
        phase = _extract64(layers, screens, q.src, q.n_pix, q.pitch, t)
        if q.kind == "sh":
            sl = _spots64(q.n_sub, 12, 24, 0.28, phase)[1]
            parts.append(sl - _spots64(q.n_sub, 12, 24, 0.28, torch.zeros_like(phase))[1])
        else:
            g = SimpleNamespace(n_pix=q.n_pix, pad=2, n_sub=q.n_sub, pup_dist=q.n_pix,
                                n_mod=c.n_mod, mod_amp=3.0, obsc=0.28)
            parts.append(_sense64(g, phase[None])[1][0])
    sl = torch.cat(parts)
    R = (_randn((c.n_modes, len(sl)), seed, 3) / math.sqrt(len(sl))).double()
    return dict(slopes=sl, modes=R @ sl)


def _philox(c, key):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    def mul(m, x):      # high and low words of the 64-bit product
        a, b = m * (x & 0xFFFF), m * (x >> 16)
        s = (a >> 16) + (b & 0xFFFF)
        return (b >> 16) + (s >> 16), ((s & 0xFFFF) << 16) | (a & 0xFFFF)
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _noise64(count, sample, stream, seed):
    """`count` complex normals of one sample (Box-Muller on Philox words)."""
    i = torch.arange((count + 1) // 2, device=DEV)
    w = _philox([i, i >> 32, torch.full_like(i, sample), torch.full_like(i, stream)], seed)
    u = [(v.double() + 0.5) / 4294967296.0 for v in w]
    z = [torch.polar(torch.sqrt(-2 * torch.log(u[k])), 2 * math.pi * u[k + 1]) for k in (0, 2)]
    return torch.stack(z, 1).reshape(-1)[:count]


def _vk_amp(f2, df, r0, L0):
    a = torch.sqrt(0.023 * r0 ** (-5.0 / 3.0) * (f2 + 1.0 / L0 ** 2) ** (-11.0 / 6.0)) * df
    return torch.where(f2 > 0, a, torch.zeros_like(a))


def _screens64(n, M, pitch, r0, L0, seed):
    """von Karman screens by FFT with three levels of subharmonics."""
    df = 1.0 / (M * pitch)
    f = torch.fft.fftfreq(M, dtype=torch.float64, device=DEV) * M * df
    amp = _vk_amp(f[None, :] ** 2 + f[:, None] ** 2, df, r0, L0)
    pos = torch.arange(M, dtype=torch.float64, device=DEV) * pitch
    modes = []
    for p in range(3):
        g = (torch.arange(3, dtype=torch.float64, device=DEV) - 1) * df / 3.0 ** (p + 1)
        e = torch.polar(torch.ones(3, M, dtype=torch.float64, device=DEV),
                        2 * math.pi * g[:, None] * pos[None, :])
        modes.append((e, _vk_amp(g[None, :] ** 2 + g[:, None] ** 2, df / 3.0 ** (p + 1), r0, L0)))
    out = []
    for k in range(n):
        s = torch.fft.ifft2(_noise64(M * M, k, 0, seed).reshape(M, M) * amp).real * (M * M)
        sub = torch.zeros(M, M, dtype=torch.float64, device=DEV)
        noise = _noise64(27, k, 1, seed).reshape(3, 3, 3)
        for p, (e, a) in enumerate(modes):
            sub += (e.T @ (noise[p] * a) @ e).real
        out.append(s + sub - sub.mean())
    return torch.stack(out)


def _exact_pairs(c, seed):
    rng_seed, scale, P = _pair_inputs(c, seed)
    o = (c.side - c.n_pix) // 2
    scr = _screens64(c.n, c.side, 8.4 / c.n_pix, 1.0, 40.0, rng_seed)
    phase = scr[:, o:o + c.n_pix, o:o + c.n_pix] * scale.double()[:, None, None]
    return dict(phase=phase, slopes=_sense64(c, phase)[1],
                labels=phase.reshape(c.n, -1) @ P.double().T)


def _exact_recon(c, seed):
    R, s = _recon_inputs(c, seed)
    hi = R.bfloat16()
    if c.precision == "fp32":
        R64 = R.double()
    elif c.precision == "bf16":
        R64 = hi.double()
    else:
        R64 = hi.double() + (R - hi.float()).bfloat16().double()
    return s.double() @ R64.T


def _gelu64(z):
    return 0.5 * z * (1 + torch.erf(z * math.sqrt(0.5)))


def _exact_train(c, seed):
    params = [p.double().requires_grad_() for pair in _net_weights(c, seed) for p in pair]
    X, T = _train_data(c, seed)
    m, v = [torch.zeros_like(p) for p in params], [torch.zeros_like(p) for p in params]
    losses = []
    for k in range(c.steps):
        rows = slice(k * c.batch, (k + 1) * c.batch)
        h = X[rows].double()
        for l in range(3):
            h = h @ params[2 * l].T + params[2 * l + 1]
            h = _gelu64(h) if l < 2 else h
        loss = ((h - T[rows].double()) ** 2).mean()
        losses.append(loss.detach())
        grads = torch.autograd.grad(loss, params)
        lr = LR * math.sqrt(1 - BETA2 ** (k + 1)) / (1 - BETA1 ** (k + 1))
        with torch.no_grad():
            for p, g, a, b in zip(params, grads, m, v):
                a.mul_(BETA1).add_(g, alpha=1 - BETA1)
                b.mul_(BETA2).addcmul_(g, g, value=1 - BETA2)
                p -= lr * a / (b.sqrt() + EPS)
    p = [q.detach() for q in params]
    return dict(loss=torch.stack(losses), layers=[[p[2 * l], p[2 * l + 1]] for l in range(3)])


def _exact_infer(c, seed):
    h = _randn((c.batch, c.n_in), seed, 8).double()
    for l, (W, b) in enumerate(_net_weights(c, seed)):   # the weights as bf16, as stored
        h = h @ W.bfloat16().double().T + b.double()
        h = _gelu64(h) if l < 2 else h
    return h


_EXACT = dict(frame=_exact_frame, loop=_exact_loop, image=_exact_image, sh=_exact_sh,
              system=_exact_system, pairs=_exact_pairs, recon=_exact_recon, train=_exact_train,
              infer=_exact_infer)


def exact(case, seed):
    c = SimpleNamespace(**case)
    return _EXACT[c.kind](c, seed)

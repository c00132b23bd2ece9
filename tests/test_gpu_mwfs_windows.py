"""The Shack-Hartmann extraction inside the multi-sensor launch, over the ways
it reads a screen (16-byte window copies, 4-byte ones, samples straight from
the screen), against specula_atmo_extract.

Both sum the same bilinear samples in the same layer order in float32, so they
differ by roundings of one interpolation only: at most 4 ulp of the largest
partial sum (4 * 6e-8 * 8 < 2e-6 of it for up to 8 such roundings a layer pair).
"""
import numpy as np
import pytest

from gpu_common import close_checked, load_pkg, need_gpu

pytestmark = pytest.mark.gpu

N_SUB, SP = 11, 12
PITCH = 0.05


@pytest.fixture(scope="module")
def env():
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    yield torch, sp, ctx
    close_checked(sp, ctx)


# (side, screen samples per pupil pixel, floats the screen starts past a
# 16-byte boundary, layers, star height)
@pytest.mark.parametrize("side, ratio, shift, layers, height", [
    (256, 1.0, 0, 3, 90e3),            # 16-byte copies, rows that repeat (cone)
    (255, 1.0, 0, 2, 90e3),            # rows that start anywhere: 4-byte copies
    (256, 1.0, 1, 2, float("inf")),    # a screen off the 16-byte boundary
    (512, 1.5, 0, 2, float("inf")),    # samples closer than pixels: skipped rows
    (40, 1.0, 0, 2, 90e3),             # strip longer than the screen: no window
    (1024, 4.0, 0, 2, float("inf")),   # window too large to stage
    (256, 0.3, 0, 20, 90e3),           # many pixels to a sample; two chunks of layers
])
def test_sh_extraction_paths(env, side, ratio, shift, layers, height):
    torch, sp, ctx = env
    n = N_SUB * SP
    g = torch.Generator(device="cuda").manual_seed(side + layers)
    scr, lay = [], []
    for l in range(layers):
        buf = torch.randn(side * side + shift, generator=g, device="cuda")
        scr.append(buf[shift:].view(side, side))
        a = 0.9 * l + 0.3
        lay.append(sp.LayerDesc(side, PITCH / ratio, 1500.0 * l / max(1, layers / 8),
                                20 * np.cos(a), 20 * np.sin(a)))
    pu, src = sp.PupilDesc(n, PITCH, 0.28), sp.SourceDesc(2e-4, -1e-4, height, 589.0)
    d = sp.WfsDesc()
    d.pupil, d.source, d.kind, d.sh = pu, src, sp.WFS_SH, sp.ShDesc(N_SUB, SP, 24)
    m = sp.Mwfs(ctx, [d], lay, scr)
    valid = sp.specula_valid_subaps_host(pu, N_SUB)
    cover = np.zeros((n, n), dtype=bool)
    for v in valid:
        a, b = divmod(int(v), N_SUB)
        cover[a * SP:(a + 1) * SP, b * SP:(b + 1) * SP] = True
    slopes, ref = torch.empty(m.n_slopes, device="cuda"), torch.empty(n, n, device="cuda")
    got = torch.empty(n, n, device="cuda")
    for t in (0.0, 0.731):
        m.frame(t, slopes)
        m.read(0, sp.MWFS_PHASE, got)
        sp.specula_atmo_extract(ctx, lay, scr, src, pu, t, ref)
        torch.cuda.synchronize()
        a, b = got.cpu().numpy(), ref.cpu().numpy()
        assert np.max(np.abs(a - b)[cover]) <= 2e-6 * layers * (1 + np.abs(b).max())
    assert sp.specula_ctx_status(ctx) == sp.OK
    m.close()

"""GPU: the closed loop's mirror shape and residual statistics at the edges of
their splits (odd pixel counts, few modes, clusters, one and many CTAs)."""
import pytest

from gpu_common import close_checked, load_pkg, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    yield torch, sp, ctx
    close_checked(sp, ctx)


@pytest.mark.parametrize("nm,npx,off", [(1, 1, 0), (3, 31, 0), (63, 128, 0), (64, 132, 0),
                                        (129, 165 * 165, 0), (500, 25600, 0), (500, 25600, 1),
                                        (12288, 64, 0), (200, 230400, 0)])
def test_mirror_shape(env, nm, npx, off):
    torch, sp, ctx = env
    g = torch.Generator(device="cuda").manual_seed(nm + npx)
    flat = torch.randn(nm * npx + off, generator=g, device="cuda")
    B = flat[off:].view(nm, npx)
    c = torch.randn(nm, generator=g, device="cuda")
    out = torch.full((npx + 32,), 5.0, device="cuda")
    sp.specula_dm_shape(ctx, B, c, out)
    ref = c.double() @ B.double()
    mag = c.double().abs() @ B.double().abs()
    # nm / 8 additions in a warp's run, then 8 warps and up to 8 CTAs
    depth = -(-nm // 8) + 20
    assert bool(((out[:npx].double() - ref).abs() <= depth * 2.0 ** -24 * mag).all())
    assert bool((out[npx:] == 5.0).all())


@pytest.mark.parametrize("npx", [1, 255, 257, 25600, 165 * 165, 230400])
def test_residual_statistics(env, npx):
    torch, sp, ctx = env
    g = torch.Generator(device="cuda").manual_seed(npx)
    amp = (torch.rand(npx, generator=g, device="cuda") > 0.3).float()
    amp[0] = 1.0
    atm, dm = (torch.randn(npx, generator=g, device="cuda") for _ in range(2))
    resid = torch.empty(npx, device="cuda")
    k = 750.0 / 1650.0
    for _ in range(3):      # the count of finished CTAs starts anew each time
        stats = torch.full((2,), -1.0, dtype=torch.float64, device="cuda")
        sp.specula_loop_residual(ctx, amp, atm, dm, k, resid, stats)
        assert torch.equal(resid, atm - dm)
        w, r = amp.double(), resid.double()
        mean = (w * r).sum() / w.sum()
        rms = ((w * r * r).sum() / w.sum() - mean * mean).clamp(min=0).sqrt()
        # cos and sin are float32 of a float32 argument: 2^-22 each
        z = torch.polar(w, (resid * k).double()).sum() / w.sum()
        assert abs(float(stats[0] - rms)) <= 1e-7 * (1.0 + float(rms))
        assert abs(float(stats[1]) - float(z.real ** 2 + z.imag ** 2)) <= 2.0 ** -20


def test_empty_pupil(env):
    torch, sp, ctx = env
    z = torch.zeros(1000, device="cuda")
    stats = torch.full((2,), -1.0, dtype=torch.float64, device="cuda")
    sp.specula_loop_residual(ctx, z, z + 1, z, 1.0, torch.empty_like(z), stats)
    assert stats.tolist() == [0.0, 0.0]

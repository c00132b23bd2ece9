"""GPU: batched von Karman screens over their whole range of sides (odd and
even powers of two, one and several transforms per CTA) and over groups."""
import numpy as np
import pytest

from gpu_common import close_checked, load_pkg, need_gpu
from oracle import philox, screens

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    yield torch, sp, ctx
    close_checked(sp, ctx)


@pytest.mark.parametrize("M,ns", [(32, 9), (128, 3), (512, 2), (1024, 1), (2048, 1), (4096, 1)])
@pytest.mark.parametrize("L0", [25.0, float("inf")])
def test_sides(env, M, ns, L0):
    torch, sp, ctx = env
    if M > 1024 and L0 != 25.0:
        pytest.skip("one outer scale for the large sides")
    seed, s0, delta, r0 = 4321 + (5 << 33), 70000, 0.1, 0.15
    out = torch.full((ns * M * M + 64,), 3.0, device="cuda")
    sp.specula_screen_generate_batch(ctx, ns, M, delta, r0, L0, seed, s0, out)
    got = out[:ns * M * M].view(ns, M, M).cpu().numpy().astype(np.float64)
    assert bool((out[ns * M * M:] == 3.0).all())
    for b in range(ns):
        cn = philox.complex_noise(seed, s0 + b, 0, M * M).reshape(M, M)
        cs = philox.complex_noise(seed, s0 + b, 1, 27).reshape(3, 3, 3)
        ref = screens.fft_screen(M, delta, r0, L0, cn, cs)
        # float64 on both sides, one rounding to float32
        assert np.max(np.abs(got[b] - ref)) <= 2.0 ** -23 * np.max(np.abs(ref)) * 1.01


@pytest.mark.parametrize("delta,r0,L0", [(1e-6, 1e-4, 1e-3), (1e4, 1e8, 1e3), (0.05, 1e-12, 40.0)])
def test_scales(env, delta, r0, L0):
    """Amplitudes far from 1: the pairs' common power of two."""
    torch, sp, ctx = env
    M = 128
    out = torch.empty(M, M, device="cuda")
    sp.specula_screen_generate_batch(ctx, 1, M, delta, r0, L0, 99, 5, out)
    ref = screens.fft_screen(M, delta, r0, L0, philox.complex_noise(99, 5, 0, M * M).reshape(M, M),
                             philox.complex_noise(99, 5, 1, 27).reshape(3, 3, 3))
    err = np.max(np.abs(out.cpu().numpy().astype(np.float64) - ref))
    assert err <= 2.0 ** -23 * np.max(np.abs(ref)) * 1.01


def test_groups_do_not_change_a_screen(env):
    """More screens than one group of the workspace holds; each equals the
    screen generated alone."""
    torch, sp, ctx = env
    M, ns = 256, 330
    many = torch.empty(ns, M, M, device="cuda")
    one = torch.empty(M, M, device="cuda")
    sp.specula_screen_generate_batch(ctx, ns, M, 0.05, 1.0, 40.0, 7, 100, many)
    for b in (0, 109, 110, 164, 165, 329):
        sp.specula_screen_generate_batch(ctx, 1, M, 0.05, 1.0, 40.0, 7, 100 + b, one)
        assert torch.equal(many[b], one)

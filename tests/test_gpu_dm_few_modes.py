"""GPU: the mirror's shape for few modes, by a warp per 128 pixels up to 8 modes and
up to 127 on large pupils, else by the warps of a CTA together, against float64: each
pixel is off by at most its number of roundings (modes + 16) 2^-24 of the sum of
magnitudes.  The order of the sums, restated with float64 products rounded after every
operation: one chain up to 8 modes, beyond eight chains added in order."""
import pytest

from gpu_common import close_checked, load_pkg, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 64, 221, 402, 480])
def test_few_modes(n):
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    g = torch.Generator(device="cuda").manual_seed(n)
    for nm in (1, 2, 8, 9, 16, 17, 63, 127, 128):
        B = torch.randn(nm, n * n, generator=g, device="cuda")
        c = torch.randn(nm, generator=g, device="cuda")
        out = torch.full((n * n + 8,), 7.0, device="cuda")
        sp.specula_dm_shape(ctx, B, c, out[:n * n])
        assert bool((out[n * n:] == 7.0).all())
        got, b, k = out[:n * n], B.double(), c.double()
        assert bool(((got.double() - k @ b).abs() <= (nm + 16) * 2.0 ** -24 * (k.abs() @ b.abs())).all())
        if nm >= 64 and n < 400:
            continue                                # narrower tiles or a cluster: more chains
        parts = 1 if nm <= 8 else 8
        total = torch.zeros(n * n, device="cuda", dtype=torch.float64)
        for q in range(parts):
            acc = torch.zeros_like(total)
            for j in range(nm * q // parts, nm * (q + 1) // parts):
                acc = (acc + k[j] * b[j]).float().double()
            total = (total + acc).float().double()
        # (float64 rounds the exact sum before float32 does: a wrong tie in 2^29)
        assert float((got.double() != total).double().mean()) <= 1e-5
    close_checked(sp, ctx)

"""GPU: bf16 and split-bf16 products of up to 31 vectors (a warp per row), around the
rounds of loads of a lane (512 slopes each; two, three, four or eight in flight), against
float64 of the stored matrices: a lane's eight products per 256 slopes, one rounding each,
the butterfly's five, the halves' sum and the result's: 8 ceil(ns / 256) + 8 at most, each
2^-24 of the sum of magnitudes."""
import pytest

from gpu_common import close_checked, load_pkg, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("ns", [8, 248, 256, 264, 512, 768, 776, 1024, 2512])
def test_rows(split, ns):
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    for nm in (1, 9, 130):
        g = torch.Generator(device="cuda").manual_seed(nm + ns)
        R = torch.randn(nm, ns, generator=g, device="cuda")
        hi = torch.empty(R.shape, dtype=torch.int16, device="cuda")
        lo = torch.empty_like(hi)
        sp.specula_recon_convert(ctx, R, sp.PREC_BF16X2, hi, lo)
        rec = sp.recon_desc(nm, ns, sp.PREC_BF16X2 if split else sp.PREC_BF16, hi, lo if split else None)
        r = hi.view(torch.bfloat16).double()
        if split:
            r = r + lo.view(torch.bfloat16).double()
        for nb in (1, 2, 4, 5, 31):
            s = torch.randn(nb, ns, generator=g, device="cuda")
            out = torch.full((nb * nm + 8,), 7.0, device="cuda")
            sp.specula_recon(ctx, rec, s, out)
            err = (out[:nb * nm].view(nb, nm).double() - s.double() @ r.T).abs()
            depth = 8 * -(-ns // 256) + 8
            assert bool((err <= depth * 2.0 ** -24 * (s.double().abs() @ r.abs().T)).all()), nb
            assert bool((out[nb * nm:] == 7.0).all())
    close_checked(sp, ctx)

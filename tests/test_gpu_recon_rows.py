"""GPU: float32 products of 2 to 8 vectors around the rules that pick their kernel (a
row per warp up to 512, 256 or 128 slopes by the load width, four warps beyond; up to
1024 modes for more than four vectors), with the bound of tests/test_gpu_recon_f32.py:
at most ceil(ns / 64) partial sums of at most 40 roundings each."""
import pytest

from gpu_common import close_checked, load_pkg, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns", [4, 128, 129, 254, 258, 508, 512, 516, 2504, 13344])
@pytest.mark.parametrize("nm", [1, 2, 9, 1023, 1025])
def test_rows(ns, nm):
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    g = torch.Generator(device="cuda").manual_seed(nm * 7 + ns)
    R = torch.randn(nm, ns, generator=g, device="cuda")
    rec = sp.recon_desc(nm, ns, sp.PREC_FP32, R)
    for nb in (2, 3, 4, 5, 8):
        s = torch.randn(nb, ns, generator=g, device="cuda")
        out = torch.full((nb * nm + 16,), 7.0, device="cuda")
        sp.specula_recon(ctx, rec, s, out)
        err = (out[:nb * nm].view(nb, nm).double() - s.double() @ R.double().T).abs()
        mag = s.double().abs() @ R.double().abs().T
        assert bool((err <= (40 + -(-ns // 64)) * 2.0 ** -24 * mag).all()), nb
        assert bool((out[nb * nm:] == 7.0).all())
    close_checked(sp, ctx)

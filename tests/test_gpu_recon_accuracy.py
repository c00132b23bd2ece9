"""GPU: rounding error of the float32 products of batches against that of one warp per
row (lane l takes the fours l, l + 32, ... in order, then a butterfly over the lanes),
restated here with float64 products rounded after every operation.  Same inputs, at
least 8192 outputs on each side, whose r.m.s. errors have a spread of 1 % each: the
kernels' may be 5 % larger at most."""
import pytest

from gpu_common import close_checked, load_pkg, need_gpu

pytestmark = pytest.mark.gpu


def _warp_per_row(torch, R, S):
    """[vectors][rows] float32, n_slopes a multiple of 4."""
    ns = R.shape[1]
    n4 = ns // 4
    f = lambda x: x.float().double()
    P = (S.double()[:, None, :] * R.double()[None]).view(len(S), len(R), n4, 4)   # exact
    d = f(P[..., 0])
    for i in (1, 2, 3):
        d = f(d + P[..., i])
    pad = -n4 % 32
    d = torch.nn.functional.pad(d, (0, pad)).view(len(S), len(R), -1, 32)
    acc = torch.zeros_like(d[:, :, 0])
    for k in range(d.shape[2]):
        acc = f(acc + d[:, :, k])
    for o in (16, 8, 4, 2, 1):
        acc = f(acc + acc[..., torch.arange(32, device="cuda") ^ o])
    return acc[..., 0]


@pytest.mark.parametrize("nm,ns", [(128, 200), (4000, 200), (500, 512), (4000, 512), (128, 1024),
                                   (4000, 1024), (500, 2512), (4000, 2512), (1000, 5000),
                                   (4000, 13344), (500, 25600)])
def test_error_of_batches(nm, ns):
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    g = torch.Generator(device="cuda").manual_seed(nm + ns)
    R = torch.randn(nm, ns, generator=g, device="cuda")
    rec = sp.recon_desc(nm, ns, sp.PREC_FP32, R)
    rows = torch.arange(128, device="cuda") * nm // 128
    Rr = R[rows]
    for nb in (3, 8, 16, 32, 100, 512):
        vecs = torch.arange(min(nb, 32), device="cuda") * nb // min(nb, 32)
        e = e_ref = 0.0
        for _ in range(-(-8192 // (128 * len(vecs)))):
            s = torch.randn(nb, ns, generator=g, device="cuda")
            out = torch.empty(nb, nm, device="cuda")
            sp.specula_recon(ctx, rec, s, out)
            sv = s[vecs]
            exact = sv.double() @ Rr.double().T
            e += float((out[vecs][:, rows].double() - exact).square().sum())
            for v in range(0, len(vecs), 4):
                e_ref += float((_warp_per_row(torch, Rr, sv[v:v + 4]) - exact[v:v + 4]).square().sum())
        assert e <= 1.05 ** 2 * e_ref, (nb, (e / e_ref) ** 0.5)
    close_checked(sp, ctx)


@pytest.mark.parametrize("nm,ns,nb", [(4000, 513, 100), (4000, 514, 100), (3990, 1022, 65),
                                      (4000, 321, 128), (2500, 516, 200)])
def test_second_sums_of_odd_sizes(nm, ns, nb):
    """Loads of one and two floats, K tails and ragged tiles where one CTA keeps a
    second sum; the bound of tests/test_gpu_recon_f32.py."""
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    g = torch.Generator(device="cuda").manual_seed(nm + ns)
    R = torch.randn(nm, ns, generator=g, device="cuda")
    s = torch.randn(nb, ns, generator=g, device="cuda")
    out = torch.full((nb * nm + 64,), 7.0, device="cuda")
    sp.specula_recon(ctx, sp.recon_desc(nm, ns, sp.PREC_FP32, R), s, out)
    err = (out[:nb * nm].view(nb, nm).double() - s.double() @ R.double().T).abs()
    depth = 40 + -(-ns // 64)
    assert bool((err <= depth * 2.0 ** -24 * (s.double().abs() @ R.double().abs().T)).all())
    assert bool((out[nb * nm:] == 7.0).all())
    close_checked(sp, ctx)

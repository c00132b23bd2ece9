"""GPU: the float32 reconstructor products at the edges of their kernels
(batch classes, tile edges, vector widths, cluster splits) against float64."""
import numpy as np
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


# (n_modes, n_slopes, batch, floats by which R starts past a 16-byte boundary)
CASES = ([(129, 2512, nb, 0) for nb in (1, 2, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65, 200)]
         + [(nm, ns, nb, 0) for nm, ns in ((1, 1), (3, 3), (127, 62), (128, 64), (5, 66), (257, 1023))
            for nb in (1, 3, 16, 20, 70)]
         + [(130, 2510, nb, 0) for nb in (1, 7, 12, 31, 40)]      # two floats per load
         + [(130, 2512, nb, off) for off in (1, 2) for nb in (1, 7, 31, 40)]
         + [(64, 25600, 256, 0), (1000, 5000, 130, 0)])           # K over eight CTAs; none


@pytest.mark.parametrize("nm,ns,nb,off", CASES)
def test_float32_products(env, nm, ns, nb, off):
    torch, sp, ctx = env
    g = torch.Generator(device="cuda").manual_seed(nm * 7 + ns + nb)
    flat = torch.randn(nm * ns + off, generator=g, device="cuda")
    R = flat[off:].view(nm, ns)
    s = torch.randn(nb, ns, generator=g, device="cuda")
    out = torch.full((nb * nm + 64,), 7.0, device="cuda")
    sp.specula_recon(ctx, sp.recon_desc(nm, ns, sp.PREC_FP32, R), s, out)
    ref = s.double() @ R.double().T
    mag = s.double().abs() @ R.double().abs().T
    # every route adds at most ceil(ns / 64) partial sums of at most 40
    # chained roundings each: |error| <= depth 2^-24 sum |R s|
    depth = 40 + -(-ns // 64)
    err = (out[:nb * nm].view(nb, nm).double() - ref).abs()
    assert bool((err <= depth * 2.0 ** -24 * mag).all())
    assert bool((out[nb * nm:] == 7.0).all())                     # nothing past the modes
    again = torch.empty(nb, nm, device="cuda")
    sp.specula_recon(ctx, sp.recon_desc(nm, ns, sp.PREC_FP32, R), s, again)
    assert torch.equal(again.view(-1), out[:nb * nm])


def test_batched_product_in_a_graph(env):
    """A batch on the tiled kernel captured without any set-up call."""
    torch, sp, ctx = env
    nm, ns, nb = 300, 1000, 50
    R, s = torch.randn(nm, ns, device="cuda"), torch.randn(nb, ns, device="cuda")
    rec = sp.recon_desc(nm, ns, sp.PREC_FP32, R)
    eager, out = torch.empty(nb, nm, device="cuda"), torch.empty(nb, nm, device="cuda")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    sp.specula_graph_begin(ctx, st)
    sp.specula_recon(ctx, rec, s, out, stream=st)
    g = sp.specula_graph_end(ctx, st)
    g.launch(st)
    sp.specula_recon(ctx, rec, s, eager)
    torch.cuda.synchronize()
    assert torch.equal(eager, out)
    g.close()


def test_non_finite_slopes_stay_in_their_frame(env):
    torch, sp, ctx = env
    nm, ns = 200, 300
    R = torch.randn(nm, ns, device="cuda")
    for nb in (6, 40):
        s = torch.randn(nb, ns, device="cuda")
        s[3, 17] = float("nan")
        out = torch.empty(nb, nm, device="cuda")
        sp.specula_recon(ctx, sp.recon_desc(nm, ns, sp.PREC_FP32, R), s, out)
        bad = torch.isnan(out).all(dim=1)
        assert bad.nonzero().flatten().tolist() == [3]
        assert bool(torch.isfinite(out[[k for k in range(nb) if k != 3]]).all())

"""GPU: the weight-streaming inference at the edges of its kernel (odd widths,
unaligned inputs, K tails, one to four vectors) against float64 on the stored
bf16 weights."""
import math

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


@pytest.mark.parametrize("sizes", [(1, 128, 128, 1), (7, 128, 256, 3), (203, 128, 128, 37),
                                   (1026, 256, 128, 100), (2512, 1024, 1024, 500),
                                   (13344, 384, 256, 4001)])
@pytest.mark.parametrize("off", [0, 1])
def test_infer(env, sizes, off):
    torch, sp, ctx = env
    rng = np.random.default_rng(sum(sizes))
    m = sp.MLP(ctx, sizes, 128)
    W, b = [], []
    for l in range(3):
        W.append(rng.uniform(-1, 1, (sizes[l + 1], sizes[l])).astype(np.float32)
                 / math.sqrt(sizes[l]))
        b.append(rng.uniform(-1, 1, sizes[l + 1]).astype(np.float32))
        m.set_layer(l, W[l], b[l])
    for nb in (1, 2, 4):
        flat = torch.tensor(rng.standard_normal(nb * sizes[0] + off).astype(np.float32),
                            device="cuda")
        X = flat[off:].view(nb, sizes[0])
        Y = torch.full((nb * sizes[3] + 16,), 9.0, device="cuda")
        m.infer(X, Y)
        h, mag = X.double(), None
        for l in range(3):
            Wl = torch.tensor(W[l], device="cuda").bfloat16().double()
            # float32 sums of at most ceil(K / 1024) + 30 roundings per layer,
            # carried through the next layer's weights; |gelu'| < 1.13
            e_in = 0.0 if mag is None else mag
            depth = 40 + -(-sizes[l] // 1024)
            mag = (1.13 * e_in @ Wl.abs().T if l else 0.0) + depth * 2.0 ** -24 * (
                h.abs() @ Wl.abs().T + 1.0)
            h = h @ Wl.T + torch.tensor(b[l], device="cuda").double()
            if l < 2:
                h = 0.5 * h * (1 + torch.erf(h * math.sqrt(0.5)))
        assert bool(((Y[:nb * sizes[3]].view(nb, -1).double() - h).abs() <= mag).all())
        assert bool((Y[nb * sizes[3]:] == 9.0).all())
    m.close()

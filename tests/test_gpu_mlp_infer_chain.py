"""GPU: inferences back to back in one graph.  Layers of a small network are resident
together (each starts under the one before), so every layer has to read its
activations as the layer before left them: each input's output equals, bit for bit,
the one of a single call with the device idle around it."""
import numpy as np
import pytest

from gpu_common import close_checked, load_pkg, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(128, 128, 128, 20), (203, 256, 128, 37), (2512, 1024, 1024, 500)])
@pytest.mark.parametrize("nb", [1, 3])
def test_chain(sizes, nb):
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    rng = np.random.default_rng(sum(sizes) + nb)
    m = sp.MLP(ctx, sizes, 128)
    for l in range(3):
        m.set_layer(l, (rng.standard_normal((sizes[l + 1], sizes[l])) / np.sqrt(sizes[l])).astype(
            np.float32), rng.uniform(-1, 1, sizes[l + 1]).astype(np.float32))
    n = 200
    X = torch.tensor(rng.standard_normal((n, nb, sizes[0])).astype(np.float32), device="cuda")
    Y = torch.full((n, nb, sizes[3]), float("nan"), device="cuda")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    sp.specula_graph_begin(ctx, stream=st)
    for i in range(n):
        m.infer(X[i], Y[i], stream=st)
    g = sp.specula_graph_end(ctx, stream=st)
    one = torch.empty(nb, sizes[3], device="cuda")
    for replay in range(3):
        Y.fill_(float("nan"))
        torch.cuda.synchronize()
        g.launch(stream=st)
        torch.cuda.synchronize()
        for i in range(n if replay == 0 else 0):
            m.infer(X[i], one)
            torch.cuda.synchronize()
            assert torch.equal(Y[i], one), i
        if replay == 0:
            first = Y.clone()
        assert torch.equal(Y, first)
    g.close()
    m.close()
    close_checked(sp, ctx)

"""GPU: weight gradients of the learned reconstructor from one row to beyond the
batches that one launch takes (padded 4096 rows), where a tile's K slices go round
the tensor-memory accumulators up to sixteen times, against a float64 chain from the
same weights: bf16 operands, 2e-2 of each layer's norm, as tests/test_gpu_mlp.py.
Then one Adam step on them: float32, 1e-6.  And gradients left by a replayed graph,
with another batch's step captured in between: bit-identical to the eager ones."""
import numpy as np
import pytest

from gpu_common import close_checked, load_pkg, need_gpu
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

DIMS = (300, 128, 256, 60)


def _net(sp, ctx, rng, bmax):
    net = sp.MLP(ctx, DIMS, bmax)
    P = []
    for l in range(3):
        W = (rng.standard_normal((DIMS[l + 1], DIMS[l])) / np.sqrt(DIMS[l])).astype(np.float32)
        b = (0.1 * rng.standard_normal(DIMS[l + 1])).astype(np.float32)
        net.set_layer(l, W, b)
        P.append((W.astype(np.float64), b.astype(np.float64)))
    return net, P


def _data(torch, rng, batch):
    return [torch.tensor(rng.standard_normal((batch, n)).astype(np.float32), device="cuda")
            for n in (DIMS[0], DIMS[3])]


@pytest.mark.parametrize("batch", [1, 31, 130, 1100, 4096, 4200])
def test_weight_gradients_and_adam(batch):
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    rng = np.random.default_rng(batch)
    net, P = _net(sp, ctx, rng, batch)
    X, T = _data(torch, rng, batch)
    net.forward(X)
    net.backward(T)
    got = [tuple(x.astype(np.float64) for x in net.get_grad(l)) for l in range(3)]
    x, t = X.double().cpu().numpy(), T.double().cpu().numpy()
    Y, cache = omlp.forward(P, x)
    ref = omlp.backward(P, cache, Y, t)
    for l in range(3):
        assert np.linalg.norm(got[l][0] - ref[l][0]) <= 2e-2 * np.linalg.norm(ref[l][0]), l
    net.adam(1e-3)
    P = omlp.Adam(P, lr=1e-3).step(P, got)
    for l in range(3):
        W, b = net.get_layer(l)
        assert np.max(np.abs(W - P[l][0])) <= 1e-6 * (1 + np.abs(P[l][0]).max())
        assert np.max(np.abs(b - P[l][1])) <= 1e-6 * (1 + np.abs(P[l][1]).max())
    net.close()
    close_checked(sp, ctx)


def test_gradients_of_replayed_graphs():
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    rng = np.random.default_rng(5)
    net, _ = _net(sp, ctx, rng, 8200)
    data = [_data(torch, rng, b) for b in (8200, 200)]
    eager = []
    for X, T in data:
        net.forward(X)
        net.backward(T)
        eager.append([net.get_grad(l) for l in range(3)])
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    graphs = []
    for X, T in data:
        sp.specula_graph_begin(ctx, stream=st)
        net.forward(X, stream=st)
        net.backward(T, stream=st)
        graphs.append(sp.specula_graph_end(ctx, stream=st))
    for k in (0, 1, 0):
        graphs[k].launch(stream=st)
        for l in range(3):
            for a, b in zip(net.get_grad(l), eager[k][l]):
                assert np.array_equal(a, b), (k, l)
    for g in graphs:
        g.close()
    net.close()
    close_checked(sp, ctx)

"""GPU: bias gradients of the learned reconstructor, summed beside the weight
gradients (padded batch up to 4096) and by their own kernel (beyond), against
float64.  Output layer: the column sums of 2 (Y - T) / (B n_out), float32 sums of B
terms.  Hidden layers: a float64 chain from the same weights; bf16 operands, 2^-9 per
rounding, about five on the way: 2e-2 of the norm."""
import numpy as np
import pytest

from gpu_common import close_checked, load_pkg, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 31, 130, 4096, 4200])
def test_bias_gradients(batch):
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    dims = (300, 128, 256, 60)
    rng = np.random.default_rng(batch)
    net = sp.MLP(ctx, dims, batch)
    Ws, bs = [], []
    for l in range(3):
        Ws.append((rng.standard_normal((dims[l + 1], dims[l])) / np.sqrt(dims[l])).astype(np.float32))
        bs.append((0.1 * rng.standard_normal(dims[l + 1])).astype(np.float32))
        net.set_layer(l, Ws[l], bs[l])
    X = torch.tensor(rng.standard_normal((batch, dims[0])).astype(np.float32), device="cuda")
    T = torch.tensor(rng.standard_normal((batch, dims[3])).astype(np.float32), device="cuda")
    Y = torch.empty(batch, dims[3], device="cuda")
    net.forward(X, Y)
    net.backward(T)
    db = [net.get_grad(l)[1].astype(np.float64) for l in range(3)]

    dY = 2.0 * (Y.double() - T.double()) / (batch * dims[3])
    ref, mag = dY.sum(0).cpu().numpy(), dY.abs().sum(0).cpu().numpy()
    assert np.all(np.abs(db[2] - ref) <= (batch + 4) * 2.0 ** -24 * mag)
    W = [torch.tensor(w, device="cuda").double() for w in Ws]
    Z, H = [], X.double()
    for l in range(2):
        Z.append(H @ W[l].T + torch.tensor(bs[l], device="cuda").double())
        H = torch.nn.functional.gelu(Z[l])
    d = dY
    for l in (1, 0):
        d = d @ W[l + 1]
        z = Z[l].detach().requires_grad_(True)
        torch.nn.functional.gelu(z).sum().backward()
        d = d * z.grad
        ref = d.sum(0).cpu().numpy()
        assert np.linalg.norm(db[l] - ref) <= 2e-2 * np.linalg.norm(ref)
    net.close()
    close_checked(sp, ctx)

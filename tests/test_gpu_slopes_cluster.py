"""GPU: pyramid slopes at the edges of their cluster and register split: one
subaperture to more than the threads keep, quadrant and map layouts."""
import numpy as np
import pytest

from gpu_common import close_checked, load_pkg, need_gpu
from oracle import geometry, slopes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    yield torch, sp, ctx
    close_checked(sp, ctx)


@pytest.mark.parametrize("n_sub,n_valid", [(1, 1), (20, 255), (20, 256), (20, 257), (64, 2047),
                                           (64, 2049), (96, 8192), (96, 8193), (100, 10000)])
@pytest.mark.parametrize("maps", [False, True])
@pytest.mark.parametrize("nb,ref", [(1, True), (3, False)])
def test_edges(env, n_sub, n_valid, maps, nb, ref):
    torch, sp, ctx = env
    rng = np.random.default_rng(n_valid + nb)
    valid = np.sort(rng.choice(n_sub * n_sub, n_valid, replace=False)).astype(np.int32)
    side = 2 * n_sub
    det = rng.uniform(0.1, 10.0, (nb, side, side)).astype(np.float32)
    quad = geometry.pyr_quadrant_index(valid, n_sub)
    if maps:
        idx, sc_side = torch.tensor(quad.astype(np.int32).ravel(), device="cuda"), side
        sc = sp.slopec_desc(sp.SLOPES_PYR_MAPS, sc_side, idx)
    else:
        idx = torch.tensor(valid, device="cuda")
        sc = sp.slopec_desc(sp.SLOPES_PYR, n_sub, idx)
    r = rng.standard_normal(2 * n_valid).astype(np.float32) if ref else None
    out = torch.full((nb * 2 * n_valid + 8,), 4.0, device="cuda")
    sp.specula_slopes(ctx, sc, torch.tensor(det, device="cuda"),
                      None if r is None else torch.tensor(r, device="cuda"),
                      out[:nb * 2 * n_valid].view(nb, -1))
    got = out.cpu().numpy().astype(np.float64)
    for b in range(nb):
        s = slopes.pyr_slopes_maps(det[b].astype(np.float64), quad, r)
        # T: up to 60 chained roundings of positive terms; numerator, quotient
        # and reference a few more on |s| + |ref| and the four values over T
        q = det[b].astype(np.float64).ravel()[quad]
        mag = q.sum(axis=0) / np.mean(q.sum(axis=0))
        tol = 64 * 2.0 ** -24 * (np.concatenate([mag, mag]) + np.abs(s) + (0 if r is None else np.abs(r)))
        assert np.all(np.abs(got[b * 2 * n_valid:(b + 1) * 2 * n_valid] - s) <= tol)
    assert np.all(got[nb * 2 * n_valid:] == 4.0)
    assert sp.specula_ctx_status(ctx) == 0


def test_bad_index_is_reported(env):
    torch, sp, ctx = env
    idx = torch.arange(700, dtype=torch.int32, device="cuda")
    idx[650] = 30 * 30
    sc = sp.slopec_desc(sp.SLOPES_PYR, 30, idx)
    sp.specula_slopes(ctx, sc, torch.ones(60, 60, device="cuda"), None, torch.empty(1400, device="cuda"))
    assert sp.specula_ctx_status(ctx) == sp.EINVAL

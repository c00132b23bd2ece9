"""GPU: the autotuner on a batch whose slots go beyond its list of small chunks.  The
plan's own tiling (32 whole elements, one launch of each kernel for the batch) is a
candidate; the list's longest chunk takes seven times the launches.  A workspace limit
below the plan's own chunk is kept to, and the choice images as before."""
import pytest

from gpu_common import close_checked, load_pkg, need_gpu

pytestmark = pytest.mark.gpu


def test_whole_elements_are_candidates():
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    n, n_mod, n_sub, batch = 32, 24, 8, 32
    pu = sp.PupilDesc(n, 0.25, 0.2)
    pw = sp.PwfsDesc(2, n_mod, n_sub, n, 3.0)
    sp.specula_pwfs_plan(ctx, pu, pw)
    amp = torch.empty(n, n, device="cuda")
    sp.specula_pupil_mask(ctx, pu, amp)
    g = torch.Generator(device="cuda").manual_seed(1)
    ph = torch.randn(batch, n, n, generator=g, device="cuda")
    ref = torch.empty(batch, 2 * n_sub, 2 * n_sub, device="cuda")
    det = torch.empty_like(ref)
    nc = n_mod // 2 + 1
    assert sp.specula_pwfs_get_tiles(ctx, pu, pw) == (batch * nc, 1, 2)
    sp.specula_pwfs_image(ctx, pu, pw, amp, ph, ref)
    chunk, ka, passes = sp.specula_pwfs_autotune(ctx, pu, pw, amp, ph, det)
    assert passes == 2 and chunk > 64
    sp.specula_pwfs_image(ctx, pu, pw, amp, ph, det)
    assert torch.equal(det, ref)
    # 100 slots: neither the present tiling nor 8 elements, but 4 of them
    limit = 100 * n * 2 * n * 8
    chunk, ka, passes = sp.specula_pwfs_autotune(ctx, pu, pw, amp, ph, det,
                                                 max_workspace_bytes=limit)
    assert chunk <= 100
    sp.specula_pwfs_image(ctx, pu, pw, amp, ph, det)
    if passes == 2:
        assert torch.equal(det, ref)
    close_checked(sp, ctx)

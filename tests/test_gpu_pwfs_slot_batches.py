"""GPU: batches over a range of modulation slots.  A chunk of a range covers more
batch elements than one of the whole circle, and must not cover more than the
workspace holds: every element's image is the one it has alone, bit for bit (the
same float32 operations), at the plan's own tiling and at given ones."""
import pytest

from gpu_common import close_checked, load_pkg, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nsub,n_mod,slots,batch,tiles", [
    (32, 16, 7, (1, 2), 70, None),          # 33 fields, 128 slots a chunk
    (160, 40, 24, (0, 4), 25, None),        # 20 fields, 247 slots
    (480, 96, 48, (18, 25), 3, None),       # 2 fields, 25 slots
    (160, 40, 24, (3, 7), 4, (13, 1, 4)),   # packed pairs, 1 field
    (160, 40, 24, (12, 13), 9, (40, 1, 2)),
])
def test_batch_of_a_range(n, nsub, n_mod, slots, batch, tiles):
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    pu = sp.PupilDesc(n, 8.0 / n, 0.11)
    pw = sp.PwfsDesc(2, n_mod, nsub, n, 3.0)
    sp.specula_pwfs_plan(ctx, pu, pw)
    if tiles:
        sp.specula_pwfs_set_tiles(ctx, pu, pw, *tiles)
    sp.specula_pwfs_set_slots(ctx, pu, pw, *slots)
    amp = torch.empty(n, n, device="cuda")
    sp.specula_pupil_mask(ctx, pu, amp)
    g = torch.Generator(device="cuda").manual_seed(n + batch)
    ph = torch.randn(batch, n, n, generator=g, device="cuda")
    det = torch.full((batch, 2 * nsub, 2 * nsub), float("nan"), device="cuda")
    sp.specula_pwfs_image(ctx, pu, pw, amp, ph, det)
    one = torch.empty(2 * nsub, 2 * nsub, device="cuda")
    for b in range(batch):
        sp.specula_pwfs_image(ctx, pu, pw, amp, ph[b], one)
        assert torch.equal(det[b], one), b
    close_checked(sp, ctx)

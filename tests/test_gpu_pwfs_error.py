"""GPU: r.m.s. error of whole detector images against the float64 oracle, averaged over
eight modulations of phases of one radian r.m.s. (a closed loop's): below 2^-23 of the
image's norm, one float32 spacing.  Twiddles rounded to float32 can make an image as a
whole too bright or too faint by more than its pixels' own errors."""
import math

import numpy as np
import pytest

from gpu_common import close_checked, kolmogorov_phase, load_pkg, need_gpu
from oracle import pyramid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,pad,nsub", [(80, 4, 20), (80, 4, 40)])
def test_image_error(n, pad, nsub):
    torch = need_gpu()
    sp = load_pkg()
    ctx = sp.Context(0)
    pu = sp.PupilDesc(n, 8.0 / n, 0.11)
    amp = torch.empty(n, n, device="cuda")
    sp.specula_pupil_mask(ctx, pu, amp)
    a64 = amp.cpu().numpy().astype(np.float64)
    logs = []
    for k, (n_mod, r, d) in enumerate([(4, 1.1, 85), (5, 2.3, 112), (6, 3.1, 140), (7, 5.6, 151),
                                       (9, 4.7, 170), (12, 1.9, 186), (13, 5.2, 213), (24, 3.0, 240)]):
        pw = sp.PwfsDesc(pad, n_mod, nsub, d, r)
        sp.specula_pwfs_plan(ctx, pu, pw)
        ph = kolmogorov_phase(n, 8.0 / n, 0.15, seed=30 + k)
        ph = (ph / np.std(ph[a64 > 0])).astype(np.float32)
        det = torch.empty(pad * nsub, pad * nsub, device="cuda")
        sp.specula_pwfs_image(ctx, pu, pw, amp, torch.tensor(ph, device="cuda"), det)
        ref = pyramid.bin_image(pyramid.pwfs_intensity(a64, ph.astype(np.float64), pad, n_mod, r, d),
                                n // nsub)
        err = np.linalg.norm(det.cpu().numpy() - ref) / np.linalg.norm(ref)
        logs.append(math.log(err))
    assert math.exp(np.mean(logs)) <= 2.0 ** -23, [math.exp(x) for x in logs]
    close_checked(sp, ctx)

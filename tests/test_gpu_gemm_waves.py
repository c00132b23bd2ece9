"""GPU parity of the GEMMs around the rule that picks CTA pairs or single CTAs, for the
number of SMs at hand: one wave of single CTAs against a second wave of pairs, an odd
number of row tiles (a pair's second CTA without rows), and the reconstructor's
two- and three-term products, whose K slices cross from one term into the next.  GEMM:
|C - ref| <= 2e-5 sum |a b|, as tests/test_gpu_gemm.py.  Reconstructor against the
product with the stored bf16 matrices: slopes split into 16 bits (2^-16 each), the
low half's product with the low matrix left out in BF16X2 (2^-18): 4e-5 sum |r s|."""
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


@pytest.mark.parametrize("tf32", [False, True])
@pytest.mark.parametrize("rows,waves,K", [(9, 0.95, 1024), (9, 1.9, 1032), (2, 0.95, 1088),
                                          (2, 1.1, 2056)])
def test_around_the_rule(env, tf32, rows, waves, K):
    torch, sp, ctx = env
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cols = max(1, int(waves * sms / rows))      # single-CTA tiles: `waves` of the SMs
    M, N = rows * 128 - 52, cols * 256 - 3
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    B = torch.randn(N, K, generator=g, device="cuda").bfloat16()
    if tf32:
        A, B = A.float(), B.float()
    C = torch.full((M, N), float("nan"), device="cuda")
    (sp.specula_gemm_tf32 if tf32 else sp.specula_gemm_bf16)(ctx, A, B, C)
    a, b = A.double(), B.double()
    assert bool(((C.double() - a @ b.T).abs() <= 2e-5 * (a.abs() @ b.abs().T)).all())


@pytest.mark.parametrize("two", [False, True])
@pytest.mark.parametrize("n_modes,n_slopes,batch", [(3999, 1304, 1100), (4000, 2504, 2048),
                                                    (2500, 4104, 512)])
def test_reconstructor_terms(env, two, n_modes, n_slopes, batch):
    torch, sp, ctx = env
    g = torch.Generator(device="cuda").manual_seed(n_modes + batch)
    R = torch.randn(n_modes, n_slopes, generator=g, device="cuda")
    S = torch.randn(batch, n_slopes, generator=g, device="cuda")
    hi = torch.empty(R.shape, dtype=torch.int16, device="cuda")
    lo = torch.empty_like(hi)
    sp.specula_recon_convert(ctx, R, sp.PREC_BF16X2, hi, lo)
    rec = sp.recon_desc(n_modes, n_slopes, sp.PREC_BF16X2 if two else sp.PREC_BF16, hi,
                        lo if two else None)
    sp.specula_recon_reserve(ctx, rec, batch)
    m = torch.full((batch, n_modes), float("nan"), device="cuda")
    sp.specula_recon(ctx, rec, S, m)
    r = hi.view(torch.bfloat16).double()
    if two:
        r = r + lo.view(torch.bfloat16).double()
    s = S.double()
    assert bool(((m.double() - s @ r.T).abs() <= 4e-5 * (s.abs() @ r.abs().T)).all())

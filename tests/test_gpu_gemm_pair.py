"""GPU parity of the GEMMs on CTA pairs (256 x 256 tiles, taken from 76 work items
and 16 K blocks on): ragged M (a pair's second CTA partly or wholly beyond it), N
and K, an odd N (scalar stores), split-K with a shorter last slice, more items than
pairs.  |C - ref| <= 2e-5 sum_k |a_ik b_jk|, the bound of the single-CTA forms."""
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
@pytest.mark.parametrize("M,N,K,splits", [(1100, 4001, 1032, 1), (130, 2600, 8200, 8),
                                          (2048, 2560, 1024, 1), (2000, 4000, 3336, 3)])
def test_pair_parity(env, tf32, M, N, K, splits):
    torch, sp, ctx = env
    g = torch.Generator(device="cuda").manual_seed(M * 7 + N * 3 + K)
    A = torch.randn(M, K, generator=g, device="cuda").bfloat16()   # exact in tf32 too
    B = torch.randn(N, K, generator=g, device="cuda").bfloat16()
    if tf32:
        A, B = A.float(), B.float()
    C = torch.full((M * N + 64,), float("nan"), device="cuda")
    work = torch.empty(splits * M * N, device="cuda") if splits > 1 else None
    fn = sp.specula_gemm_tf32 if tf32 else sp.specula_gemm_bf16
    fn(ctx, A, B, C[:M * N].view(M, N), splits=splits, work=work)
    torch.cuda.synchronize()
    assert sp.specula_ctx_status(ctx) == 0
    a, b = A.double(), B.double()
    got = C[:M * N].view(M, N).double()
    assert bool(torch.isnan(C[M * N:]).all())
    assert bool((((got - a @ b.T).abs()) <= 2e-5 * (a.abs() @ b.abs().T)).all())

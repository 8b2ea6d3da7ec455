"""GPU checks of the tensor-core product where a CTA walks several tiles:
two accumulators used in turn, the operand ring running on from tile to tile,
a last round that is not full, fewer K steps than ring stages."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2405_12866_gb300 import build, qfs
    build.build()
    c = qfs.Context(0)
    yield c
    c.close()


def _check(ctx, M, N, K, bias, gelu, M_valid):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(M + 3 * N + 7 * K)
    A = torch.randn(M, K, generator=gen, device="cuda").to(torch.bfloat16)
    B = torch.randn(N, K, generator=gen, device="cuda").to(torch.bfloat16)
    v = torch.randn(N, generator=gen, device="cuda") if bias else None
    C32, C16 = ctx.gemm_bf16(A, B, bias=v, gelu=gelu, want_f32=True, want_bf16=True, M_valid=M_valid)
    rows = M_valid or M
    a, b = A[:rows].double(), B.double()
    ref = a @ b.T
    # FP32 accumulation of exact products: K roundings of at most 2^-23 (a
    # truncating adder) of sum |a||b|, and the bias's one.
    tol = K * 2.0 ** -23 * (a.abs() @ b.abs().T)
    if bias:
        ref = ref + v.double()
        tol = tol + 2.0 ** -24 * ref.abs()
    assert bool(((C32[:rows].double() - ref).abs() <= tol).all())
    # The bf16 copy: GELU's slope is below 1.13 and its formula 1e-5 off at
    # most, then one rounding to 8 bits.
    out = 0.5 * ref * (1 + torch.tanh(0.7978845608028654 * (ref + 0.044715 * ref ** 3))) if gelu else ref
    tol16 = 1.13 * tol + 1e-5 * (1 + ref.abs()) + 2.0 ** -8 * out.abs()
    assert bool(((C16[:rows].double() - out).abs() <= tol16).all())


# (tiles of 128 x 256, or 128 x 128 where N is no multiple of 256, on at most
# 160 SMs: one round that is just not full, two, a ragged third, five)
@pytest.mark.parametrize("M,N,K", [(128, 128, 64), (128 * 64, 512, 64), (128 * 152, 256, 192), (128 * 153, 256, 320),
                                   (128 * 161, 384, 256), (128 * 170, 1024, 64), (128 * 77, 1024, 512)])
@pytest.mark.parametrize("bias,gelu", [(True, True), (False, False)])
def test_gemm_many_tiles_per_cta(ctx, M, N, K, bias, gelu):
    _check(ctx, M, N, K, bias, gelu, 0)


def test_gemm_many_tiles_ragged_rows(ctx):
    _check(ctx, 128 * 80, 1024, 128, True, True, 128 * 79 + 5)


@pytest.mark.parametrize("M,N,K", [(128, 256, 4096), (1024, 1024, 4096), (2048, 256, 832)])
def test_gemm_split_k_items(ctx, M, N, K):
    """C32 alone with a bias: K split over work items."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=gen, device="cuda").to(torch.bfloat16)
    B = torch.randn(N, K, generator=gen, device="cuda").to(torch.bfloat16)
    v = torch.randn(N, generator=gen, device="cuda")
    C32, _ = ctx.gemm_bf16(A, B, bias=v)
    ref = A.double() @ B.double().T + v.double()
    # As above; the splits' partial sums add one rounding each.
    tol = (K + 64) * 2.0 ** -23 * (A.double().abs() @ B.double().abs().T + v.double().abs())
    assert bool(((C32.double() - ref).abs() <= tol).all())

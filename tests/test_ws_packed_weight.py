"""The weight-stationary kernel's weight block made from the packed weight: every level, the reductions that split its blocks of
128 among a quarter's warps in each way, features that end inside a block of 32."""
import pytest
import torch

LEVELS = [(1, 4), (2, 4), (1, 8), (2, 8), (1, 16), (2, 16)]


@pytest.mark.gpu
@pytest.mark.parametrize("N,M", LEVELS)
@pytest.mark.parametrize("rows,k,out", [(1, 128, 8), (145, 256, 264), (300, 384, 520), (290, 640, 512), (577, 768, 1000), (130, 896, 256)])
def test_packed_weight_and_image_give_the_same(rows, k, out, N, M):
    # the masked form's block comes from an image of the same weight, on the same kernel: the operands are equal, so the results are
    from paper_2409_09708_b200 import binding as lib
    gen = torch.Generator().manual_seed(1000 * k + 10 * N + M)
    X = torch.randn(rows, k, generator=gen).to(torch.bfloat16).cuda()
    W = (0.02 * torch.randn(out, k, generator=gen)).to(torch.bfloat16).cuda()
    bias = (0.02 * torch.randn(out, generator=gen)).to(torch.bfloat16).cuda()
    lib.elsa_set_linear_variant(lib.VARIANT_TC_SPARSE_WS)
    try:
        vals, idx = lib.elsa_nm_compress(W, N, M)
        y = lib.elsa_nm_linear(X, vals, idx, bias, out, k, N, M)
        y_image = lib.elsa_nm_linear_masked(X, W, bias, N, M)
    finally:
        lib.elsa_set_linear_variant(lib.VARIANT_AUTO)
    assert torch.equal(y, y_image)
    # and they are the masked product's: fp32 sums of k terms (error at most k 2^-24 of their absolute sum), one rounding to bf16
    keep = lib.elsa_nm_unpack(vals, idx, out, k, N, M).double()
    exact = X.double() @ keep.t() + bias.double()
    bound = 2.0 ** -8 * exact.abs() + k * 2.0 ** -24 * (X.double().abs() @ keep.abs().t() + bias.double().abs())
    assert bool(((y.double() - exact).abs() <= bound).all())

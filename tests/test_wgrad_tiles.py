"""The weight gradient's tile widths: 256 and 128 columns, one range and several, ragged edges, with the bias gradient beside it.
Small integers: every sum is exact in fp32, so the results are the exact ones after their one rounding."""
import pytest
import torch


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("rows,out,in_", [(63, 576, 192), (700, 2304, 768), (1000, 1152, 384), (1500, 768, 768), (257, 3072, 1024), (900, 520, 200), (640, 2056, 776),
                                          (130, 4096, 1024)])
@pytest.mark.parametrize("N,M", [(2, 8), (4, 4)])
def test_exact_sums(rows, out, in_, N, M, dtype):
    from paper_2409_09708_b200 import binding as lib
    gen = torch.Generator().manual_seed(rows)
    ints = lambda *s: torch.randint(-1, 2, s, generator=gen).to(dtype).cuda()
    W = torch.randn(out, in_, generator=gen).to(dtype).cuda()
    X, dY = ints(rows, in_), ints(rows, out)
    vals, idx = lib.elsa_nm_compress(W, N, M)
    _, dW, db = lib.elsa_nm_linear_backward(dY, X, vals, idx, out, in_, N, M)
    # positions kept: those of a weight of ones with W's index words (a kept value may be zero); the dense level keeps all
    keep = lib.elsa_nm_unpack(torch.ones_like(vals), idx, out, in_, N, M) != 0
    assert torch.equal(dW, torch.where(keep, dY.double().t() @ X.double(), 0.0).to(dtype))
    assert torch.equal(db.view(-1), dY.double().sum(0).to(dtype))


@pytest.mark.gpu
@pytest.mark.parametrize("rows,out,in_", [(4000, 1216, 1280), (3000, 3136, 704), (5000, 704, 3136), (6000, 1984, 1152)])
def test_bias_gradient_comes_with_the_product(rows, out, in_):
    """Shapes whose tiles fit the SM pairs in fewer ranges than dW alone would take: the bias gradient is no pass of its own (one launch more
    at most, which adds its parts), and right."""
    from paper_2409_09708_b200 import binding as lib
    gen = torch.Generator().manual_seed(rows)
    ints = lambda *s: torch.randint(-1, 2, s, generator=gen).to(torch.bfloat16).cuda()
    vals, idx = lib.elsa_nm_compress(torch.randn(out, in_, generator=gen).to(torch.bfloat16).cuda(), 2, 8)
    X, dY = ints(rows, in_), ints(rows, out)

    def launches(want):
        before = lib.elsa_launch_count()
        lib.elsa_nm_linear_backward(dY, X, vals, idx, out, in_, 2, 8, want=want)
        return lib.elsa_launch_count() - before

    assert launches(("dW", "db")) <= launches(("dW",)) + 1
    _, dW, db = lib.elsa_nm_linear_backward(dY, X, vals, idx, out, in_, 2, 8)
    keep = lib.elsa_nm_unpack(torch.ones_like(vals), idx, out, in_, 2, 8) != 0
    assert torch.equal(dW, torch.where(keep, dY.double().t() @ X.double(), 0.0).to(torch.bfloat16))
    assert torch.equal(db.view(-1), dY.double().sum(0).to(torch.bfloat16))

"""Attention of few images, sixteen query rows a CTA: row tiles and key tiles that end anywhere, warps without a key tile, both head
dimensions, scores far apart."""
import pytest
import torch


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("images,tokens,heads,d", [(1, 1, 1, 64), (1, 15, 2, 64), (2, 16, 1, 64), (1, 17, 3, 64), (3, 65, 2, 64), (1, 197, 12, 64), (2, 255, 1, 64),
                                                   (1, 256, 2, 64), (1, 66, 1, 32), (2, 145, 3, 32), (1, 256, 4, 32)])
@pytest.mark.parametrize("spread", [1.0, 6.0])
def test_few_images(images, tokens, heads, d, dtype, spread):
    from paper_2409_09708_b200 import binding as lib
    dim = heads * d
    gen = torch.Generator().manual_seed(tokens * 100 + heads)
    qkv = (spread * torch.randn(images * tokens, 3 * dim, generator=gen)).to(dtype).cuda()
    guard = torch.full((images * tokens + 64, dim), 7.0, dtype=dtype, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    lib.elsa_attention(qkv, tokens, heads, guard[:images * tokens], dev_status=status)
    q, k, v = qkv.double().view(images, tokens, 3, heads, d).permute(2, 0, 3, 1, 4)
    ref = torch.softmax(q @ k.transpose(-1, -2) / d ** 0.5, -1) @ v
    # one rounding of the result, and the probabilities' rounding for the second product: u / 4 relative each, |sum p v| <= max |v|;
    # the exponent's argument is in fp32, 2^-24 of it as a relative error of p
    u = 2.0 ** -7 if dtype == torch.bfloat16 else 2.0 ** -10
    top = v.abs().amax(dim=-2, keepdim=True)
    scores = (q @ k.transpose(-1, -2) / d ** 0.5).abs().amax(dim=(-1, -2), keepdim=True)
    bound = u * ref.abs() + (u / 2) * top + 1e-5 + 2.0 ** -21 * scores * top
    got = guard[:images * tokens].double().view(images, tokens, heads, d).permute(0, 2, 1, 3)
    assert int(status.item()) == 0
    assert bool(((got - ref).abs() <= bound).all())
    assert bool((guard[images * tokens:] == 7.0).all())


@pytest.mark.gpu
@pytest.mark.parametrize("images,tokens,heads", [(4, 208, 8), (4, 224, 6), (5, 224, 6), (10, 209, 3), (3, 256, 9)])
def test_either_side_of_the_rule(images, tokens, heads):
    """Heads of 64: up to 208 tokens 444 row tiles of sixteen, beyond 370 (of 148 SMs)."""
    test_few_images(images, tokens, heads, 64, torch.bfloat16, 1.0)

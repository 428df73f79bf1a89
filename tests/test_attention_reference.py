"""Attention where the scores' maximum moves along a row: the kernel takes the first unit's maximum as the reference of the
exponentials and follows a later one that lies far above it by rescaling what it has.  Scores that climb by more than the
slack from unit to unit, that climb within it, that fall, one key far above all others at either end of a unit, rows that differ
from lane to lane; token counts around the units of 16 and 32 keys and the 128-row tiles.  Tolerance as for every attention here:
|err| <= u |ref| + (u / 2) max|v| + 1e-5 with u one unit in the last place (the rescaling is by powers of two)."""
import numpy as np
import pytest
import torch

from oracle import elsa_block_oracle as bo
from paper_2409_09708_b200 import synth

SHAPES = [(3, 17, 1, 64), (2, 64, 2, 64), (2, 65, 2, 64), (1, 128, 1, 32), (2, 129, 2, 64), (2, 197, 3, 64), (1, 256, 2, 64), (1, 200, 2, 32),
          (3, 65, 2, 32), (2, 80, 1, 32), (2, 97, 3, 32)]


def profile(kind, tokens):
    t = np.arange(tokens)
    if kind == "steep":
        return 0.9 * t                                   # 14 to 29 natural units a unit of keys
    if kind == "gentle":
        return 0.05 * t
    if kind == "falling":
        return -0.9 * t
    s = np.zeros(tokens)
    s[{"spike_last": tokens - 1, "spike_16": min(16, tokens - 1), "spike_47": min(47, tokens - 1)}[kind]] = 60.0
    return s


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("kind", ["steep", "gentle", "falling", "spike_last", "spike_16", "spike_47"])
def test_moving_maximum(kind, dtype):
    from paper_2409_09708_b200 import binding as lib
    u = 2.0 ** -7 if dtype == torch.bfloat16 else 2.0 ** -10
    for images, tokens, heads, d in SHAPES:
        dim = heads * d
        qkv = synth.randn((images * tokens, 3 * dim), tokens, 1.0, torch.float32)
        # column 0 of every head: the score's profile for odd rows, nothing for even ones
        row = torch.arange(images * tokens) % tokens
        prof = torch.from_numpy(profile(kind, tokens)).float()
        for h in range(heads):
            qkv[:, h * d] = (row % 2).float() * d ** 0.5
            qkv[:, dim + h * d] = prof[row]
        qkv = qkv.to(dtype)
        a = torch.empty((images * tokens, dim), dtype=dtype, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        lib.elsa_attention(qkv.cuda(), tokens, heads, a=a, dev_status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0, "device status %#x" % int(status.item())
        q64 = qkv.double().numpy()
        ref = bo.attention(q64, tokens, heads)
        err = np.abs(a.double().cpu().numpy() - ref)
        assert (err <= u * np.abs(ref) + u / 2 * np.abs(q64[:, 2 * dim:]).max() + 1e-5).all(), (images, tokens, heads, d, float(err.max()))

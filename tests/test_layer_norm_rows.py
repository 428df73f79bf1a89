"""LayerNorm at the compiled widths, alone and behind a residual add: rows below, at and above what a warp, a block and a wave of
blocks take at a time, one wave and several.  Through the block's stages: x1 = LN(x) and, from the library's own stored x2,
x3 = LN(x2), against fp64 statistics of the stored rows: one rounding, |err| <= u |ref| + 4e-6 (u half a unit in the last place
of a normal value, the rest for fp32 statistics of values of order one and the subnormal range)."""
import numpy as np
import pytest
import torch

from paper_2409_09708_b200 import synth

CASES = [(1, 128), (9, 128), (163000, 128), (65, 192), (5000, 192), (17, 256), (40000, 256), (33, 384), (7000, 384), (8, 512), (5000, 512),
         (9, 768), (3600, 768), (1, 1024), (2500, 1024), (100, 320)]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("case", CASES, ids=["%dx%d" % c for c in CASES])
def test_layer_norm_rows(case, dtype):
    from paper_2409_09708_b200 import binding as lib
    rows, dim = case
    mlp = 64
    x = synth.randn((rows, dim), 5, 1.0, dtype, "cuda") + 0.5
    lin = {}
    for i, (name, k, o) in enumerate((("qkv", dim, 3 * dim), ("proj", dim, dim), ("fc1", dim, mlp), ("fc2", mlp, dim))):
        lin[name] = (synth.randn((o, k), 10 + i, 1.0 / np.sqrt(k), dtype, "cuda"), None, synth.randn((o,), 20 + i, 0.02, dtype, "cuda"), 4, 4)
    ln = [(synth.randn((dim,), 30 + i, 0.1, dtype, "cuda") + (1.0 if i % 2 == 0 else 0.0)).to(dtype) for i in range(4)]
    w, keep = lib.make_block_weights(*ln, lin)
    total, off = lib.elsa_vit_block_scratch_bytes(rows, dim, mlp, w, lib.dtype_code(dtype))
    scratch = torch.zeros(total, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    y = torch.empty_like(x)
    lib.elsa_vit_block(x, mlp, w, y=y, scratch=scratch, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0, "device status %#x" % int(status.item())
    u = 2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -11
    region = lambda n: lib.block_region(scratch, off, n, rows, dim, dtype).double()
    for got, src, g, b in ((region("x1"), x.double(), ln[0], ln[1]), (region("x3"), region("x2"), ln[2], ln[3])):
        mean = src.mean(1, keepdim=True)
        ref = (src - mean) / ((src - mean).pow(2).mean(1, keepdim=True) + 1e-6).sqrt() * g.double() + b.double()
        assert ((got - ref).abs() <= u * ref.abs() * (1 + 2.0 ** -10) + 4e-6).all(), float(((got - ref).abs() - u * ref.abs()).max())

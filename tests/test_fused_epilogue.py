"""The dense pair kernel's epilogue with GELU and with a residual, chunk by chunk in 16 warps: widths that leave a warp one
chunk or none (out of 64, 72, 136, 200, 1000), rows around the 256-row tile, one K block and several, many tiles per SM
pair; through the chained block, each stage against fp64 from the library's own stored inputs (|err| <= u (|ref| +
|linear|) + 5e-4, u one unit in the last place: the tolerance of the block's stages)."""
import numpy as np
import pytest
import torch

from paper_2409_09708_b200 import synth

CASES = [(257, 64, 136), (1, 64, 200), (300, 72, 1000), (20000, 64, 72), (513, 200, 64), (40000, 128, 512)]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16], ids=["f16", "bf16"])
@pytest.mark.parametrize("case", CASES, ids=["%dx%dx%d" % c for c in CASES])
def test_gelu_and_residual_on_the_pair_kernel(case, dtype):
    from paper_2409_09708_b200 import binding as lib
    rows, dim, mlp = case
    x = synth.randn((rows, dim), 5, 1.0, dtype, "cuda")
    dense = {}
    for i, (name, k, o) in enumerate((("qkv", dim, 3 * dim), ("proj", dim, dim), ("fc1", dim, mlp), ("fc2", mlp, dim))):
        dense[name] = (synth.randn((o, k), 10 + i, 2.0 / np.sqrt(k), dtype, "cuda"), synth.randn((o,), 20 + i, 0.02, dtype, "cuda"))
    ln = [(synth.randn((dim,), 30 + i, 0.1, dtype, "cuda") + (1.0 if i % 2 == 0 else 0.0)).to(dtype) for i in range(4)]
    w, keep = lib.make_block_weights(*ln, {n: (W, None, b, 4, 4) for n, (W, b) in dense.items()})
    code = lib.dtype_code(dtype)
    total, off = lib.elsa_vit_block_scratch_bytes(rows, dim, mlp, w, code)
    scratch = torch.zeros(total, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    guard = torch.full((rows + 300, dim), 7.0, dtype=dtype, device="cuda")
    lib.elsa_set_linear_variant(lib.VARIANT_TC_PAIR)
    try:
        lib.elsa_vit_block(x, mlp, w, y=guard[:rows], scratch=scratch, dev_status=status)
        torch.cuda.synchronize()
    finally:
        lib.elsa_set_linear_variant(lib.VARIANT_AUTO)
    assert int(status.item()) == 0, "device status %#x" % int(status.item())
    assert (guard[rows:] == 7.0).all()
    region = lambda n, c: lib.block_region(scratch, off, n, rows, c, dtype).double()
    u = 2.0 ** -7 if dtype == torch.bfloat16 else 2.0 ** -10

    def check(got, ref, lin):
        ref = ref.to(dtype).double()
        assert ((got - ref).abs() <= u * (ref.abs() + lin.abs()) + 5e-4).all()

    def product(name, a):
        W, b = dense[name]
        return a @ W.double().t() + b.double()

    lin = product("fc1", region("x3", dim))
    check(region("h", mlp), 0.5 * lin * (1.0 + torch.erf(lin / 2.0 ** 0.5)), lin)
    lin = product("proj", region("a", dim))
    check(region("x2", dim), x.double() + lin, lin)
    lin = product("fc2", region("h", mlp))
    check(guard[:rows].double(), region("x2", dim) + lin, lin)

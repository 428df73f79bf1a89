"""A block's residuals added in the epilogues of the weight-stationary and streaming kernels: row counts that end inside a step of 16
rows, a warp's run and a tile.  LayerNorm with gains of zero, small integers and GELU at 8 and 16 (where it is its argument) make every
sum exact in fp32, so the results are the exact ones after their one rounding."""
import pytest
import torch


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("rows", [1, 16, 47, 145, 193, 300, 450, 1155, 5000])
@pytest.mark.parametrize("kernel,dim,mlp", [("WS", 256, 512), ("WS", 768, 896), ("ST", 256, 1536), ("ST", 128, 384)])
def test_exact_block(kernel, dim, mlp, rows, dtype):
    from paper_2409_09708_b200 import binding as lib
    gen = torch.Generator().manual_seed(rows + dim)
    ints = lambda lo, hi, *s: torch.randint(lo, hi + 1, s, generator=gen).to(dtype).cuda()
    x = ints(-8, 8, rows, dim)
    ln = [torch.zeros(dim, dtype=dtype, device="cuda"), ints(-1, 1, dim), torch.zeros(dim, dtype=dtype, device="cuda"), ints(-1, 1, dim)]
    linears, dense = {}, {}
    for name, k, o in (("qkv", dim, 3 * dim), ("proj", dim, dim), ("fc1", dim, mlp), ("fc2", mlp, dim)):
        W = ints(-1, 1, o, k) if name != "fc1" else torch.zeros(o, k, dtype=dtype, device="cuda")
        vals, idx = lib.elsa_nm_compress(W, 1, 8)
        bias = ints(-3, 3, o) if name != "fc1" else 8 * ints(1, 2, o)
        linears[name] = (vals, idx, bias, 1, 8)
        dense[name] = (lib.elsa_nm_unpack(vals, idx, o, k, 1, 8).double(), bias.double())
    w, keep = lib.make_block_weights(*ln, linears, eps=1e-6)
    need, off = lib.elsa_vit_block_scratch_bytes(rows, dim, mlp, w, lib.dtype_code(dtype))
    scratch = lib.alloc_workspace(need)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    guard = torch.full((rows + 256, dim), 7.0, dtype=dtype, device="cuda")
    lib.elsa_set_linear_variant(lib.VARIANT_TC_SPARSE_WS if kernel == "WS" else lib.VARIANT_TC_SPARSE_ST)
    try:
        lib.elsa_vit_block(x, mlp, w, y=guard[:rows], scratch=scratch, dev_status=status)       # the stand-in a = V
        torch.cuda.synchronize()
    finally:
        lib.elsa_set_linear_variant(lib.VARIANT_AUTO)
    assert int(status.item()) == 0
    apply = lambda v, name: v @ dense[name][0].t() + dense[name][1]
    a = apply(ln[1].double().expand(rows, dim), "qkv")[:, 2 * dim:].to(dtype).double()
    x2 = (x.double() + apply(a, "proj")).to(dtype)
    y = (x2.double() + apply(dense["fc1"][1].expand(rows, mlp), "fc2")).to(dtype)
    assert torch.equal(lib.block_region(scratch, off, "x2", rows, dim, dtype), x2)
    assert torch.equal(guard[:rows], y)
    assert bool((guard[rows:] == 7.0).all())


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("kernel", ["WS", "ST"])
@pytest.mark.parametrize("rows,dim,mlp", [(25000, 256, 512), (5400, 640, 256), (18600, 128, 384)])
def test_several_tiles_a_pair(rows, dim, mlp, kernel, dtype):
    """A pair takes a second tile in which some of its warps have no rows (25000: the last of 143 tiles of 176 rows has 8) or no features
    (640: the third block of 256 has 128), while the stores of the first one still read the staging rows.  Three times over: nothing but
    an order of reads and writes can go wrong, and that need not show at once."""
    for _ in range(3):
        test_exact_block(kernel, dim, mlp, rows, dtype)

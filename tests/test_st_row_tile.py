"""The streaming sparse kernel's row tiles: row counts for which it takes 128 to 224 token rows a tile, odd and even numbers of
16-row steps for the epilogue's two warps, a ragged last tile, several layers in a launch; rows after the output stay.  Small
integers: every product and sum is exact in fp32, so the result is the oracle's after its one rounding."""
import numpy as np
import pytest
import torch

from oracle import elsa_oracle as eo
from paper_2409_09708_b200 import synth

CASES = [(1, 256, 256), (129, 1024, 512), (1600, 256, 768), (2960, 256, 768), (3152, 384, 760), (3553, 256, 768), (4097, 128, 1024), (4740, 256, 1024)]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("case", CASES, ids=["%dx%dx%d" % c for c in CASES])
def test_row_tiles(case, dtype):
    from paper_2409_09708_b200 import binding as lib
    rows, in_, out = case
    rng = np.random.default_rng(rows)
    ints = lambda *s: torch.from_numpy(rng.integers(-3, 4, s).astype(np.float32)).to(dtype)
    X, W, b = ints(rows, in_), ints(out, in_), ints(out)
    vals, idx = lib.elsa_nm_compress(W.cuda(), 2, 8)
    guard = torch.full((rows + 256, out), 7.0, dtype=dtype, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    lib.elsa_set_linear_variant(lib.VARIANT_TC_SPARSE_ST)
    try:
        lib.elsa_nm_linear(X.cuda(), vals, idx, b.cuda(), out, in_, 2, 8, Y=guard[:rows], dev_status=status)
        torch.cuda.synchronize()
    finally:
        lib.elsa_set_linear_variant(lib.VARIANT_AUTO)
    assert int(status.item()) == 0, "device status %#x" % int(status.item())
    Wm = W.double() * torch.from_numpy(eo.nm_mask(synth.bits(W), 2, 8).astype(np.float64))
    ref = (X.double() @ Wm.t() + b.double()).to(dtype)
    assert torch.equal(guard[:rows].cpu(), ref)
    assert (guard[rows:] == 7.0).all()

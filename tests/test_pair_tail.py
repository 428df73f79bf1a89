"""The dense pair kernel where a layer's tiles overflow the last full wave of SM pairs by a few and the last rows get narrow
tiles: one row tile over and several, the last tile full, ragged and of one row, widths around the tiles', 16-bit and INT8.  Small
integers: sums are exact, so the result is the product after its one rounding; rows after the output stay."""
import numpy as np
import pytest
import torch

CASES = [(74 * 256 + 1, 64, 256), (75 * 256, 128, 136), (76 * 256 - 1, 64, 200), (37 * 256 + 3, 192, 512), (49 * 256 + 64, 64, 2304),
         (98 * 256 + 128, 64, 768), (149 * 256 + 17, 64, 72)]


def ints(rng, low, high, *shape):
    return torch.from_numpy(rng.integers(low, high, shape).astype(np.float32))


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("case", CASES, ids=["%dx%dx%d" % c for c in CASES])
def test_narrow_tiles_for_the_last_rows(case, dtype):
    from paper_2409_09708_b200 import binding as lib
    rows, in_, out = case
    rng = np.random.default_rng(out)
    X, W, b = (ints(rng, -3, 4, *s).to(dtype).cuda() for s in ((rows, in_), (out, in_), (out,)))
    vals, idx = lib.elsa_nm_compress(W, 4, 4)
    guard = torch.full((rows + 300, out), 7.0, dtype=dtype, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    lib.elsa_set_linear_variant(lib.VARIANT_TC_PAIR)
    try:
        lib.elsa_nm_linear(X, vals, idx, b, out, in_, 4, 4, Y=guard[:rows], dev_status=status)
        torch.cuda.synchronize()
    finally:
        lib.elsa_set_linear_variant(lib.VARIANT_AUTO)
    assert int(status.item()) == 0, "device status %#x" % int(status.item())
    assert torch.equal(guard[:rows], (X.double() @ W.double().t() + b.double()).to(dtype))
    assert (guard[rows:] == 7.0).all()


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES[:4], ids=["%dx%dx%d" % c for c in CASES[:4]])
def test_int8(case):
    from paper_2409_09708_b200 import binding as lib
    rows, in_, out = case
    rng = np.random.default_rng(rows)
    X, W = (ints(rng, -9, 10, *s).to(torch.int8).cuda() for s in ((rows, in_), (out, in_)))
    scale, b = torch.full((out,), 0.5, device="cuda"), ints(rng, -3, 4, out).half().cuda()
    vals, idx = lib.elsa_nm_compress_i8(W, 4, 4)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Y = lib.elsa_nm_linear_i8(X, 0.25, vals, idx, scale, b, out, in_, 4, 4, torch.float16, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0, "device status %#x" % int(status.item())
    assert torch.equal(Y, (X.double() @ W.double().t() * 0.125 + b.double()).half())

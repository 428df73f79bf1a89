"""The bias gradient as parts of the weight gradient's launch, and the transposed masked weight straight from the packed form:
rows below, at and above the 64-row K block (so that some tile columns take no block at all), features and columns around the
256 and 64 wide tiles, the reduction cut and whole, more tiles than SM pairs (the separate column sums), every kept width the
transposition is compiled for and one it is not.

Small integers make every product and sum exact in fp32, so the results equal the oracle's after its one rounding.  With random
values the bound is that of the additions one value goes through (9001 rows, 776 features, 768 columns: a tile column has 8 of a
range's 24 K blocks, one to a running sum: 4 products of 16 rows, then 8 running sums and 18 parts): fewer than 96 units of 2^-23
(truncation allowed for) of sum |dY|, a tenth of what one row contributes, and the rounding adds at most 2^-9 (2^-12) of twice
the result."""
import numpy as np
import pytest
import torch

from oracle import elsa_backward_oracle as bwo
from oracle import elsa_oracle as eo
from paper_2409_09708_b200 import synth

CASES = [
    (1, 64, 8, 2, 4), (63, 256, 256, 1, 8), (64, 520, 264, 2, 8), (65, 264, 520, 4, 8), (129, 768, 768, 3, 8), (300, 1032, 64, 1, 4),
    (640, 2560, 128, 5, 16), (257, 72, 96, 3, 4), (200, 136, 1024, 4, 4), (130, 2048, 2048, 2, 4), (130, 4096, 2312, 2, 8),
]


def backward(dY, X, W, N, M, want):
    from paper_2409_09708_b200 import binding as lib
    vals, idx = lib.elsa_nm_compress(W.cuda(), N, M)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = lib.elsa_nm_linear_backward(dY.cuda(), X.cuda(), vals, idx, W.shape[0], W.shape[1], N, M, want=want, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0, "device status %#x" % int(status.item())
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("case", CASES, ids=["%dx%dx%d_%d:%d" % c for c in CASES])
def test_integers_are_exact(case, dtype):
    rows, in_, out, N, M = case
    rng = np.random.default_rng(rows + in_)
    ints = lambda *s: torch.from_numpy(rng.integers(-2, 3, s).astype(np.float32)).to(dtype)
    dY, X, W = ints(rows, out), ints(rows, in_), ints(out, in_)
    code = eo.F16 if dtype == torch.float16 else eo.BF16
    refs = bwo.linear_backward_f64(synth.bits(dY), synth.bits(X), synth.bits(W), N, M, code)
    for want in (("dX", "dW", "db"), ("dX", "db")):      # with the weight's gradient, and the column sums on their own
        got = backward(dY, X, W, N, M, want)
        for name, g, ref in zip(("dX", "dW", "db"), got, refs):
            if name in want:
                assert torch.equal(g.cpu().double(), torch.from_numpy(np.asarray(ref)).to(dtype).double()), (name, want)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
def test_sums_of_random_values(dtype):
    rows, in_, out = 9001, 768, 776
    dY, X, W = (synth.randn(s, i, 0.5, dtype) for i, s in enumerate(((rows, out), (rows, in_), (out, in_))))
    db = backward(dY, X, W, 2, 4, ("dW", "db"))[2].cpu().double()
    d = dY.double()
    half_unit = 2.0 ** -9 if dtype == torch.bfloat16 else 2.0 ** -12
    assert ((db - d.sum(0)).abs() <= 96 * 2.0 ** -23 * d.abs().sum(0) + half_unit * d.sum(0).abs() * 2).all()


# Rows in the thousands, where a part of the sums has many K blocks: (rows, in, out) with 1, 2, 3 and 4 tile columns that take the K
# blocks in turn, the reduction cut into 8, 4, 2 ranges and whole, remainders of the 64-row block, parts of unequal length,
# and the row count above which the sums are a pass of their own.
LONG = [(9001, 64, 256), (25216, 256, 256), (25217, 512, 1024), (9023, 1024, 520), (12608, 768, 2304), (39400, 768, 768), (4159, 1024, 4096),
        (65536, 64, 256), (65600, 256, 264), (409600, 64, 72), (409601, 64, 72)]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("case", LONG, ids=["%dx%dx%d" % c for c in LONG])
def test_long_sums_of_integers_are_exact(case, dtype):
    """Integers up to 3, so that losing or repeating one row shows: |sums| < 2^24 in any order, one rounding at the end."""
    rows, in_, out = case
    rng = np.random.default_rng(rows)
    ints = lambda *s: torch.from_numpy(rng.integers(-3, 4, s).astype(np.float32)).to(dtype)
    dY, X, W = ints(rows, out), ints(rows, in_), ints(out, in_)
    db = backward(dY, X, W, 2, 4, ("dW", "db"))[2].cpu()
    assert torch.equal(db.double(), dY.double().sum(0).to(dtype).double())


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("case", [(25216, 64, 256), (65536, 64, 256), (401408, 64, 128), (420000, 64, 128)], ids=lambda c: "%dx%dx%d" % c)
def test_long_sums_of_one_sign_lose_nothing_to_their_length(case, dtype):
    """Values of one sign are where a running fp32 sum loses most.  At most 400 accumulations follow one another in a running sum and
    8 such sums and 8 ranges are added after, each losing at most a unit (2^-23, truncation allowed for); as a pass of its own 64
    additions of a thread, 8 of threads and one for every 512 rows, each rounded to nearest (2^-24).  The rounding at the end adds
    half a unit of the type."""
    rows, in_, out = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows)
    dY = (torch.rand((rows, out), device="cuda", generator=gen) * 0.1 + 0.05).to(dtype)
    X = torch.zeros((rows, in_), dtype=dtype, device="cuda")
    W = synth.randn((out, in_), 3, 0.05, dtype)
    db = backward(dY, X, W, 2, 4, ("dW", "db"))[2].double()
    exact = dY.double().sum(0)
    half_unit = 2.0 ** torch.floor(torch.log2(exact)) * (2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -11)
    chain = max(416 * 2.0 ** -23, (72 + rows / 512) * 2.0 ** -24)
    assert ((db - exact).abs() <= half_unit + chain * exact).all(), float(((db - exact).abs() / half_unit).max())

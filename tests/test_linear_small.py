"""The few-rows linear kernel (weight tiles expanded from the packed form, reduction cut over a cluster) against the
oracle, with the tolerances of the other linear kernels: relative Frobenius 5e-3, |err| <= 1e-2 (|ref| + 1).

Sizes: rows around the 128-row tile, `in` around the 64-wide K block and at 1, 2, 4 and 8 ranges of the reduction
(8 ranges need 32 K blocks), `out` below a 64-feature tile, ragged, and several waves of tiles; levels with each of the
expansion's load widths for every group size.
"""
import numpy as np
import pytest
import torch

from oracle import elsa_oracle as eo
from paper_2409_09708_b200 import synth

CASES = [(1, 128, 64, 1, 4), (127, 64, 8, 2, 4), (128, 72, 72, 3, 4), (129, 1032, 136, 2, 8), (197, 768, 768, 4, 8),
         (197, 3072, 768, 1, 8), (300, 200, 384, 3, 8), (50, 256, 320, 7, 8), (64, 512, 1000, 2, 16), (197, 1040, 72, 15, 16),
         (33, 768, 104, 5, 16), (197, 768, 2304, 8, 8), (70, 3072, 64, 4, 4), (1700, 320, 3080, 2, 4), (1700, 384, 3072, 8, 8)]


@pytest.fixture(scope="module")
def lib():
    from paper_2409_09708_b200 import binding
    return binding


def close(Y, ref):
    err = Y.double().cpu().numpy() - ref
    assert np.isfinite(err).all()
    assert np.linalg.norm(err) <= 5e-3 * np.linalg.norm(ref)
    assert (np.abs(err) <= 1e-2 * (np.abs(ref) + 1.0)).all()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16], ids=["f16", "bf16"])
@pytest.mark.parametrize("case", CASES, ids=["%dx%dx%d_%dof%d" % c for c in CASES])
def test_small_linear_matches_oracle_packed_and_masked(lib, case, dtype):
    rows, in_, out, N, M = case
    X = synth.randn((rows, in_), 3 * rows + in_, synth.X_STD, dtype)
    W = synth.randn((out, in_), 5 * out + in_, synth.W_STD, dtype)
    bias = synth.randn((out,), 7 * out, synth.B_STD, dtype)
    ovals, oidx, _ = eo.nm_compress(synth.bits(W), N, M)
    ref = eo.nm_linear_f64(synth.bits(X), ovals, oidx, synth.bits(bias), out, in_, N, M, eo.F16 if dtype == torch.float16 else eo.BF16)
    Xd, Wd, bd = X.cuda(), W.cuda(), bias.cuda()
    vals, idx = lib.elsa_nm_compress(Wd, N, M)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    guard = torch.full((rows + 130, out), 7.0, dtype=dtype, device="cuda")        # rows after the last stay
    lib.elsa_set_linear_variant(lib.VARIANT_TC_SMALL)
    try:
        Y = lib.elsa_nm_linear(Xd, vals, idx, bd, out, in_, N, M, Y=guard[:rows], dev_status=status)
        Y_masked = lib.elsa_nm_linear_masked(Xd, Wd, bd, N, M, dev_status=status)
        Y_plain = lib.elsa_nm_linear(Xd, vals, idx, None, out, in_, N, M, dev_status=status)
        torch.cuda.synchronize()
    finally:
        lib.elsa_set_linear_variant(lib.VARIANT_AUTO)
    assert int(status.item()) == 0, "device status %#x" % int(status.item())
    assert (guard[rows:] == 7.0).all()
    close(Y, ref)
    assert torch.equal(Y, Y_masked)                                               # the same tiles from either source
    close(Y_plain, ref - bias.double().numpy())


@pytest.mark.gpu
@pytest.mark.parametrize("level", [(1, 4), (2, 4), (3, 4), (4, 4), (2, 8), (3, 8), (4, 8), (4, 16), (8, 16)], ids=lambda l: "%dof%d" % l)
def test_few_rows_under_the_automatic_choice(lib, level):
    """The packed weight and the shared one, whichever kernel a wave of small tiles goes to at this level; 1:4 and 2:4 are one launch."""
    N, M = level
    for rows, in_, out in [(1, 128, 64), (49, 768, 2304), (197, 768, 768), (394, 1024, 200), (100, 3072, 768)]:
        X = synth.randn((rows, in_), rows + in_, synth.X_STD, torch.bfloat16).cuda()
        W = synth.randn((out, in_), out + in_, synth.W_STD, torch.bfloat16).cuda()
        bias = synth.randn((out,), out, synth.B_STD, torch.bfloat16).cuda()
        vals, idx = lib.elsa_nm_compress(W, N, M)
        Wm = W if N == M else lib.elsa_nm_unpack(vals, idx, out, in_, N, M)
        ref = (X.double() @ Wm.double().t() + bias.double()).cpu().numpy()
        before = lib.elsa_launch_count()
        Y = lib.elsa_nm_linear(X, vals, idx, bias, out, in_, N, M)
        launches = lib.elsa_launch_count() - before
        close(Y, ref)
        close(lib.elsa_nm_linear_masked(X, W, bias, N, M), ref)
        if (rows, in_, out) == (197, 768, 768):
            assert launches == (1 if M == 4 and N != 3 else 2)


@pytest.mark.gpu
def test_small_layers_of_a_table_share_a_launch(lib):
    """More layers than one launch carries, of every weight source, against the same table run layer by layer."""
    dtype = torch.bfloat16
    code = lib.dtype_code(dtype)
    shapes = [(49, 256, 768), (197, 64, 72), (100, 1024, 256), (1, 128, 8)]
    levels = [(1, 4), (2, 4), (1, 8), (4, 8), (8, 8), (2, 16), (4, 4)]
    dev = []
    for i in range(80):
        (rows, k, o), (N, M) = shapes[i % 4], levels[i % 7]
        layer = synth.Layer("l%d" % i, rows, k, o, N, M, 3 * i, 3 * i + 1, 3 * i + 2)
        X, W, b = synth.layer_tensors(layer, dtype, device="cuda")
        vals, idx = lib.elsa_nm_compress(W, N, M)
        dev.append(dict(X=X, W=W, vals=vals, idx=idx, bias=b, N=N, M=M, Y=torch.empty((rows, o), dtype=dtype, device="cuda")))
    table = lib.make_layer_table(dev)
    ws = lib.alloc_workspace(lib.elsa_vit_workspace_bytes(table, code))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    before = lib.elsa_launch_count()
    lib.elsa_vit_linears(table, code, ws, dev_status=status)
    assert lib.elsa_launch_count() - before == 3          # the weight images, then 72 layers and 8
    torch.cuda.synchronize()
    shared = [d["Y"].clone() for d in dev]
    lib.elsa_set_grouping(False)
    try:
        lib.elsa_vit_linears(table, code, ws, dev_status=status)
        torch.cuda.synchronize()
    finally:
        lib.elsa_set_grouping(True)
    assert int(status.item()) == 0
    for d, y in zip(dev, shared):
        assert torch.equal(d["Y"], y)
        out, in_ = d["W"].shape
        Wm = d["W"] if d["N"] == d["M"] else lib.elsa_nm_unpack(d["vals"], d["idx"], out, in_, d["N"], d["M"])
        close(y, (d["X"].double() @ Wm.double().t() + d["bias"].double()).cpu().numpy())


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [1, 15, 16, 17, 33, 64, 65, 127, 128, 130, 197])
@pytest.mark.parametrize("k,out", [(1024, 256), (1040, 200), (1024, 1544), (1024, 2376)])       # up to 128 rows cut into 8, 8, 4 and 2 ranges
def test_both_ways_of_the_sums_give_the_same(rows, k, out):
    """A call on a dense weight sends its sums as bulk copies, one behind an image as stores: the same operands, order and rounding."""
    from paper_2409_09708_b200 import binding as lib
    gen = torch.Generator().manual_seed(rows + k)
    X = torch.randn(rows, k, generator=gen).to(torch.bfloat16).cuda()
    W = (0.05 * torch.randn(out, k, generator=gen)).to(torch.bfloat16).cuda()
    bias = torch.randn(out, generator=gen).to(torch.bfloat16).cuda()
    vals, idx = lib.elsa_nm_compress(W, 3, 8)
    dense = lib.elsa_nm_unpack(vals, idx, out, k, 3, 8)
    guard = torch.full((rows + 130, out), 7.0, dtype=torch.bfloat16, device="cuda")
    lib.elsa_nm_linear(X, vals, idx, bias, out, k, 3, 8, Y=guard[:rows])
    assert torch.equal(guard[:rows], lib.elsa_nm_linear(X, dense, None, bias, out, k, 8, 8))
    assert bool((guard[rows:] == 7.0).all())
    exact = X.double() @ dense.double().t() + bias.double()
    # fp32 sums of k terms (error at most k 2^-24 of their absolute sum), one rounding to bf16
    bound = 2.0 ** -8 * exact.abs() + k * 2.0 ** -24 * (X.double().abs() @ dense.double().abs().t() + bias.double().abs())
    assert bool(((guard[:rows].double() - exact).abs() <= bound).all())

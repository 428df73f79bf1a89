"""The weight images behind the tensor-core kernels: with X = I the product is the masked weight itself, rounded once, so
a position or metadata mistake of any image shows exactly.  Rows below, at and past the 16- and 128-row units of the
2-of-4 form, fewer and more than a block's worth of units, every level with N <= 2 (and some above for the dense image),
from the packed weight and from the dense shared weight.
"""
import numpy as np
import pytest
import torch

from oracle import elsa_oracle as eo
from paper_2409_09708_b200 import synth

LEVELS = [(1, 4), (2, 4), (1, 8), (2, 8), (1, 16), (2, 16)]
CASES = [(8, 128), (136, 256), (40, 384), (1000, 640)]


@pytest.fixture(scope="module")
def lib():
    from paper_2409_09708_b200 import binding
    return binding


def masked(W, N, M):
    vals, idx, mask = eo.nm_compress(synth.bits(W), N, M)
    return W.double().numpy() * mask


@pytest.mark.gpu
@pytest.mark.parametrize("variant", ["tc_sparse", "tc_sparse_pair", "tc_sparse_ws", "tc_sparse_st", "tc_pair", "tc_dense"])
@pytest.mark.parametrize("level", LEVELS, ids=["%dof%d" % l for l in LEVELS])
def test_identity_product_is_the_masked_weight(lib, level, variant):
    N, M = level
    for out, in_ in CASES:
        W = synth.randn((out, in_), 3 * out + in_ + N, synth.W_STD, torch.float16)
        X = torch.eye(in_, dtype=torch.float16, device="cuda")
        Wd = W.cuda()
        vals, idx = lib.elsa_nm_compress(Wd, N, M)
        lib.elsa_set_linear_variant(getattr(lib, "VARIANT_" + variant.upper()))
        try:
            Y = lib.elsa_nm_linear(X, vals, idx, None, out, in_, N, M)
            Y_masked = Y if variant == "tc_sparse" else lib.elsa_nm_linear_masked(X, Wd, None, N, M)
            torch.cuda.synchronize()
        finally:
            lib.elsa_set_linear_variant(lib.VARIANT_AUTO)
        ref = masked(W, N, M).T
        assert np.array_equal(Y.double().cpu().numpy(), ref), (out, in_)
        assert np.array_equal(Y_masked.double().cpu().numpy(), ref), (out, in_)


@pytest.mark.gpu
@pytest.mark.parametrize("level", [(1, 4), (2, 4), (3, 4), (4, 4), (1, 8), (2, 8), (3, 8), (4, 8), (7, 8), (5, 16), (16, 16)],
                         ids=lambda l: "%dof%d" % l)
def test_unpack_around_a_block_of_units(lib, level):
    N, M = level
    for out, in_ in [(8, 16), (64, 128), (65 * 8, 16), (24, 16 * 23)]:          # 16 units, exactly 1024, one more row, ragged
        W = synth.randn((out, in_), out + in_ + N, synth.W_STD, torch.bfloat16)
        vals, idx = lib.elsa_nm_compress(W.cuda(), N, M)
        got = lib.elsa_nm_unpack(vals, idx, out, in_, N, M)
        assert np.array_equal(got.double().cpu().numpy(), masked(W, N, M)), (out, in_)


@pytest.mark.gpu
@pytest.mark.parametrize("M", [8, 16])
def test_every_level_packs_unpacks_and_masks_as_the_oracle(lib, M):
    """Ties and signs throughout, all N < M one call each: packed bytes, the rebuilt weight, and (X = I) the weight as projected from the
    shared one; one group a row and a block, ragged counts, and enough for a warp to take four segments."""
    rng = np.random.default_rng(M)
    for out, in_ in [(8, 16), (264, 16), (24, 16 * 23), (16, 4096 + 16), (2400, 1024)]:
        W = torch.from_numpy(rng.integers(-4, 5, (out, in_)).astype(np.float32)).to(torch.float16)
        Wd, Wb, X = W.cuda(), synth.bits(W), torch.eye(in_, dtype=torch.float16, device="cuda")
        for N in range(1, M):
            ovals, oidx, mask = eo.nm_compress(Wb, N, M)
            vals, idx = lib.elsa_nm_compress(Wd, N, M)
            assert (synth.bits(vals) == ovals).all() and (idx.cpu().numpy().view(np.uint32) == oidx).all(), (out, in_, N)
            want = torch.from_numpy(W.numpy() * mask)
            assert torch.equal(lib.elsa_nm_unpack(vals, idx, out, in_, N, M).cpu(), want), (out, in_, N)
            lib.elsa_set_linear_variant(lib.VARIANT_TC_PAIR)
            try:
                got = lib.elsa_nm_linear_masked(X, Wd, None, N, M).cpu()
            finally:
                lib.elsa_set_linear_variant(lib.VARIANT_AUTO)
            assert torch.equal(got, want.t()), (out, in_, N)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16], ids=["f16", "bf16"])
def test_ties_of_many_kinds_compress_as_the_oracle(lib, dtype):
    """Few distinct magnitudes, so most groups have ties around the threshold: every level, rows whose index bits do and do
    not fill whole words, one segment per warp and four."""
    rng = np.random.default_rng(11)
    for out, in_ in [(8, 48), (24, 16 * 23), (2400, 1024)]:
        W = torch.from_numpy(rng.integers(-3, 4, (out, in_)).astype(np.float32)).to(dtype)
        Wd, Wb = W.cuda(), synth.bits(W)
        for M in (4, 8, 16):
            levels = [n for n in (1, 2, 3, 4, 5, 8, 11) if n <= M]
            for N, (vals, idx) in zip(levels, lib.elsa_nm_compress_levels(Wd, levels, M)):
                ovals, oidx, _ = eo.nm_compress(Wb, N, M)
                assert (synth.bits(vals) == ovals).all(), (out, in_, N, M)
                if N < M:
                    assert (idx.cpu().numpy().view(np.uint32) == oidx).all(), (out, in_, N, M)


@pytest.mark.gpu
def test_an_image_of_more_units_than_32_bits_count():
    """2^32 units of eight positions and a few rows more (a 64 GB image, from 5 GB of packed values and words drawn at random: at 1:16
    every field is a position): rows from the start, the middle and the end."""
    from paper_2409_09708_b200 import binding as lib
    in_, out = 1 << 15, (1 << 20) + 8
    free, _ = torch.cuda.mem_get_info()
    if free < 90 << 30:
        pytest.skip("needs 90 GB of free device memory")
    vals = torch.randint(1, 1 << 14, (out, in_ // 16), dtype=torch.int16, device="cuda").view(torch.float16)
    idx = torch.randint(-(1 << 31), 1 << 31, (out, in_ // 128), dtype=torch.int64, device="cuda").to(torch.int32)
    Wm = torch.empty((out, in_), dtype=torch.float16, device="cuda")
    for r in (0, 1, out // 2 - 1, out // 2, out - 9, out - 8, out - 1):
        Wm[r].fill_(7.0)
    lib.elsa_nm_unpack(vals, idx, out, in_, 1, 16, W_masked=Wm)
    torch.cuda.synchronize()
    for r in (0, 1, out // 2 - 1, out // 2, out - 9, out - 8, out - 1):
        words = idx[r].cpu().numpy().view(np.uint32)
        pos = (words[:, None] >> (4 * np.arange(8, dtype=np.uint32))[None, :]).reshape(-1) & 15
        want = np.zeros((in_ // 16, 16), np.int16)
        want[np.arange(in_ // 16), pos] = vals[r].view(torch.int16).cpu().numpy()
        assert (Wm[r].view(torch.int16).cpu().numpy() == want.reshape(-1)).all(), r

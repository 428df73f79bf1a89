"""Window attention with a whole window per warp (heads of 32, at most 64 tokens) against the block oracle.

Sizes: one token, below / at / above a 16-row tile, 49 (7 x 7), the last size of the seven-tile form (56), the first and
the last of the eight-tile form (57, 64), and 65, the first that the tile kernel takes; more windows than an SM's warps
and more heads than SMs.  Tolerance as for every attention here: |err| <= u |ref| + (u / 2) max|v| + 1e-5 with u one unit
in the last place (probabilities are rounded to 16 bits for the second product, sum of p |v| <= max|v|).
"""
import numpy as np
import pytest
import torch

from oracle import elsa_block_oracle as bo
from paper_2409_09708_b200 import synth

CASES = [(3, 1, 2), (2, 15, 3), (2, 16, 1), (2, 17, 1), (40, 49, 5), (2, 56, 2), (2, 57, 2), (3, 64, 3), (2, 65, 2), (2, 9, 160),
         (2000, 4, 1)]


@pytest.fixture(scope="module")
def lib():
    from paper_2409_09708_b200 import binding
    return binding


def tolerance(ref, v, tokens, heads, dtype):
    u = 2.0 ** -7 if dtype == torch.bfloat16 else 2.0 ** -10
    rows, dim = v.shape
    shape = (rows // tokens, tokens, heads, dim // heads)
    vmax = np.broadcast_to(np.abs(v).reshape(shape).max(axis=(1, 3), keepdims=True), shape).reshape(rows, dim)
    return u * np.abs(ref) + 0.5 * u * vmax + 1e-5


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("tables", ["none", "bias", "bias+mask"])
@pytest.mark.parametrize("case", CASES, ids=["%dx%dx%d" % c for c in CASES])
def test_window_in_a_warp_matches_oracle(lib, case, tables, dtype):
    windows, T, heads = case
    dim = 32 * heads
    rng = np.random.default_rng(T)
    qkv = synth.randn((windows * T, 3 * dim), 41, 1.5, dtype)
    guard = torch.full((windows * T + 64, dim), 7.0, dtype=dtype, device="cuda")     # rows after the last window stay
    a = guard[:windows * T]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    extra = np.zeros((windows, heads, T, T))
    if tables == "none":
        lib.elsa_attention(qkv.cuda(), T, heads, a=a, dev_status=status)
    else:
        bias = rng.standard_normal((heads, T, T)).astype(np.float32)
        extra += bias
        mask = None
        if tables == "bias+mask":
            mask = np.where(rng.random((3, T, T)) < 0.3, -100.0, 0.0).astype(np.float32)
            mask[:, np.arange(T), np.arange(T)] = 0.0
            extra += mask[np.arange(windows) % 3][:, None]
            mask = lib.pad_score_table(torch.from_numpy(mask).cuda())
        lib.elsa_window_attention(qkv.cuda(), T, heads, lib.pad_score_table(torch.from_numpy(bias).cuda()), mask, a=a, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0, "device status %#x" % int(status.item())
    assert (guard[windows * T:] == 7.0).all()
    q64 = qkv.double().numpy()
    q, k, v = (q64[:, i * dim:(i + 1) * dim].reshape(windows, T, heads, 32).transpose(0, 2, 1, 3) for i in range(3))
    s = q @ k.transpose(0, 1, 3, 2) / np.sqrt(32) + extra
    e = np.exp(s - s.max(axis=-1, keepdims=True))
    ref = ((e / e.sum(axis=-1, keepdims=True)) @ v).transpose(0, 2, 1, 3).reshape(windows * T, dim)
    if tables == "none":
        assert np.allclose(ref, bo.attention(q64, T, heads), atol=1e-12)              # the oracle's loops, same formula
    got = a.double().cpu().numpy()
    assert np.isfinite(got).all()
    err, tol = np.abs(got - bo._round16(ref, dtype)), tolerance(ref, q64[:, 2 * dim:], T, heads, dtype)
    worst = (err - tol).argmax()
    assert (err <= tol).all(), "error %g at tolerance %g" % (err.flat[worst], tol.flat[worst])


@pytest.mark.gpu
@pytest.mark.parametrize("filler", [float("nan"), float("inf")], ids=["nan", "inf"])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("T", [1, 9, 15, 36, 47, 48, 49, 56, 57, 63, 65])
def test_what_lies_behind_the_tables_rows_takes_no_part(lib, T, dtype, filler):
    """A table's rows have bias_pitch floats; those from the window's last token on are the caller's to leave as they are."""
    windows, heads = 5, 2
    rng = np.random.default_rng(T)
    qkv = synth.randn((windows * T, 3 * 32 * heads), 43, 1.5, dtype, "cuda")
    bias = torch.from_numpy(rng.standard_normal((heads, T, T)).astype(np.float32))
    mask = torch.from_numpy(np.where(rng.random((3, T, T)) < 0.3, -100.0, 0.0).astype(np.float32))

    def padded(table, pitch, value):
        out = torch.full((table.shape[0], T, pitch), value)
        out[:, :, :T] = table
        return out.cuda()

    for pitch in ((T + 3) // 4 * 4, (T + 3) // 4 * 4 + 12):
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        got = [lib.elsa_window_attention(qkv, T, heads, padded(bias, pitch, v), padded(mask, pitch, v), dev_status=status)
               for v in (0.0, filler)]
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        assert torch.isfinite(got[0]).all() and torch.equal(got[0], got[1])

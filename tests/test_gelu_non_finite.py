"""GELU of values that are not finite, in every kernel that applies it: the fused epilogues (dense pair, few-rows, weight-stationary,
streaming) and the pass of its own behind the others.  v Phi(v) keeps NaN, is +inf at +inf and tends to 0 at -inf, where the
oracle's 0.5 v (1 + erf) is inf * 0; so NaN and +inf are compared with the oracle and -inf with the limit.  The values come in by
fc1's bias, in both halves of a pair of columns; the columns beside them stay what they are without."""
import numpy as np
import pytest
import torch

from oracle import elsa_block_oracle as bo
from paper_2409_09708_b200 import fit_gelu, synth

KINDS = ["TC_PAIR", "TC_SMALL", "TC_SPARSE_WS", "TC_SPARSE_ST", "TC_DENSE", "TC_SPARSE", "TC_SPARSE_PAIR", "SIMT", "AUTO"]
PLANTED = {0: float("nan"), 3: float("nan"), 8: float("inf"), 11: float("inf"), 16: float("-inf"), 31: float("-inf"), 255: float("nan")}


def test_the_restatement_keeps_them():
    co = fit_gelu.fit(rounds=1)
    v = np.array([np.nan, np.inf, -np.inf, 1.0, -1e30], np.float32)
    got = fit_gelu.gelu_f32(v, co)
    assert np.isnan(got[0]) and got[1] == np.inf and abs(got[2]) < 1e-6 and abs(got[4]) < 1e-6
    with np.errstate(invalid="ignore"):
        ref = bo.gelu(v[:2].astype(np.float64))
    assert np.isnan(ref[0]) and ref[1] == np.inf


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16], ids=["f16", "bf16"])
@pytest.mark.parametrize("kind", KINDS)
def test_every_kernel_kind(kind, dtype):
    from paper_2409_09708_b200 import binding as lib
    rows, dim, mlp = 300, 256, 512
    x = synth.randn((rows, dim), 5, 1.0, dtype, "cuda")
    ln = [(synth.randn((dim,), 30 + i, 0.1, dtype, "cuda") + (1.0 if i % 2 == 0 else 0.0)).to(dtype) for i in range(4)]
    packed = {}
    for i, (name, k, o) in enumerate((("qkv", dim, 3 * dim), ("proj", dim, dim), ("fc1", dim, mlp), ("fc2", mlp, dim))):
        W = synth.randn((o, k), 10 + i, 1.0 / np.sqrt(k), dtype, "cuda")
        packed[name] = lib.elsa_nm_compress(W, 2, 8) + (synth.randn((o,), 20 + i, 0.02, dtype, "cuda"), 2, 8)

    def h(bias):
        w, keep = lib.make_block_weights(*ln, dict(packed, fc1=packed["fc1"][:2] + (bias, 2, 8)))
        total, off = lib.elsa_vit_block_scratch_bytes(rows, dim, mlp, w, lib.dtype_code(dtype))
        scratch = torch.zeros(total, dtype=torch.uint8, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        lib.elsa_set_linear_variant(getattr(lib, "VARIANT_" + kind))
        try:
            lib.elsa_vit_block(x, mlp, w, scratch=scratch, dev_status=status)
            torch.cuda.synchronize()
        finally:
            lib.elsa_set_linear_variant(lib.VARIANT_AUTO)
        assert int(status.item()) == 0, "device status %#x" % int(status.item())
        return lib.block_region(scratch, off, "h", rows, mlp, dtype).clone()

    bias = packed["fc1"][2]
    planted = bias.clone()
    for c, v in PLANTED.items():
        planted[c] = v
    plain, got = h(bias), h(planted)
    assert torch.isfinite(plain).all()
    for c, v in PLANTED.items():
        if np.isnan(v):
            assert torch.isnan(got[:, c]).all(), (kind, c)
        elif v > 0:
            assert (got[:, c] == v).all(), (kind, c)
        else:
            assert (got[:, c].float().abs() <= 1e-6).all(), (kind, c)
    others = [c for c in range(mlp) if c not in PLANTED]
    assert torch.equal(got[:, others], plain[:, others])

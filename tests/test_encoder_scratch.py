"""What scratch the encoder takes: with elsa_vit_encoder_scratch_bytes it builds every block's weight images ahead of the chain, with
less, down to the largest block's scratch and two activation buffers, each block's before the block; the results are the same bits."""
import numpy as np
import pytest
import torch

from paper_2409_09708_b200 import synth


@pytest.mark.gpu
@pytest.mark.parametrize("images", [1, 9, 70])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
def test_scratch_between_the_least_and_the_most(images, dtype):
    from paper_2409_09708_b200 import binding as lib
    dim, tokens, heads, n = 256, 65, 4, 5
    mlp, rows, code = 4 * dim, images * tokens, lib.dtype_code(dtype)
    levels = [(2, 4), (1, 8), (4, 8), (4, 4), (2, 8), (3, 8)]
    blocks, keep, largest = [], [], 0
    for b in range(n):
        lin = {}
        for i, (name, k, o) in enumerate((("qkv", dim, 3 * dim), ("proj", dim, dim), ("fc1", dim, mlp), ("fc2", mlp, dim))):
            N, M = levels[(b + i) % 6]
            W = synth.randn((o, k), 10 * b + i, 1.0 / np.sqrt(k), dtype, "cuda")
            lin[name] = lib.elsa_nm_compress(W, N, M) + (synth.randn((o,), 7 + i, 0.02, dtype, "cuda"), N, M)
        ln = [(synth.randn((dim,), 50 + i, 0.1, dtype, "cuda") + (1.0 if i % 2 == 0 else 0.0)).to(dtype) for i in range(4)]
        w, k = lib.make_block_weights(*ln, lin)
        blocks.append(w)
        keep.append(k)
        largest = max(largest, lib.elsa_vit_block_scratch_bytes(rows, dim, mlp, w, code)[0])
    up = lambda v: (v + 255) // 256 * 256
    least = up(largest) + 2 * up(rows * dim * 2)
    table = lib.make_encoder_table(blocks)
    x = synth.randn((rows, dim), 3, 1.0, dtype, "cuda")
    gain, beta = synth.randn((dim,), 91, 0.1, dtype, "cuda") + 1.0, synth.randn((dim,), 92, 0.1, dtype, "cuda")

    def run(nbytes):
        guarded = torch.full((nbytes + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        y, _ = lib.elsa_vit_encoder(x, tokens, heads, mlp, table, gain, beta, scratch=guarded[:nbytes], dev_status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        assert (guarded[nbytes:] == 0x5A).all()
        return y

    most = int(lib._encoder_scratch(images, tokens, dim, mlp, table, n, code))
    assert most >= least
    want = run(most)
    assert torch.equal(run(least), want)
    assert torch.equal(run((least + most) // 2), want)
    with pytest.raises(lib.ElsaError) as e:
        run(least - 256)
    assert e.value.status == 6                                       # ELSA_ERR_WORKSPACE

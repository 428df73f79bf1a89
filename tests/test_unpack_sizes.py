"""The dense image with one unit per thread (few blocks) and with several (many), on either side of the size where the launch
changes from one to the other and at remainders of a block, for levels compiled in and not, groups of 16 with odd and even N."""
import numpy as np
import pytest
import torch

from oracle import elsa_oracle as eo
from paper_2409_09708_b200 import synth

LEVELS = [(1, 4), (3, 4), (2, 8), (4, 8), (5, 8), (1, 16), (7, 16), (8, 16), (15, 16)]
CASES = [(8, 16), (24, 176), (512, 2048), (2360, 1024), (2376, 1024), (1032, 2608)]


@pytest.mark.gpu
@pytest.mark.parametrize("level", LEVELS, ids=["%dof%d" % l for l in LEVELS])
def test_unpack_is_the_masked_weight(level):
    from paper_2409_09708_b200 import binding as lib
    N, M = level
    for out, in_ in CASES:
        W = synth.randn((out, in_), out + in_ + N, synth.W_STD, torch.bfloat16)
        vals, idx = lib.elsa_nm_compress(W.cuda(), N, M)
        got = lib.elsa_nm_unpack(vals, idx, out, in_, N, M)
        torch.cuda.synchronize()
        ref = np.where(eo.nm_mask(synth.bits(W), N, M) != 0, synth.bits(W), 0)
        assert np.array_equal(synth.bits(got.cpu()), ref), (out, in_)

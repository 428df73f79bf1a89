"""Tables of layers with few rows on either side of where they move from the few-rows kernel to the pair kernel: few layers and
many, rows below and above a wave of small tiles, with one scratch region per layer (shared launches) and with the largest layer's
only (one after the other), which must give the same bits.  Small integers: the products are exact."""
import numpy as np
import pytest
import torch

from oracle import elsa_oracle as eo
from paper_2409_09708_b200 import synth

CASES = [(2, 100, 128, 192), (12, 197, 192, 200), (60, 197, 64, 264), (5, 3000, 128, 136), (30, 130, 320, 72)]


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES, ids=["%dx%dx%dx%d" % c for c in CASES])
def test_small_layers_of_a_table(case):
    from paper_2409_09708_b200 import binding as lib
    n, rows, in_, out = case
    rng = np.random.default_rng(n)
    ints = lambda *s: torch.from_numpy(rng.integers(-3, 4, s).astype(np.float32)).half()
    layers, refs = [], []
    for l in range(n):
        N, M = ((2, 4), (4, 8), (8, 8), (1, 4))[l % 4]
        X, W, b = ints(rows, in_), ints(out, in_), ints(out)
        vals, idx = lib.elsa_nm_compress(W.cuda(), N, M)
        layers.append(dict(X=X.cuda(), Y=torch.full((rows, out), 7.0, dtype=torch.float16, device="cuda"), vals=vals, idx=idx, bias=b.cuda(), N=N, M=M))
        Wm = W.double() * torch.from_numpy(eo.nm_mask(synth.bits(W), N, M).astype(np.float64))
        refs.append((X.cuda().double() @ Wm.cuda().t() + b.cuda().double()).half())
    table = lib.make_layer_table(layers)
    code = lib.F16
    largest = max(lib.elsa_workspace_bytes(rows, in_, out, l["N"], l["M"], code) for l in layers)
    for bytes_ in (lib.elsa_vit_workspace_bytes(table, code), largest):
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        for l in layers:
            l["Y"].fill_(7.0)
        lib.elsa_vit_linears(table, code, lib.alloc_workspace(bytes_), dev_status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0, "device status %#x" % int(status.item())
        for l, ref in zip(layers, refs):
            assert torch.equal(l["Y"], ref)

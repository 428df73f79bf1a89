"""Calls that build weight images on a side stream, made from several threads on streams of their own at once: every result
equals the one of the same call made alone (a call whose images were ordered after another call's work would not)."""
import threading

import pytest
import torch

from paper_2409_09708_b200 import synth


@pytest.mark.gpu
def test_encoders_and_tables_of_several_threads_do_not_disturb_each_other():
    from paper_2409_09708_b200 import binding as lib
    dtype, dim, tokens, heads = torch.bfloat16, 256, 65, 4
    code = lib.dtype_code(dtype)
    levels = [(2, 4), (1, 8), (4, 8), (4, 4), (2, 8)]

    def case(seed):
        blocks, keep = [], []
        for b in range(4):
            lin = {}
            for i, (name, k, o) in enumerate((("qkv", dim, 3 * dim), ("proj", dim, dim), ("fc1", dim, 4 * dim), ("fc2", 4 * dim, dim))):
                N, M = levels[(seed + b + i) % 5]
                W = synth.randn((o, k), 100 * seed + 10 * b + i, 0.05, dtype, "cuda")
                lin[name] = lib.elsa_nm_compress(W, N, M) + (synth.randn((o,), 7 + i, 0.02, dtype, "cuda"), N, M)
            ln = [synth.randn((dim,), 50 + i, 0.1, dtype, "cuda") + (1.0 if i % 2 == 0 else 0.0) for i in range(4)]
            w, k = lib.make_block_weights(*[t.to(dtype) for t in ln], lin)
            blocks.append(w)
            keep.append(k)
        images = 3 + 20 * (seed % 3)                                 # one wave of small tiles, and more
        x = synth.randn((images * tokens, dim), seed, 1.0, dtype, "cuda")
        layers = []
        for i, (N, M) in enumerate([(4, 4), (2, 4), (1, 8), (4, 8)]):
            layer = synth.Layer("l", 9000, 512, 512, N, M, 3 * i + seed, 3 * i + 1, 3 * i + 2)
            X, W, bias = synth.layer_tensors(layer, dtype, device="cuda")
            vals, idx = lib.elsa_nm_compress(W, N, M)
            layers.append(dict(X=X, vals=vals, idx=idx, bias=bias, N=N, M=M, Y=torch.empty((9000, 512), dtype=dtype, device="cuda")))
        table = lib.make_layer_table(layers)
        ws = lib.alloc_workspace(lib.elsa_vit_workspace_bytes(table, code))
        return dict(x=x, table=lib.make_encoder_table(blocks), keep=(keep, layers), layers=table, Y=[l["Y"] for l in layers], ws=ws)

    def run(c):
        y, c["scratch"] = lib.elsa_vit_encoder(c["x"], tokens, heads, 4 * dim, c["table"], scratch=c.get("scratch"))
        for t in c["Y"]:
            t.zero_()
        lib.elsa_vit_linears(c["layers"], code, c["ws"])
        return [y.clone()] + [t.clone() for t in c["Y"]]

    cases = [case(s) for s in range(4)]
    alone = [run(c) for c in cases]
    torch.cuda.synchronize()
    wrong, errors = [], []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(10):
                    got = run(cases[i])
                    torch.cuda.current_stream().synchronize()
                    if not all(torch.equal(a, b) for a, b in zip(got, alone[i])):
                        wrong.append(i)
        except Exception as e:                                       # a failed call fails the test, not the thread alone
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
    assert not wrong, wrong


@pytest.mark.gpu
def test_a_capture_in_progress_keeps_its_side_stream_to_itself():
    """A table's images fork to a side stream, which stays part of a capture until the capture ends.  Calls made meanwhile on other
    streams, captured into another graph or not, succeed, the captures stay valid, and everything computes the same."""
    from paper_2409_09708_b200 import binding as lib
    dtype = torch.bfloat16
    code = lib.dtype_code(dtype)

    def table(seed):
        layers = []
        for i, (N, M) in enumerate([(4, 4), (2, 4), (1, 8), (4, 8)]):
            X, W, bias = synth.layer_tensors(synth.Layer("l", 9000, 512, 512, N, M, 3 * i + seed, 3 * i + 1, 3 * i + 2), dtype, device="cuda")
            vals, idx = lib.elsa_nm_compress(W, N, M)
            layers.append(dict(X=X, vals=vals, idx=idx, bias=bias, N=N, M=M, Y=torch.empty((9000, 512), dtype=dtype, device="cuda")))
        lt = lib.make_layer_table(layers)
        return dict(lt=lt, Y=[l["Y"] for l in layers], ws=lib.alloc_workspace(lib.elsa_vit_workspace_bytes(lt, code)), keep=layers)

    def run(t):
        lib.elsa_vit_linears(t["lt"], code, t["ws"])

    tables = [table(s) for s in (0, 100, 200)]
    for t in tables:
        run(t)
    torch.cuda.synchronize()
    want = [[y.clone() for y in t["Y"]] for t in tables]
    for t in tables:
        for y in t["Y"]:
            y.zero_()
    torch.cuda.synchronize()

    first, second, plain = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Stream()
    g1, g2 = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    errors = []

    def meanwhile():
        """What another thread does while the first capture is open: an ordinary call, then a capture of its own."""
        try:
            with torch.cuda.stream(plain):
                run(tables[2])
            with torch.cuda.stream(second):
                g2.capture_begin(capture_error_mode="thread_local")
                run(tables[1])
                run(tables[1])
                g2.capture_end()
        except Exception as e:
            errors.append(e)

    with torch.cuda.stream(first):
        g1.capture_begin(capture_error_mode="thread_local")
        run(tables[0])
        other = threading.Thread(target=meanwhile)
        other.start()
        other.join()
        run(tables[0])                                               # the capture's own pipe again
        g1.capture_end()
    assert not errors, errors[0]
    g1.replay()
    g2.replay()
    run(tables[2])                                                   # pipes of ended captures serve ordinary calls
    torch.cuda.synchronize()
    for t, ys in zip(tables, want):
        for y, w in zip(t["Y"], ys):
            assert torch.equal(y, w)

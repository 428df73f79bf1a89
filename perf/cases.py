"""The workloads whose speed this library is judged by.

Each case is one call, or one short sequence of calls, that a program built on
the library makes: a linear layer at inference, all linear layers of a model
under a level table, the chained encoder at one image and at a full batch, the
Swin blocks, the supernet's forward, a training step, the INT8 form, and the
compression of a shared weight to all its levels.  Shapes and level tables are
those of ``paper_2409_09708_b200/synth.py`` and of the benches at the
repository root; ``draw`` spreads sizes, types and levels over the same ranges.

A case is a dict of plain values.  ``kind`` names the path:

  linear    elsa_nm_linear on one layer with its packed weight at hand
  table     elsa_vit_compress + elsa_vit_linears over a table of layers
  encoder   elsa_vit_encoder, packed weights at hand
  swin      elsa_swin_block, block after block inside each stage
  supernet  elsa_nm_linear_masked over the four linears of a block
  train     per linear of a block: elsa_nm_compress, elsa_nm_linear, elsa_nm_linear_backward
  int8      elsa_nm_linear_i8 over the four linears of a block
  levels    elsa_nm_compress_levels of one weight
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2409_09708_b200 import synth

TOKENS = 197                 # a 224 x 224 image in 16 x 16 patches and the class token
WINDOW = 7
DTYPES = {"f16": torch.float16, "bf16": torch.bfloat16}
N4_LEVELS = "1:4 2:4 4:4"
N8_LEVELS = "1:8 2:8 4:8 8:8"
SWIN_LEVELS = "1:4 2:4 1:8 2:8 4:8"
BLOCK_LEVELS = "4:8 2:8 2:8 1:8"
ALL_LEVELS = ((1, 4), (2, 4), (1, 8), (2, 8), (4, 8), (8, 8), (1, 16), (2, 16), (4, 16), (8, 16))


def listed():
    return [
        # One linear of one image: the smallest call, where launches and host work are what is paid for.
        {"name": "linear_one_image", "kind": "linear", "rows": 197, "in": 768, "out": 768, "N": 4, "M": 8, "dtype": "f16"},
        # An ordinary inference layer at a batch that fills no tile evenly (25 images), at a level of the N:4 space.
        {"name": "linear_fc1_25_images", "kind": "linear", "rows": 4925, "in": 768, "out": 3072, "N": 2, "M": 4, "dtype": "bf16"},
        # The four linears of a DeiT-B block at batch 64, weights pruned anew (a configuration just sampled).
        {"name": "table_deit_b_block_b64", "kind": "table", "model": "deit", "dim": 768, "blocks": 1, "batch": 64,
         "levels": BLOCK_LEVELS, "levels_seed": -1, "dtype": "f16"},
        # The headline workload: all 48 linears of DeiT-B at batch 256 under a mixed level table.
        {"name": "table_deit_b_b256", "kind": "table", "model": "deit", "dim": 768, "blocks": 12, "batch": 256,
         "levels": N8_LEVELS, "levels_seed": 3, "dtype": "bf16"},
        # The same of Swin-B at batch 128: 96 linears of four widths, many of them small.
        {"name": "table_swin_b_b128", "kind": "table", "model": "swin", "dim": 128, "blocks": 24, "batch": 128,
         "levels": SWIN_LEVELS, "levels_seed": 4, "dtype": "bf16"},
        # Serving one image: the whole encoder under an N:4 configuration, bound by latency and launches.
        {"name": "encoder_deit_b_one_image", "kind": "encoder", "dim": 768, "blocks": 12, "batch": 1, "tokens": TOKENS,
         "levels": N4_LEVELS, "levels_seed": 7, "dtype": "bf16"},
        # Evaluating at full batch.
        {"name": "encoder_deit_b_b256", "kind": "encoder", "dim": 768, "blocks": 12, "batch": 256, "tokens": TOKENS,
         "levels": N8_LEVELS, "levels_seed": 3, "dtype": "bf16"},
        # The 24 blocks of Swin-B at full batch: shifted windows of 49 tokens, narrow rows in the first stages.
        {"name": "swin_b_blocks_b128", "kind": "swin", "dim": 128, "depths": "2 2 18 2", "batch": 128,
         "levels": SWIN_LEVELS, "levels_seed": 4, "dtype": "bf16"},
        # Supernet evaluation: levels applied to the shared dense weights while they are used.
        {"name": "supernet_block_b64", "kind": "supernet", "dim": 768, "batch": 64, "levels": BLOCK_LEVELS,
         "levels_seed": -1, "dtype": "bf16"},
        # Supernet training: weights change every step, so prune, forward and backward of a block's linears.
        {"name": "train_block_b128", "kind": "train", "dim": 768, "batch": 128, "levels": N8_LEVELS, "levels_seed": 5,
         "dtype": "bf16"},
        # The quantised form of a block's linears.
        {"name": "int8_block_b64", "kind": "int8", "dim": 768, "batch": 64, "levels": BLOCK_LEVELS, "levels_seed": -1,
         "dtype": "bf16"},
        # A shared weight (fc1 of DeiT-B) to every level of its search space.
        {"name": "levels_fc1", "kind": "levels", "in": 768, "out": 3072, "M": 8, "levels": "1 2 4 8", "dtype": "bf16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("linear", "linear", "table", "table", "encoder", "encoder", "swin", "supernet", "train", "int8", "levels"))
    dtype = rng.choice(("f16", "bf16"))
    seed = rng.randrange(1000)
    dim = 64 * rng.choice((3, 4, 6, 8, 12, 16))
    # rows x dim^2 stays at or below that of a DeiT-B block at batch 256
    def batch(most, smallest=1):
        return max(smallest, min(_log(rng, smallest, most), int(most * (768.0 / max(dim, 768)) ** 2)))

    if kind == "linear":
        k, o = rng.choice(((dim, 3 * dim), (dim, dim), (dim, 4 * dim), (4 * dim, dim)))
        n, m = rng.choice(ALL_LEVELS)
        return {"kind": kind, "rows": _log(rng, 49, 50432), "in": k, "out": o, "N": n, "M": m, "dtype": dtype}
    if kind == "table":
        if rng.random() < 0.5:
            return {"kind": kind, "model": "swin", "dim": rng.choice((96, 128)), "blocks": 24, "batch": _log(rng, 1, 100),
                    "levels": rng.choice((SWIN_LEVELS, N4_LEVELS)), "levels_seed": seed, "dtype": dtype}
        return {"kind": kind, "model": "deit", "dim": dim, "blocks": rng.choice((1, 2, 4, 6, 12)), "batch": batch(240),
                "levels": rng.choice((N8_LEVELS, N4_LEVELS)), "levels_seed": seed, "dtype": dtype}
    if kind == "encoder":
        return {"kind": kind, "dim": dim, "blocks": 12, "batch": batch(220), "tokens": rng.choice((TOKENS, TOKENS, 196, 145, 65)),
                "levels": rng.choice((N8_LEVELS, N4_LEVELS)), "levels_seed": seed, "dtype": dtype}
    if kind == "swin":
        return {"kind": kind, "dim": rng.choice((96, 128)), "depths": rng.choice(("2 2 6 2", "2 2 18 2")), "batch": _log(rng, 1, 100),
                "levels": rng.choice((SWIN_LEVELS, N4_LEVELS)), "levels_seed": seed, "dtype": dtype}
    if kind == "levels":
        k, o = rng.choice(((dim, 3 * dim), (dim, dim), (dim, 4 * dim), (4 * dim, dim)))
        m, lv = rng.choice(((4, "1 2 4"), (8, "1 2 4 8"), (8, "1 2 3 4"), (16, "1 2 4 8")))
        return {"kind": kind, "in": k, "out": o, "M": m, "levels": lv, "dtype": dtype}
    return {"kind": kind, "dim": dim, "batch": batch(200), "levels": rng.choice((N8_LEVELS, N4_LEVELS)), "levels_seed": seed,
            "dtype": dtype}


# ---------------------------------------------------------------------------------------------- shapes and levels

def _block_shapes(dim):
    return (("qkv", dim, 3 * dim), ("proj", dim, dim), ("fc1", dim, 4 * dim), ("fc2", 4 * dim, dim))


def _levels(case, count):
    """One (N, M) per linear: the listed levels in turn, or a seeded uniform choice among them."""
    choices = [tuple(int(v) for v in s.split(":")) for s in case["levels"].split()]
    if case["levels_seed"] < 0:
        return [choices[i % len(choices)] for i in range(count)]
    at = np.random.default_rng(case["levels_seed"]).integers(0, len(choices), count)
    return [choices[int(i)] for i in at]


def _stages(case):
    """Swin's stages: (dim, depth, grid side, heads)."""
    depths = [int(v) for v in case.get("depths", "2 2 18 2").split()]
    return [(case["dim"] << s, depths[s], 56 >> s, (case["dim"] << s) // 32) for s in range(4)]


def _layers(case):
    """(group, index in group, rows, in, out, N, M) of every linear of the case, in order; the linears of a group have
    one shape, so that their outputs can be one tensor."""
    kind = case["kind"]
    if kind == "linear":
        return [("y", 0, case["rows"], case["in"], case["out"], case["N"], case["M"])]
    if kind in ("supernet", "train", "int8"):
        plan = [(1, case["dim"], case["batch"] * TOKENS, "")]
    elif kind == "swin" or case.get("model") == "swin":
        plan = [(depth, dim, case["batch"] * g * g, "stage%d." % s) for s, (dim, depth, g, _) in enumerate(_stages(case))]
    else:
        plan = [(case["blocks"], case["dim"], case["batch"] * case.get("tokens", TOKENS), "")]
    shapes = [(prefix + name, b, rows, k, o) for depth, dim, rows, prefix in plan for b in range(depth)
              for name, k, o in _block_shapes(dim)]
    return [s + lv for s, lv in zip(shapes, _levels(case, len(shapes)))]


# ---------------------------------------------------------------------------------------------- inputs

class _Source:
    """Seeded tensors on the GPU: activations N(0, 1), weights and biases N(0, 0.02), as synth.py describes them."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def normal(self, shape, std, dtype, mean=0.0):
        return torch.empty(shape, dtype=torch.float32, device="cuda").normal_(mean, std, generator=self.gen).to(dtype)

    def int8(self, shape):
        return torch.randint(-128, 128, shape, dtype=torch.int8, device="cuda", generator=self.gen)


def _packed(lib, src, k, o, n, m, dtype):
    """(vals, idx, bias, N, M) of a linear, as a model loaded for inference holds them."""
    vals, idx = lib.elsa_nm_compress(src.normal((o, k), synth.W_STD, dtype), n, m)
    return vals, idx, src.normal((o,), synth.B_STD, dtype), n, m


def _block_weights(lib, src, dim, layers, dtype):
    linears = {name: _packed(lib, src, k, o, n, m, dtype)
               for (name, _, _), (_, _, _, k, o, n, m) in zip(_block_shapes(dim), layers)}
    ln = [src.normal((dim,), 0.1, dtype, mean=1.0 if i % 2 == 0 else 0.0) for i in range(4)]
    return lib.make_block_weights(*ln, linears, eps=1e-6)


def prepare(case, seed):
    from paper_2409_09708_b200 import binding as lib
    src = _Source(seed)
    kind, dtype = case["kind"], DTYPES[case["dtype"]]
    code = lib.dtype_code(dtype)
    layers = [] if kind == "levels" else _layers(case)
    state = {"lib": lib, "kind": kind, "code": code}

    if kind == "levels":
        state.update(W=src.normal((case["out"], case["in"]), synth.W_STD, dtype), M=case["M"],
                     levels=[int(v) for v in case["levels"].split()])
    elif kind == "linear":
        _, _, rows, k, o, n, m = layers[0]
        vals, idx, bias, _, _ = _packed(lib, src, k, o, n, m, dtype)
        state.update(args=(src.normal((rows, k), synth.X_STD, dtype), vals, idx, bias, o, k, n, m),
                     workspace=lib.alloc_workspace(lib.elsa_workspace_bytes(rows, k, o, n, m, code)))
    elif kind == "table":
        depth = {}
        for g, b, *_ in layers:
            depth[g] = b + 1
        # every layer's packed form lies in one arena, 256 bytes apart, as a checkpoint's weights do
        up = lambda v: (v + 255) // 256 * 256
        vbytes = [up(lib.elsa_nm_values_bytes(o, k, n, m, code)) for _, _, _, k, o, n, m in layers]
        ibytes = [up(lib.elsa_nm_index_bytes(o, k, n, m)) for _, _, _, k, o, n, m in layers]
        vals = torch.zeros(sum(vbytes) // 2, dtype=dtype, device="cuda")
        idx = torch.zeros(max(1, sum(ibytes) // 4), dtype=torch.int32, device="cuda")
        X, Y, table, vat, iat = {}, {}, [], 0, 0
        for (g, b, rows, k, o, n, m), vb, ib in zip(layers, vbytes, ibytes):
            if g not in Y:
                X[g] = torch.empty((depth[g], rows, k), dtype=dtype, device="cuda")
                Y[g] = torch.empty((depth[g], rows, o), dtype=dtype, device="cuda")
            X[g][b].normal_(0.0, synth.X_STD, generator=src.gen)
            table.append(dict(X=X[g][b], Y=Y[g][b], W=src.normal((o, k), synth.W_STD, dtype),
                              bias=src.normal((o,), synth.B_STD, dtype), N=n, M=m,
                              vals=vals[vat:vat + o * (k // m) * n].view(o, -1),
                              idx=idx[iat:iat + lib.elsa_nm_index_bytes(o, k, n, m) // 4] if ib else None))
            vat, iat = vat + vb // 2, iat + ib // 4
        lt = lib.make_layer_table(table)
        state.update(weights=lib.make_weight_table(table), layers=lt, keep=table, outputs={"vals": vals, "idx": idx, **Y},
                     workspace=lib.alloc_workspace(lib.elsa_vit_workspace_bytes(lt, code)))
    elif kind == "encoder":
        dim, tokens = case["dim"], case["tokens"]
        blocks = [_block_weights(lib, src, dim, layers[4 * b:4 * b + 4], dtype) for b in range(case["blocks"])]
        x = src.normal((case["batch"] * tokens, dim), synth.X_STD, dtype)
        table = lib.make_encoder_table([w for w, _ in blocks])
        gain, beta = src.normal((dim,), 0.1, dtype, mean=1.0), src.normal((dim,), 0.1, dtype)
        y, scratch = lib.elsa_vit_encoder(x, tokens, dim // 64, 4 * dim, table, gain, beta)     # sizes the scratch
        state.update(x=x, tokens=tokens, heads=dim // 64, mlp=4 * dim, table=table, final=(gain, beta), y=y, scratch=scratch,
                     keep=blocks)
    elif kind == "swin":
        stages, at = [], 0
        T = WINDOW * WINDOW
        for dim, depth, g, heads in _stages(case):
            rows, blocks, need = case["batch"] * g * g, [], 0
            for b in range(depth):
                w, keep = _block_weights(lib, src, dim, layers[at:at + 4], dtype)
                at += 4
                shift = WINDOW // 2 if b % 2 == 1 and g > WINDOW else 0
                rel = lib.pad_score_table(src.normal((heads, T, T), 0.5, torch.float32))
                mask = lib.elsa_swin_mask(g, g, WINDOW, shift).cuda() if shift else None
                blocks.append((w, shift, rel, mask, keep))
                need = max(need, lib.elsa_vit_block_scratch_bytes(rows, dim, 4 * dim, w, code)[0])
            x = src.normal((rows, dim), synth.X_STD, dtype)
            stages.append(dict(grid=g, heads=heads, mlp=4 * dim, blocks=blocks, scratch=lib.alloc_workspace(need), x=x,
                               buffers=[torch.empty_like(x), torch.empty_like(x)]))
        state.update(stages=stages)
    elif kind == "supernet":
        state.update(linears=[(src.normal((rows, k), synth.X_STD, dtype), src.normal((o, k), synth.W_STD, dtype),
                               src.normal((o,), synth.B_STD, dtype), n, m,
                               lib.alloc_workspace(lib.elsa_workspace_bytes(rows, k, o, n, m, code)))
                              for _, _, rows, k, o, n, m in layers])
    elif kind == "train":
        state.update(linears=[(src.normal((rows, k), synth.X_STD, dtype), src.normal((o, k), synth.W_STD, dtype),
                               src.normal((o,), synth.B_STD, dtype), src.normal((rows, o), 0.05, dtype), n, m,
                               lib.alloc_workspace(lib.elsa_workspace_bytes(rows, k, o, n, m, code)),
                               lib.alloc_workspace(lib.elsa_backward_workspace_bytes(rows, k, o, n, m, code)))
                              for _, _, rows, k, o, n, m in layers])
    elif kind == "int8":
        linears = []
        for _, _, rows, k, o, n, m in layers:
            vals, idx = lib.elsa_nm_compress_i8(src.int8((o, k)), n, m)
            scale = torch.rand(o, device="cuda", generator=src.gen) * 1e-3 + 1e-4
            linears.append((src.int8((rows, k)), 0.02, vals, idx, scale, src.normal((o,), synth.B_STD, dtype), o, k, n, m, dtype))
        state.update(linears=linears)
    return state


# ---------------------------------------------------------------------------------------------- one pass

def run(state):
    lib, kind = state["lib"], state["kind"]
    if kind == "linear":
        return lib.elsa_nm_linear(*state["args"], workspace=state["workspace"])
    if kind == "table":
        lib.elsa_vit_compress(state["weights"], state["code"])
        lib.elsa_vit_linears(state["layers"], state["code"], state["workspace"])
        return state["outputs"]
    if kind == "encoder":
        y, _ = lib.elsa_vit_encoder(state["x"], state["tokens"], state["heads"], state["mlp"], state["table"], *state["final"],
                                    y=state["y"], scratch=state["scratch"])
        return y
    if kind == "swin":
        outputs = []
        for s in state["stages"]:
            x = s["x"]
            for b, (w, shift, rel, mask, _) in enumerate(s["blocks"]):
                x, _ = lib.elsa_swin_block(x, s["grid"], s["grid"], WINDOW, shift, s["heads"], s["mlp"], w, rel, mask,
                                           y=s["buffers"][b & 1], scratch=s["scratch"])
            outputs.append(x)
        return outputs
    if kind == "supernet":
        return [lib.elsa_nm_linear_masked(X, W, bias, n, m, workspace=ws) for X, W, bias, n, m, ws in state["linears"]]
    if kind == "train":
        outputs = []
        for X, W, bias, dY, n, m, ws, bws in state["linears"]:
            o, k = W.shape
            vals, idx = lib.elsa_nm_compress(W, n, m)
            Y = lib.elsa_nm_linear(X, vals, idx, bias, o, k, n, m, workspace=ws)
            outputs.append((Y,) + lib.elsa_nm_linear_backward(dY, X, vals, idx, o, k, n, m, workspace=bws))
        return outputs
    if kind == "int8":
        return [lib.elsa_nm_linear_i8(*args) for args in state["linears"]]
    return lib.elsa_nm_compress_levels(state["W"], state["levels"], state["M"])


# ---------------------------------------------------------------------------------------------- work and tolerance

def _index_bytes(k, o, n, m):
    bits = {4: 2, 8: 3, 16: 4}[m]
    return 0 if n == m else o * -(-(k // m * n * bits) // 32) * 4


def work(case):
    kind = case["kind"]
    if kind == "levels":
        k, o, m = case["in"], case["out"], case["M"]
        packed = sum(o * (k // m) * int(n) * 2 + _index_bytes(k, o, int(n), m) for n in case["levels"].split())
        return {"bytes": 2 * o * k + packed, "flops": 0}
    nbytes = flops = 0.0
    for _, _, rows, k, o, n, m in _layers(case):
        packed = o * (k // m) * n * (1 if kind == "int8" else 2) + _index_bytes(k, o, n, m) + 2 * o
        kept = 2.0 * rows * k * o * n / m
        flops += kept
        if kind in ("encoder", "swin"):        # only the chain's ends cross memory of necessity
            nbytes += packed
        elif kind == "table":                  # dense weight in, packed form out, then the layer
            nbytes += 2 * rows * (k + o) + 2 * o * k + packed
        elif kind == "supernet":
            nbytes += 2 * rows * (k + o) + 2 * o * k + 2 * o
        elif kind == "train":                  # X, W, dY in; Y, dX, dW, db out; three products over the kept weights
            nbytes += 2 * rows * (2 * k + 2 * o) + 2 * o * k + 2 * o * k + 4 * o
            flops += 2 * kept
        elif kind == "int8":
            nbytes += rows * (k + 2 * o) + packed + 4 * o
        else:
            nbytes += 2 * rows * (k + o) + packed
    if kind == "encoder":
        rows, dim, t = case["batch"] * case["tokens"], case["dim"], case["tokens"]
        nbytes += 2 * 2 * rows * dim
        flops += case["blocks"] * 4.0 * rows * t * dim
    elif kind == "swin":
        for dim, depth, g, _ in _stages(case):
            rows = case["batch"] * g * g
            nbytes += 2 * 2 * rows * dim
            flops += depth * 4.0 * rows * WINDOW * WINDOW * dim
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Packed forms are bytes.  INT8 products are exact in int32 and the epilogue's fp32 operations are fixed, so they
    come out the same.  The rest: fp32 accumulation in any order, one rounding to 16 bits per stored tensor.  Measured:
    a layer against the fp64 product rounded once, and dense-rate against sparse-rate kernels, rel up to 2.8e-4 (bf16)
    and 1e-4 (fp16), max one unit in the last place; a chain with the residual added in the linear's epilogue against
    one with it added by the next pass, rel 8.8e-3 and 1.1e-3, max 0.067 and 0.012."""
    kind, bf16 = case["kind"], case["dtype"] == "bf16"
    if kind in ("levels", "int8"):
        return "exact"
    if kind in ("encoder", "swin"):
        return {"rel": 2e-2 if bf16 else 4e-3, "max": 0.25 if bf16 else 0.05}
    return {"rel": 1.2e-3 if bf16 else 4e-4, "max": 0.016 if bf16 else 0.002}

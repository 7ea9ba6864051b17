"""The work that a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain values. ``listed()`` names the fixed ones, ``draw(rng)`` makes another of the same ranges,
``prepare(case, seed)`` builds what a user's program holds before the call, ``run(state)`` is one pass through the
public entry points, ``work(case)`` the bytes and operations the pass cannot do without, and ``tolerance(case)`` the
difference another correct implementation of the same precision may show.

Kinds of work:
  gemm      ``binding.gemm``: FP32 operands in, both converted by the call, FP32 product out
  serve     ``binding.gemm_q``: a small batch of FP32 activations times weights packed ahead of time
  dense     one training step of a stack of ``HbfpLinear`` layers (forward, backward, update in wide storage)
  conv      one training step of an ``HbfpConv3x3`` layer
  quantize  ``binding.quantize``: one FP32 tensor to packed block floating point
  update    ``binding.wide_update``: the optimiser's FP32 update into 16-bit weight storage, views refreshed
"""
from __future__ import annotations

import math

import torch

from paper_1804_01526_b200 import autograd as hbfp_nn
from paper_1804_01526_b200 import binding as hb

# ----------------------------------------------------------------------------- cases


def listed():
    return [
        # the smallest product of the benchmark configurations: three short launches, so host time and latency
        dict(name="gemm_256", kind="gemm", M=256, N=256, K=256, ta=0, tb=0, m=8, b=32, sr=0, law="normal"),
        # a layer whose three extents fit nothing (no multiple of a tile, a vector or a block), in the paper's tile of 24
        dict(name="gemm_ragged", kind="gemm", M=1111, N=777, K=3001, ta=0, tb=0, m=8, b=24, sr=1, law="normal"),
        # a backward-weight product, both operands converted down their columns, in the shortest block of the sweep
        dict(name="gemm_wgrad_b32", kind="gemm", M=1024, N=4096, K=4096, ta=1, tb=0, m=8, b=32, sr=0, law="half_normal"),
        # 12-bit mantissas, the paper's wider format, with stochastic rounding
        dict(name="gemm_4096_m12", kind="gemm", M=4096, N=4096, K=4096, ta=0, tb=0, m=12, b=64, sr=1, law="outliers"),
        # the largest product of the sweep, the benchmark's own workload
        dict(name="gemm_16384", kind="gemm", M=16384, N=16384, K=16384, ta=0, tb=0, m=8, b=128, sr=0, law="lognormal"),
        # inference on a handful of rows against weights that were packed once: bound by reading the weights
        dict(name="serve_16_rows", kind="serve", M=16, N=4096, K=4096, m=8, t=64, sr=0),
        # the small classifier 784-1024-1024-10 at batch 128 with 24 x 24 weight tiles: many short launches
        dict(name="dense_mlp", kind="dense", batch=128, d0=784, d1=1024, d2=1024, d3=10, m=8, t=24, bb=24, loss=1),
        # the two projections of a transformer's feed-forward block, 4096 tokens, 12-bit mantissas
        dict(name="dense_ffn_m12", kind="dense", batch=4096, d0=1024, d1=4096, d2=1024, d3=0, m=12, t=64, bb=64, loss=0),
        # a 3 x 3 convolution of a residual network's first stage at batch 128
        dict(name="conv_64", kind="conv", n=128, hw=32, c=64, f=64, m=8, bb=64),
        # a convolution that doubles the feature maps (the backward-data product differs in kind)
        dict(name="conv_64_to_128", kind="conv", n=128, hw=16, c=64, f=128, m=8, bb=64),
        # a whole 1 GiB activation tensor converted once along its rows
        dict(name="quantize_1gib", kind="quantize", d0=16384, d1=16384, axis=1, m=8, b=32, sr=0),
        # the optimiser's update of a large weight matrix
        dict(name="update_8192", kind="update", d0=8192, d1=8192, m=8, t=64, sr=0),
    ]


_LARGEST = 2 * 16384 ** 3       # operations of the largest listed case


def _log(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]: any value, or one rounded to a multiple of 8 or 64."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    step = rng.choice((1, 1, 8, 64))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(("gemm", "gemm", "serve", "dense", "conv", "quantize", "update"))
    m = rng.choice((4, 8, 8, 8, 12))
    sr = rng.choice((0, 1))
    if kind == "gemm":
        while True:
            M, N, K = (_log(rng, 64, 16384) for _ in range(3))
            # 12-bit and short-block products run at a fraction of the 8-bit rate per operation
            if 8 * M * N * K <= _LARGEST:
                break
        b = rng.choice((24, 32, 64, 128, 0 if m <= 8 else 48))
        return dict(kind=kind, M=M, N=N, K=K, ta=rng.choice((0, 1)), tb=rng.choice((0, 1)), m=m, b=b, sr=sr,
                    law=rng.choice(("normal", "half_normal", "outliers", "lognormal")))
    if kind == "serve":
        return dict(kind=kind, M=_log(rng, 1, 512), N=_log(rng, 256, 8192), K=_log(rng, 256, 8192), m=m,
                    t=rng.choice((24, 32, 64, 128)), sr=sr)
    if kind == "dense":
        return dict(kind=kind, batch=_log(rng, 32, 4096), d0=_log(rng, 64, 4096), d1=_log(rng, 64, 4096),
                    d2=_log(rng, 8, 1024), d3=0, m=rng.choice((8, 8, 12)), t=rng.choice((24, 32, 64)),
                    bb=rng.choice((24, 32, 64)), loss=rng.choice((0, 1)))
    if kind == "conv":
        return dict(kind=kind, n=_log(rng, 8, 128), hw=rng.choice((8, 16, 32)), c=rng.choice((32, 64, 64, 96, 128)),
                    f=rng.choice((32, 64, 64, 96, 128, 256)), m=rng.choice((4, 8, 8)), bb=64)
    if kind == "quantize":
        while True:
            d0, d1 = _log(rng, 64, 65536), _log(rng, 64, 65536)
            if d0 * d1 <= 1 << 28:
                break
        return dict(kind=kind, d0=d0, d1=d1, axis=rng.choice((0, 1)), m=m, b=rng.choice((24, 32, 64, 128)), sr=sr)
    return dict(kind=kind, d0=_log(rng, 256, 8192), d1=_log(rng, 256, 8192), m=m, t=rng.choice((24, 32, 64, 128)), sr=sr)


# ----------------------------------------------------------------------------- inputs


def _values(law, shape, gen):
    """FP32 values of the benchmark configurations' laws, drawn on the GPU."""
    x = torch.randn(shape, generator=gen, device="cuda")
    if law == "half_normal":
        x.clamp_(min=0)                              # what a ReLU leaves
    elif law == "grad":
        x.mul_(1e-3 ** 0.5)
    elif law == "outliers":
        hit = torch.rand(shape, generator=gen, device="cuda") < 0.01
        x[hit] *= 100.0
    elif law == "lognormal":
        x = x.mul_(2.0).exp_()
        x *= torch.randint(0, 2, shape, generator=gen, device="cuda").mul_(2).sub_(1)
    return x


def _fmt(m, b, sr, sid, tile=0, seed=1):
    return hb.Format(mant_bits=m, block=b, tile=tile, rounding=sr, seed=seed, stream_id=sid)


def _dims(case):
    return [d for d in (case["d0"], case["d1"], case["d2"], case["d3"]) if d]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
    kind, m = case["kind"], case["m"]
    s = dict(case)
    if kind == "gemm":
        M, N, K, ta, tb = (case[k] for k in ("M", "N", "K", "ta", "tb"))
        s["A"] = _values(case["law"], (K, M) if ta else (M, K), gen)
        s["B"] = _values("lognormal" if case["law"] == "lognormal" else "normal", (N, K) if tb else (K, N), gen)
        s["fa"], s["fb"] = _fmt(m, case["b"], case["sr"], 0), _fmt(m, case["b"], case["sr"], 1)
    elif kind == "serve":
        w = _values("normal", (case["K"], case["N"]), gen).mul_((2.0 / case["K"]) ** 0.5)
        s["x"] = _values("half_normal", (case["M"], case["K"]), gen)
        s["w"] = hb.quantize_tiles(w, _fmt(m, case["t"], case["sr"], 1, tile=case["t"]), want_grid=False)[0]
        s["fa"] = _fmt(m, case["t"], case["sr"], 0)
    elif kind == "dense":
        dims = _dims(case)
        torch.manual_seed(seed)                      # the layers draw their initial weights
        s["layers"] = [hbfp_nn.HbfpLinear(i, o, mant_bits=m, tile=case["t"], rounding=1, seed=1, stream_id=10 * k,
                                          batch_block=case["bb"]) for k, (i, o) in enumerate(zip(dims, dims[1:]))]
        s["x"] = _values("normal", (case["batch"], dims[0]), gen)
        if case["loss"]:
            s["labels"] = torch.randint(0, dims[-1], (case["batch"],), generator=gen, device="cuda")
        else:                                        # a layer inside a larger model: the gradient comes from above
            s["x"].requires_grad_(True)
            s["dy"] = _values("grad", (case["batch"], dims[-1]), gen)
    elif kind == "conv":
        n, hw, c, f = (case[k] for k in ("n", "hw", "c", "f"))
        torch.manual_seed(seed)
        s["layer"] = hbfp_nn.HbfpConv3x3(c, f, mant_bits=m, pixel_block=case["bb"])
        s["x"] = _values("half_normal", (n, hw, hw, c), gen).requires_grad_(True)
        s["dy"] = _values("grad", (n, hw, hw, f), gen)
    elif kind == "quantize":
        s["x"] = _values("normal", (case["d0"], case["d1"]), gen)
        s["fmt"] = _fmt(m, case["b"], case["sr"], 0)
    else:
        d0, d1 = case["d0"], case["d1"]
        s["fmt"] = _fmt(m, case["t"], case["sr"], 0, tile=case["t"])
        w = _values("normal", (d0, d1), gen).mul_((2.0 / d0) ** 0.5)
        s["wide"], s["views"] = hb.wide_quantize(w, s["fmt"])
        s["delta"] = _values("grad", (d0, d1), gen).mul_(1e-3)
    return s


# ----------------------------------------------------------------------------- one pass

_LR = 1e-3


def _packed(p):
    """The bytes a packed operand is defined by (the buffers' tails beyond the last row are not written)."""
    lay = hb.packed_layout(p.rows, p.k, p.fmt)
    planes = p.mant.view(lay["planes"], lay["plane_stride"])[:, :p.rows * lay["kst"]]
    return [planes, p.exps[:lay["nkb"] * lay["rs"]]]


def run(s):
    kind = s["kind"]
    if kind == "gemm":
        return hb.gemm(s["ta"], s["tb"], s["A"], s["B"], s["fa"], s["fb"])
    if kind == "serve":
        return hb.gemm_q(s["M"], s["N"], s["K"], s["x"], s["w"], fmtA=s["fa"])
    if kind == "quantize":
        return _packed(hb.quantize(s["x"], s["axis"], s["fmt"]))
    if kind == "update":
        hb.wide_update(s["wide"], s["delta"], s["fmt"], views=s["views"])
        return [s["wide"].mant, s["wide"].exps, _packed(s["views"][0]), _packed(s["views"][1])]
    if kind == "dense":
        layers, x = s["layers"], s["x"]
        x.grad = None
        for layer in layers:
            layer.weight.grad = layer.bias.grad = None
        h = x
        for k, layer in enumerate(layers):
            h = layer(h if k == 0 else torch.relu(h))
        if s["loss"]:
            torch.nn.functional.cross_entropy(h, s["labels"]).backward()
        else:
            h.backward(s["dy"])
        out = {"y": h.detach(), "dx": x.grad, "dw": [p.weight.grad for p in layers], "db": [p.bias.grad for p in layers]}
    else:
        layers, x = [s["layer"]], s["x"]
        x.grad = layers[0].weight.grad = None
        y = layers[0](x)
        y.backward(s["dy"])
        out = {"y": y.detach(), "dx": x.grad, "dw": layers[0].weight.grad}
    with torch.no_grad():
        for layer in layers:
            layer.apply_update(layer.weight.grad * -_LR)
            if kind == "dense":
                layer.bias.sub_(layer.bias.grad, alpha=_LR)
    out["w"] = [layer.weight.detach() for layer in layers]
    out["wide"] = [(layer.wide.mant, layer.wide.exps) for layer in layers]
    return out


# ----------------------------------------------------------------------------- what a pass cannot do without


def _mant(m):
    return 1 if m <= 8 else 2           # bytes per stored mantissa


def work(case):
    kind, m = case["kind"], case["m"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 4 * (M * K + K * N + M * N), "flops": 2 * M * N * K}
    if kind == "serve":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 4 * (M * K + M * N) + _mant(m) * K * N, "flops": 2 * M * N * K}
    if kind == "quantize":
        n = case["d0"] * case["d1"]
        return {"bytes": 4 * n + _mant(m) * n + n // case["b"], "flops": 0}
    if kind == "update":
        n = case["d0"] * case["d1"]     # wide words read and written, the update read, two narrow views written
        return {"bytes": 2 * n + 4 * n + 2 * n + 2 * _mant(m) * n, "flops": 0}
    if kind == "dense":
        dims, batch = _dims(case), case["batch"]
        by = fl = 0
        for k, (i, o) in enumerate(zip(dims, dims[1:])):
            passes = 3 if k or not case["loss"] else 2            # the first layer's input may need no gradient
            fl += 2 * passes * batch * i * o
            # X, Y, dY (and dX), dW; the weights' narrow view per pass; wide words in and out, FP32 copy, two views
            by += 4 * (batch * i * (passes - 1) + 2 * batch * o + i * o) + (passes - 1) * _mant(m) * i * o
            by += i * o * (4 + 4 + 2 * _mant(m))
        return {"bytes": by, "flops": fl}
    n, hw, c, f = case["n"], case["hw"], case["c"], case["f"]
    px, w = n * hw * hw, 9 * c * f
    return {"bytes": 4 * (2 * px * c + 2 * px * f + w) + w * (2 + 4 + 4 + 2), "flops": 3 * 2 * px * w}


# Conversions are exact: packed bytes and wide words have one right answer for given FP32 input. A single product
# differs in the order of its FP32 sums (against the same path with its sums in binary64: at most 2.6e-7 and, for
# single values, 5e-6; blocks of 8-bit mantissas of like magnitude add up exactly). In a dense training step such a
# difference moves a few later conversions to the neighbouring mantissa, and through the update a few wide words with
# them: with 12 bits 3.3e-5, 1.8e-3 for single values and 9e-4 of the words; with 8 bits 1.4e-7 and no word in the
# runs seen, where one moved mantissa would show as some 1e-4 of a value. The convolutions showed no difference.
def tolerance(case):
    if case["kind"] in ("quantize", "update"):
        return "exact"
    if case["kind"] in ("gemm", "serve"):
        return {"rel": 1e-6, "max": 2e-5}
    if case["kind"] == "conv":
        return {"rel": 1e-6, "max": 1e-5, "differ": 1e-4}
    if case["m"] > 8:
        return {"rel": 1.5e-4, "max": 8e-3, "differ": 4e-3}
    return {"rel": 2e-6, "max": 1e-3, "differ": 1e-4}

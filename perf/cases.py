"""Performance cases of the vector-quantized linear layer, through the package's public entry points.

A case is one piece of work of a program that serves or builds a quantized model:

  linear    one projection (DeviceLayer.linear)
  attn      the projections of an attention block: q/k/v over one input (FusedLayers), o (DeviceLayer)
  mlp       the projections of an MLP: gate/up over one input (FusedLayers), down (DeviceLayer)
  layer     a decoder layer: attn and mlp
  restore   the FP16 weight of one projection (DeviceLayer.dequant)
  quantize  one Lloyd iteration of the quantizer on one weight matrix and the packing of its index matrix
            (vptq_assign, vptq_kmeans_update, vptq_pack)

Formats are those of the synthetic workloads (synth.CONFIGS): vector length, main and residual codebook, share of outlier
columns with a codebook of their own, column groups.  Inputs are drawn on the GPU from the seed: uniform indices (what a
codebook made by k-means gives, nearly), normal codebooks and activations, scale and bias per input column.
"""
from __future__ import annotations

import math

import torch

from paper_2409_17066_b200 import binding as vb
from paper_2409_17066_b200 import synth

#: name -> (v, k1, k2, percent of outlier columns, v0, k0, column groups)
FORMATS = {
    "v8_256": (8, 256, 0, 0.0, 0, 0, 1),                    # 1 bit, the smallest codebook
    "v8_65536": (8, 65536, 0, 0.0, 0, 0, 1),                # 2 bit
    "v8_65536_256": (8, 65536, 256, 0.0, 0, 0, 1),          # 3 bit with a residual stage
    "v6_4096_256_out": (6, 4096, 256, 1.0, 4, 4096, 1),     # 3.3 bit with outlier columns
    "v12_4096_4096_out_g4": (12, 4096, 4096, 1.0, 4, 8192, 4),   # the published 2.26-bit setting
}


def listed():
    return [
        # the smallest call: nothing but latency
        dict(name="tiny_decode_b1", kind="linear", fmt="v8_256", M=256, N=512, B=1, x="fp16", out="fp16"),
        # one projection of a 7B model while it generates for one user
        dict(name="7b_q_decode_b1", kind="linear", fmt="v8_65536", M=4096, N=4096, B=1, x="fp16", out="fp16"),
        # the attention projections of a 7B model, four sequences at a time
        dict(name="7b_attn_decode_b4", kind="attn", fmt="v8_65536", hidden=4096, kv=4096, B=4, x="fp16", out="fp16"),
        # the MLP of a 7B model with outlier columns: one user, and a small batch
        dict(name="7b_mlp_decode_b1", kind="mlp", fmt="v6_4096_256_out", hidden=4096, inner=11008, B=1, x="fp16", out="fp16"),
        dict(name="7b_mlp_decode_b16", kind="mlp", fmt="v6_4096_256_out", hidden=4096, inner=11008, B=16, x="fp16", out="fp16"),
        # a decoder layer of a 7B model in the published 2.26-bit setting, one user
        dict(name="7b_2p26_decode_b1", kind="layer", fmt="v12_4096_4096_out_g4", hidden=4096, kv=4096, inner=11008, B=1,
             x="fp16", out="fp16"),
        # a decoder layer of a 70B model, one user, over prepared images
        dict(name="70b_layer_decode_b1", kind="layer", fmt="v8_65536_256", hidden=8192, kv=1024, inner=28672, B=1,
             x="fp16", out="fp16", prepared=True),
        # prompts: the MLP of an 8B model over 512 tokens with FP32 results; the attention projections of a 70B model
        # over a prompt of no round length; a decoder layer in the published setting, whose outlier columns lie where
        # the quantizer found them
        dict(name="8b_mlp_prefill_512", kind="mlp", fmt="v8_65536_256", hidden=4096, inner=14336, B=512, x="bf16", out="fp32"),
        dict(name="70b_attn_prefill_333", kind="attn", fmt="v8_65536_256", hidden=8192, kv=1024, B=333, x="fp16", out="fp16"),
        dict(name="7b_2p26_prefill_512", kind="layer", fmt="v12_4096_4096_out_g4", hidden=4096, kv=4096, inner=11008, B=512,
             x="fp16", out="fp16", perm=True),
        # the restored weight of a large projection (export, inspection, other kernels)
        dict(name="70b_down_restore", kind="restore", fmt="v8_65536_256", M=8192, N=28672),
        # building a model: one Lloyd iteration and the packing of a 7B projection
        dict(name="7b_q_quantize", kind="quantize", M=4096, N=4096, v=8, k=65536),
    ]


def _size(rng, lo, hi):
    """A length between lo and hi, spread over its logarithm: half of the time a multiple of 64, else any number."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, max(lo, n // 64 * 64)) if rng.random() < 0.5 else n


def draw(rng):
    what = rng.choice(["one", "one", "block", "prefill", "prefill", "restore", "quantize"])
    if what == "quantize":
        v, k = rng.choice([(8, 65536), (8, 4096), (6, 4096), (12, 4096), (8, 256), (4, 256)])
        return dict(kind="quantize", M=_size(rng, 384, 4096) // v * v, N=_size(rng, 384, 4096), v=v, k=k)
    fmt = rng.choice(sorted(FORMATS))
    if what == "restore":
        return dict(kind="restore", fmt=fmt, M=_size(rng, 256, 14336), N=_size(rng, 256, 14336))
    c = dict(kind="linear", fmt=fmt, x=rng.choice(["fp16", "bf16"]), out=rng.choice(["fp16", "bf16", "fp32"]))
    if FORMATS[fmt][3] and rng.random() < 0.5:
        c["perm"] = True
    if what == "prefill":
        c.update(M=_size(rng, 1024, 14336), N=_size(rng, 1024, 14336), B=int(round(math.exp(rng.uniform(math.log(17), math.log(1024))))))
        return c
    c["B"] = rng.choice([1, 1, 1, 2, 3, 4, 5, 8, 11, 16])
    if what == "one":
        c.update(M=_size(rng, 256, 28672), N=_size(rng, 512, 14336))
    else:
        hidden, inner = _size(rng, 1024, 8192), _size(rng, 2048, 14336)
        kind = rng.choice(["attn", "mlp"])
        c.update(dict(kind=kind, hidden=hidden, inner=inner) if kind == "mlp" else
                 dict(kind=kind, hidden=hidden, kv=max(128, hidden // rng.choice([1, 4, 8]))))
    if fmt == "v8_65536_256" and c["B"] == 1:
        c["prepared"] = rng.random() < 0.5
    return c


# ---- shapes ------------------------------------------------------------------------------------------

def _calls(c):
    """The case's calls: (shapes [(M, N), ...] of the projections that share the call's input)."""
    if c["kind"] in ("linear", "restore"):
        return [[(c["M"], c["N"])]]
    h = c["hidden"]
    out = []
    if c["kind"] in ("attn", "layer"):
        out += [[(h, h), (c["kv"], h), (c["kv"], h)], [(h, h)]]
    if c["kind"] in ("mlp", "layer"):
        out += [[(c["inner"], h)] * 2, [(h, c["inner"])]]
    return out


def _spec(c, M, N):
    v, k1, k2, pct, v0, k0, groups = FORMATS[c["fmt"]]
    return synth.LayerSpec("p", M, N, v=v, k1=k1, k2=k2, n_out=synth.outlier_columns(N, pct), v0=v0, k0=k0,
                           x_dtype=c.get("x", "fp16"), out_dtype=c.get("out", "fp16"), n_groups=groups,
                           permuted=bool(c.get("perm")))


# ---- inputs ------------------------------------------------------------------------------------------

def _layer(spec, gen):
    """A resident layer with tables and indices drawn on the GPU."""
    def ints(k, shape):
        return torch.randint(0, k, shape, generator=gen, device="cuda", dtype=torch.int32).cpu().numpy()

    def normal(sd, shape):
        return (torch.randn(shape, generator=gen, device="cuda") * sd).half().cpu().numpy()

    d = dict(spec=spec, idx1=ints(spec.k1, (spec.R, spec.Nc)), idx2=ints(spec.k2, (spec.R, spec.Nc)) if spec.k2 else None,
             idx0=ints(spec.k0, (spec.R0, spec.n_out)) if spec.n_out else None,
             c1=normal(0.02, (spec.n_groups * spec.k1, spec.v)),
             c2=normal(0.005, (spec.n_groups * spec.k2, spec.v)) if spec.k2 else None,
             c0=normal(0.02, (spec.k0, spec.v0)) if spec.n_out else None,
             scale=(torch.rand(spec.N, generator=gen, device="cuda") + 0.5).half().cpu().numpy(), bias=normal(0.01, (spec.N,)))
    if spec.permuted:
        d["col_perm"] = torch.randperm(spec.N, generator=gen, device="cuda").int().cpu().numpy()
    return vb.DeviceLayer(d)


class _Call:
    """Projections that share an input: one DeviceLayer, or several behind FusedLayers, with input and results."""

    def __init__(self, c, shapes, gen):
        layers = [_layer(_spec(c, M, N), gen) for M, N in shapes]
        if c.get("prepared"):
            n_sm = torch.cuda.get_device_properties(0).multi_processor_count
            rows = [dl.spec.R for dl in layers]
            shares = [0] if len(layers) == 1 else vb.prepared_shares(rows, n_sm, -(-layers[0].spec.k1 // 4096))
            layers = [dl.prepared(n) for dl, n in zip(layers, shares)]
        x_t = {"fp16": torch.float16, "bf16": torch.bfloat16}[c["x"]]
        out_t = {"fp16": torch.float16, "bf16": torch.bfloat16, "fp32": torch.float32}[c["out"]]
        self.x = torch.randn((c["B"], shapes[0][1]), generator=gen, device="cuda").to(x_t)
        self.outs = [torch.empty((c["B"], M), dtype=out_t, device="cuda") for M, _ in shapes]
        self.layer = layers[0] if len(layers) == 1 else vb.FusedLayers(layers)
        self.one = len(layers) == 1

    def run(self):
        return [self.layer.linear(self.x, self.outs[0])] if self.one else self.layer.linear(self.x, self.outs)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if case["kind"] == "quantize":
        M, N, v, k = case["M"], case["N"], case["v"], case["k"]
        return dict(kind="quantize", v=v, k=k, W=(torch.randn((M, N), generator=gen, device="cuda") * 0.02).half(),
                    codebook=(torch.randn((k, v), generator=gen, device="cuda") * 0.02).half(),
                    weight=torch.rand(N, generator=gen, device="cuda") + 0.1)
    if case["kind"] == "restore":
        return dict(kind="restore", layer=_layer(_spec(case, case["M"], case["N"]), gen))
    return dict(kind="linear", calls=[_Call(case, shapes, gen) for shapes in _calls(case)])


def run(state):
    if state["kind"] == "quantize":
        codebook = state["codebook"].clone()        # the old one is kept: the iteration ends when it no longer moves
        idx = vb.vptq_assign(state["W"], state["v"], codebook)
        vb.vptq_kmeans_update(state["W"], state["v"], idx, codebook, state["weight"])
        return dict(idx=idx, codebook=codebook, packed=vb.vptq_pack(idx, state["k"]))
    if state["kind"] == "restore":
        return state["layer"].dequant()
    return [call.run() for call in state["calls"]]


# ---- what a pass cannot do without ---------------------------------------------------------------------

def _bits(k):
    return max(1, (k - 1).bit_length())


def _layer_bytes(s):
    """Index streams, codebooks, scale and bias (and the column order) of a layer, each once."""
    n = s.R * s.Nc * (_bits(s.k1) + (_bits(s.k2) if s.k2 else 0)) / 8 + 2 * s.n_groups * s.v * (s.k1 + s.k2) + 4 * s.N
    if s.n_out:
        n += s.R0 * s.n_out * _bits(s.k0) / 8 + 2 * s.k0 * s.v0
    return n + (4 * s.N if s.permuted else 0)


def work(case):
    if case["kind"] == "quantize":
        M, N, v, k = case["M"], case["N"], case["v"], case["k"]
        vectors = -(-M // v) * N
        # a distance is v products and sums (||c||^2 - 2 x.c: the rest of it does not depend on the pair)
        return {"bytes": 2.0 * M * N + 4.0 * N + 4.0 * k * v + 4.0 * vectors + vectors * _bits(k) / 8, "flops": 2.0 * vectors * k * v}
    if case["kind"] == "restore":
        s = _spec(case, case["M"], case["N"])
        return {"bytes": _layer_bytes(s) + 2.0 * s.M * s.N, "flops": 2.0 * s.M * s.N}
    B, out_b = case["B"], 4 if case["out"] == "fp32" else 2
    nbytes = flops = 0.0
    for shapes in _calls(case):
        nbytes += 2.0 * B * shapes[0][1]
        for M, N in shapes:
            nbytes += _layer_bytes(_spec(case, M, N)) + 1.0 * B * M * out_b
            flops += 2.0 * B * M * N
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "restore":
        return "exact"
    if case["kind"] == "quantize":
        # indices and packed bytes are exact; centroids are FP32 sums rounded to FP16
        return {"rel": 2e-4, "max": 2e-3, "differ": 0.0}
    # x*scale and the centroid sum are rounded to FP16 (2^-11 each) before FP32 sums; then the result's own rounding
    return {"rel": 4e-3, "max": 2e-2} if case["out"] == "bf16" else {"rel": 1e-3, "max": 5e-3}

"""Timed cases of the codebook-binary linear layer: what a program that serves or builds such a model has it do.

Every case is a dict of plain values; `kind` names the part of the work it stands for:

  layer      one projection called on its own, `linear(...)`: decode for up to 8 rows of x, prefill above; optionally with
             the mean term (`mu`), a 16-bit output and the activation transform (k1 x k2 Kronecker factors)
  step       the seven projections of a transformer block as one `GemvBatch` (q, k, v, o: H x H; gate, up: I x H;
             down: H x I), indices in uint16 containers or as dense bit fields
  token      a token's walk through all blocks of a model: {q, k, v}, {o}, {gate, up}, {down}, each reading what the one
             before it wrote (fp16 between the layers)
  shared     one activation transform, then the layers that read its result as one `GemvBatch`
  codebook   binary K-means over the blocks of a sign matrix

Widths are those of the 7B / 13B layer sets in workloads/gen.py, codebook sizes those of its configurations and of the
table of codebook shapes at 0.8 bit (v8c85, v10c256, v12c777, v14c2353, v16c7132, v18c21619, v20c65536).  K/v is a multiple
of 8, as it is for every projection of those layer sets.
"""
from __future__ import annotations

import math

import torch

import paper_2506_12040_b200 as btc

_DT = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
_SHAPES = ((8, 85), (10, 256), (12, 777), (14, 2353), (16, 4096), (16, 7132), (16, 8192), (18, 21619), (20, 65536))
_LARGEST_MNK = 2048 * 11008 * 4096


def _layer(name, N, K, v, Kc, M, x="f16", out="f32", dist="uniform", mu=False, k1=0, k2=0):
    c = dict(kind="layer", N=N, K=K, v=v, Kc=Kc, M=M, x=x, out=out, dist=dist, mu=mu, k1=k1, k2=k2)
    return dict(c, name=name) if name else c


def _step(name, H, I, v, Kc, M, packed=False, x="f16", dist="uniform"):
    c = dict(kind="step", H=H, I=I, v=v, Kc=Kc, M=M, packed=packed, x=x, dist=dist)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one attention projection, one token (configuration 1); launches and host work are all of it
        _layer("decode_4096x4096", 4096, 4096, 16, 4096, 1),
        # four sequences through a 13B gate projection; a codebook of 65536 does not fit shared memory (configuration 3)
        _layer("decode_13824x5120_v20_m4", 13824, 5120, 20, 65536, 4, dist="zipf"),
        # the 13B down projection with the v = 18 codebook of the table: a block length that is not a multiple of 4
        _layer("decode_5120x13824_v18", 5120, 13824, 18, 21619, 1, mu=True),
        # the layer set of a 7B block (configuration 2): one sequence, eight sequences, and on 13-bit index rows
        _step("step_7b_m1", 4096, 11008, 16, 8192, 1),
        _step("step_7b_m8", 4096, 11008, 16, 8192, 8),
        _step("step_7b_packed", 4096, 11008, 16, 8192, 1, packed=True),
        # one token of a 32-block 7B model (configuration 5): 128 dependent launches over 810 MB of indices
        dict(name="token_7b", kind="token", H=4096, I=11008, v=16, Kc=4096, M=1, blocks=32, dist="uniform"),
        # q, k and v of a block behind the one transform of their input
        dict(name="qkv_transform", kind="shared", N=4096, layers=3, k1=64, k2=64, v=16, Kc=8192, M=1, x="f16"),
        # a short prompt of odd length through the long-K projection, mean term, 16-bit result
        _layer("prefill_77_4096x11008", 4096, 11008, 16, 8192, 77, out="f16", mu=True),
        # a prompt through a projection with its transform (configuration 4 at 512 rows)
        _layer("prefill_512_transform", 4096, 4096, 16, 8192, 512, x="bf16", out="bf16", k1=64, k2=64),
        # the largest prefill (configuration 4 at 2048 rows)
        _layer("prefill_2048_11008x4096", 11008, 4096, 16, 8192, 2048, x="bf16"),
        # the codebook of a 4096 x 4096 layer
        dict(name="codebook_1m_v16", kind="codebook", n=1048576, v=16, Kc=8192),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi, v):
    """A width near a log-uniform draw that blocks of v divide into a multiple of 8 blocks."""
    return max(1, round(_log(rng, lo, hi) / (8 * v))) * 8 * v


def draw(rng):
    """One more case: half of them single layers (decode and prefill alike), the rest block steps, tokens, shared
    transforms and codebooks; sizes log-uniform, odd row counts and ragged N among them."""
    kind = rng.choice(("decode", "decode", "prefill", "prefill", "step", "token", "shared", "codebook"))
    x, out = rng.choice(("f16", "bf16")), rng.choice(("f32", "f16", "bf16"))
    v, Kc = rng.choice(_SHAPES)
    if kind == "decode":
        return _layer("", _log(rng, 1000, 16000), _width(rng, 1024, 16384, v), v, Kc, rng.randint(1, 8), x, out,
                      rng.choice(("uniform", "zipf")), rng.random() < 0.3)
    if kind == "prefill":
        M, N = _log(rng, 9, 2048), _log(rng, 1000, 12000)
        if rng.random() < 0.25:
            k1, k2 = rng.choice((16, 32, 40, 48, 64, 86)), rng.choice((64, 128))
            v, Kc = rng.choice(((16, 4096), (16, 7132), (16, 8192)))
            N = max(1000, min(N, _LARGEST_MNK // (M * k1 * k2)))
            return _layer("", N, k1 * k2, v, Kc, M, x, out, "uniform", False, k1, k2)
        K = _width(rng, 1024, min(12000, max(1100, _LARGEST_MNK // (M * N))), v)
        return _layer("", N, K, v, Kc, M, x, out, rng.choice(("uniform", "zipf")), rng.random() < 0.3)
    if kind == "step":
        packed = rng.random() < 0.3
        v, Kc = rng.choice(((16, 4096), (16, 7132), (16, 8192))) if packed else rng.choice(((8, 85), (12, 777), (16, 4096), (16, 8192), (20, 65536)))
        H = _width(rng, 1024, 5120, v)
        return _step("", H, round(H * 2.7 / (8 * v)) * 8 * v, v, Kc, rng.randint(1, 8), packed, x, rng.choice(("uniform", "zipf")))
    if kind == "token":
        H = _width(rng, 1024, 4096, 16)
        return dict(kind="token", H=H, I=round(H * 2.7 / 128) * 128, v=16, Kc=rng.choice((256, 4096, 8192, 65536)), M=rng.randint(1, 4),
                    blocks=rng.randint(4, 32), dist=rng.choice(("uniform", "zipf")))
    if kind == "shared":
        return dict(kind="shared", N=_log(rng, 1000, 12000), layers=rng.randint(2, 3), k1=rng.choice((16, 32, 40, 64, 86)), k2=rng.choice((64, 128)),
                    v=16, Kc=rng.choice((4096, 7132, 8192)), M=rng.randint(1, 8), x=x)
    v, Kc = rng.choice(((12, 777), (14, 2353), (16, 4096), (16, 7132), (16, 8192)))
    return dict(kind="codebook", n=_log(rng, 65536, 1048576), v=v, Kc=Kc)


# ---------------------------------------------------------------------------------------------- inputs
def _codebook(v, Kc, g):
    """Kc distinct sign patterns, packed for the kernels."""
    pats = torch.randperm(1 << v, generator=g, device="cuda")[:Kc]
    bits = (pats[:, None] >> torch.arange(v, device="cuda")[None, :]) & 1
    return btc.codebook_pack((2 * bits - 1).to(torch.int8).contiguous())


def _indices(N, Kb, Kc, dist, g):
    if dist == "zipf":
        w = torch.arange(1, Kc + 1, dtype=torch.float64, device="cuda") ** -1.1
        cdf = torch.cumsum(w, 0) / w.sum()
        idx = torch.searchsorted(cdf, torch.rand(N * Kb, generator=g, device="cuda", dtype=torch.float64), right=True).clamp_(max=Kc - 1)
        return idx.to(torch.int32).to(torch.int16).view(N, Kb)
    return torch.randint(0, Kc, (N, Kb), generator=g, device="cuda", dtype=torch.int32).to(torch.int16)


def _activations(M, K, dt, g):
    """N(0, 1), with one channel in a thousand twenty times larger (activation outliers)."""
    x = torch.randn((M, K), generator=g, device="cuda")
    x[:, torch.randperm(K, generator=g, device="cuda")[: math.ceil(K / 1000)]] *= 20.0
    return x.to(_DT[dt])


def _weights(N, K, v, Kc, dist, g, unit_gain=False, mu=False):
    """One layer: row scales |N(0, 0.02^2)|, or N(0, 1/K) for chains, which keep the activations' magnitude."""
    a = torch.randn(N, generator=g, device="cuda")
    a = a / math.sqrt(K) if unit_gain else a.abs() * 0.02
    return dict(idx=_indices(N, K // v, Kc, dist, g), C_packed=_codebook(v, Kc, g), alpha=a.half(), v=v, Kc=Kc,
                mu=(torch.randn(N, generator=g, device="cuda") * 0.002).half() if mu else None)


def _transform(k1, k2, g):
    """Sign flips and two orthogonal factors, as a learned transformation pair has them."""
    K = k1 * k2
    sigma = torch.randint(-(1 << 31), 1 << 31, ((K + 31) // 32,), generator=g, device="cuda").to(torch.int32)
    q = [torch.linalg.qr(torch.randn((k, k), generator=g, device="cuda"))[0].contiguous() for k in (k1, k2)]
    return sigma, q[0], q[1]


def _projections(H, I):
    return [(H, H)] * 4 + [(I, H)] * 2 + [(H, I)]


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind, v, Kc = case["kind"], case["v"], case["Kc"]
    if kind == "codebook":
        # blocks near one of 4096 prototypes (Zipf frequencies), every element flipped with probability 0.06
        n = case["n"]
        pick = _indices(n, 1, 4096, "zipf", g).view(-1).long()
        words = torch.randint(0, 1 << v, (4096,), generator=g, device="cuda", dtype=torch.int32)[pick]
        for t in range(v):
            words ^= (torch.rand(n, generator=g, device="cuda") < 0.06).to(torch.int32) << t
        return dict(case=case, vecs=words)
    if kind == "layer":
        w = _weights(case["N"], case["K"], v, Kc, case["dist"], g, mu=case["mu"])
        w["transform"] = _transform(case["k1"], case["k2"], g) if case["k1"] else None
        return dict(case=case, x=_activations(case["M"], case["K"], case["x"], g), w=w, out_dtype=_DT[case["out"]])
    if kind == "step":
        xs = {K: _activations(case["M"], K, case["x"], g) for K in (case["H"], case["I"])}
        layers = []
        for N, K in _projections(case["H"], case["I"]):
            w = dict(_weights(N, K, v, Kc, case["dist"], g), x=xs[K])
            if case["packed"]:
                w.update(idx=btc.index_pack(w["idx"], Kc), idx_bits=btc.index_bits(Kc))
            layers.append(w)
        return dict(case=case, batch=btc.GemvBatch(layers))
    if kind == "shared":
        K = case["k1"] * case["k2"]
        xt = torch.empty((case["M"], K), dtype=torch.float32, device="cuda")
        layers = [dict(_weights(case["N"], K, v, Kc, "uniform", g), x=xt) for _ in range(case["layers"])]
        return dict(case=case, x=_activations(case["M"], K, case["x"], g), xt=xt, transform=_transform(case["k1"], case["k2"], g),
                    batch=btc.GemvBatch(layers))
    # token: fp16 activations, unit-gain layers, the buffers of a block kept from block to block as a decoder keeps them
    M, H, I = case["M"], case["H"], case["I"]
    x = torch.randn((M, H), generator=g, device="cuda").half()
    buf = lambda N: torch.empty((M, N), dtype=torch.float16, device="cuda")
    stages, h = [], x
    for _ in range(case["blocks"]):
        qkv, o, gu, down = [buf(H) for _ in range(3)], buf(H), [buf(I) for _ in range(2)], buf(H)
        for K, src, outs in ((H, h, qkv), (H, qkv[0], [o]), (H, o, gu), (I, gu[0], [down])):
            stages.append(btc.GemvBatch([dict(_weights(t.shape[1], K, v, Kc, case["dist"], g, unit_gain=True), x=src, out=t) for t in outs]))
        h = down
    return dict(case=case, stages=stages)


def run(state):
    kind = state["case"]["kind"]
    if kind == "layer":
        w = state["w"]
        return btc.linear(state["x"], w["idx"], w["C_packed"], w["alpha"], w["v"], w["Kc"], mu=w["mu"], out_dtype=state["out_dtype"],
                          transform=w["transform"])
    if kind == "step":
        return state["batch"].run()
    if kind == "shared":
        btc.activation_transform(state["x"], state["transform"], out=state["xt"])
        return [state["xt"], *state["batch"].run()]
    if kind == "token":
        for stage in state["stages"]:
            stage.run()
        return [stage.outs for stage in state["stages"][-4:]]
    return btc.codebook_kmeans(state["vecs"], state["case"]["v"], state["case"]["Kc"])


# ---------------------------------------------------------------------------------------------- what a pass needs
def _layer_work(M, N, K, v, Kc, ysize, bits=16, mu=False, xsize=2):
    """Indices, public codewords, scales, activations and result once each; the contraction's operations."""
    b = N * (K // v) * bits / 8 + 4 * Kc + (4 if mu else 2) * N + xsize * M * K + ysize * M * N
    return b, 2.0 * M * N * K


def work(case):
    kind, v, Kc = case["kind"], case["v"], case["Kc"]
    if kind == "codebook":
        # vectors in, assignments and centroids out; two rounds of nearest-centroid searches at least (the second finds
        # nothing changed) over the distinct vectors, at most 2^v
        return {"bytes": 6.0 * case["n"] + 4.0 * Kc, "flops": 2 * 2.0 * v * min(case["n"], 1 << v) * Kc}
    M = case["M"]
    if kind == "layer":
        parts = [_layer_work(M, case["N"], case["K"], v, Kc, _DT[case["out"]].itemsize, mu=case["mu"])]
        if case["k1"]:
            parts.append((4.0 * (case["k1"] ** 2 + case["k2"] ** 2), 2.0 * M * case["K"] * (case["k1"] + case["k2"])))
    elif kind == "step":
        bits = btc.index_bits(Kc) if case["packed"] else 16
        parts = [_layer_work(M, N, K, v, Kc, 4, bits=bits) for N, K in _projections(case["H"], case["I"])]
    elif kind == "shared":
        K = case["k1"] * case["k2"]
        parts = [_layer_work(M, case["N"], K, v, Kc, 4, xsize=0) for _ in range(case["layers"])]
        parts.append((2.0 * M * K + 4.0 * M * K + 4.0 * (case["k1"] ** 2 + case["k2"] ** 2), 2.0 * M * K * (case["k1"] + case["k2"])))
    else:
        parts = [_layer_work(M, N, K, v, Kc, 2) for N, K in _projections(case["H"], case["I"])] * case["blocks"]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    """Integer results are unique.  Decode sums are fp32 over activations held to 2^-20 of the largest magnitude among a few
    hundred neighbours (an outlier costs the others bits); prefill sums are fp32 over exact products; a 16-bit result, and
    16-bit activations behind a transform or between the layers of a chain, carry that type's rounding."""
    if case["kind"] == "codebook":
        return "exact"
    if case["kind"] == "token":
        return {"rel": 1e-2}                                       # fp16 roundings of up to 128 layers in a row
    rounded = {"f32": 1e-4 if case["M"] <= 8 else 2e-5, "f16": 1e-3, "bf16": 8e-3}
    if case["kind"] == "layer":
        rel = rounded[case["out"]]
        return {"rel": max(rel, rounded[case["x"]]) if case["k1"] and case["M"] > 8 else rel}
    return {"rel": 1e-4}

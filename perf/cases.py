"""Performance cases: the work a user of this package has it do, through the public entry points of
``paper_2205_12268_b200.wcc``.

A case is a dict of plain values with an ``op`` (which entry point) and its sizes.  The listed cases are the named
workloads of ``inputs.CONFIGS`` and ``bench.py`` plus generic sizes for the options and formats around the layer;
``draw`` gives more cases of the same ranges.

    layer      wcc.forward: one compressed 1x1 convolution, workspace and output buffer kept by the caller
    deployed   wcc.forward with what a trained network fixes: 4-bit weight codes prepared once, a clipping
               parameter, skip connection and ReLU on the way out
    padded     wcc.forward_padded: maps whose sides are no multiples of 2^levels
    chain      wcc.Chain: a stack of layers with ReLU between them
    block      wcc.Block: the inverted residual block (expand, depthwise 3x3, project, skip)
    transform  wcc.haar_fwd -> wcc.select_topk -> wcc.haar_inv: the wavelet analysis and synthesis on their own
"""
from __future__ import annotations

import math

import torch

from paper_2205_12268_b200 import inputs
from paper_2205_12268_b200 import wcc


def _named(name, workload, **over):
    N, Cin, Cout, H, W, dtype, levels, gamma, bits, _, _ = inputs.CONFIGS[workload]
    c = dict(name=name, op="layer", N=N, Cin=Cin, Cout=Cout, H=H, W=W, dtype=dtype, levels=levels, gamma=gamma, bits=bits)
    c.update(over)
    return c


def listed():
    return [
        # smallest call: one 64 x 64 map, where launches and latencies are the time
        _named("layer_small_f32", "C1"),
        # projection (many channels to few) on a stride-8 segmentation map, half of the positions kept
        _named("layer_project_bf16", "C2"),
        # expansion (few channels to many) on a large map without quantization: a network before it is quantized
        _named("layer_expand_bf16_unquantized", "C3u"),
        # depth-estimation batch, fp32 maps, one position in eight kept: the headline layer of the benchmark
        _named("layer_headline_f32", "C4"),
        # the same layer at twice the batch: input and output beyond what the L2 holds
        _named("layer_large_batch_f32", "C4", N=24),
        # rows that are no multiple of 16 bytes and channel counts of no round size: an odd stage of a detection network
        dict(name="layer_ragged_bf16", op="layer", N=3, Cin=58, Cout=70, H=60, W=92, dtype="bf16", levels=2, gamma=0.25, bits=8),
        # more channels than one operand tile of the fused kernels: the low-resolution end of a backbone
        dict(name="layer_wide_bf16", op="layer", N=2, Cin=384, Cout=512, H=64, W=128, dtype="bf16", levels=3, gamma=0.25, bits=8),
        # a layer of a trained, quantized network: weight codes and clipping parameter fixed, skip connection and ReLU
        dict(name="deployed_bf16", op="deployed", N=4, Cin=96, Cout=96, H=128, W=256, dtype="bf16", levels=3, gamma=0.25, bits=8),
        # 513 x 1025 input at stride 4: both sides odd
        dict(name="padded_odd_bf16", op="padded", N=2, Cin=64, Cout=64, H=129, W=257, dtype="bf16", levels=3, gamma=0.25, bits=8),
        # six layers 32 -> 192 -> 32 ... with ReLU between them
        dict(name="chain_six_bf16", op="chain", N=2, narrow=32, wide=192, layers=6, H=256, W=512, dtype="bf16", levels=3, gamma=0.25, bits=8),
        # inverted residual block, 256 channels expanded four times
        dict(name="block_bf16", op="block", N=4, C=256, E=1024, H=128, W=128, dtype="bf16", levels=3, gamma=0.25, bits=8),
        # analysis, joint selection and synthesis on their own, fp32
        dict(name="transform_f32", op="transform", N=4, C=64, H=192, W=320, dtype="f32", levels=3, gamma=0.125),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _side(rng, lo, hi, unit):
    return max(1, _log_int(rng, lo, hi) // unit) * unit


def _fit(most, per_image, n):
    """As many of n images as `most` elements allow; 0 when not even one."""
    return min(n, most // per_image)


def draw(rng):
    op = rng.choice(["layer"] * 5 + ["wide", "deployed", "padded", "chain", "block", "transform"])
    while True:
        levels = rng.choice([1, 2, 2, 3, 3, 3])
        c = dict(op=op, N=_log_int(rng, 1, 24), dtype=rng.choice(["f32", "bf16", "bf16"]), levels=levels,
                 gamma=rng.choice([0.5, 0.25, 0.125, 0.0625]))
        unit = 1 << levels
        if op in ("layer", "deployed", "padded"):
            c.update(Cin=_log_int(rng, 8, 256), Cout=_log_int(rng, 8, 256), bits=rng.choice([8, 8, 8, 6, 4] + ([0] if op != "deployed" else [])))
            u = 1 if op == "padded" else unit
            c.update(H=_side(rng, 16, 512, u), W=_side(rng, 16, 512, u))
            most, per = 24 * 64 * 2 * 96 * 320, (c["Cin"] + c["Cout"]) * c["H"] * c["W"]
            if op == "padded":
                most //= 4
        elif op == "wide":
            c.update(op="layer", Cin=_log_int(rng, 257, 1024), Cout=_log_int(rng, 64, 1024), bits=rng.choice([8, 8, 0]),
                     H=_side(rng, 16, 128, unit), W=_side(rng, 16, 128, max(4, unit)))
            most, per = 2 * (384 + 512) * 64 * 128, (c["Cin"] + c["Cout"]) * c["H"] * c["W"]
        elif op == "chain":
            narrow = _log_int(rng, 8, 48)
            c.update(narrow=narrow, wide=narrow * rng.randint(2, 5), layers=rng.randint(2, 6), bits=8,
                     H=_side(rng, 32, 512, unit), W=_side(rng, 32, 512, max(4, unit)))
            most, per = 2 * (32 + 192) * 256 * 512, (c["narrow"] + c["wide"]) * c["H"] * c["W"]
        elif op == "block":
            C = _log_int(rng, 32, 384)
            c.update(C=C, E=C * rng.randint(1, 6), bits=8, H=_side(rng, 16, 160, unit), W=_side(rng, 16, 160, max(4, unit)))
            most, per = 4 * (256 + 1024) * 128 * 128, (c["C"] + c["E"]) * c["H"] * c["W"]
            if c["dtype"] == "f32":
                most //= 2
        else:
            c.update(C=_log_int(rng, 8, 256), H=_side(rng, 16, 512, unit), W=_side(rng, 16, 512, unit))
            most, per = 4 * 64 * 192 * 320, c["C"] * c["H"] * c["W"]
        c["N"] = _fit(most, per, c["N"])
        if c["N"] >= 1:
            return c


def _keep(case):
    """Kept positions per image (of the padded map where the sides are padded)."""
    u = (1 << case["levels"]) if case["op"] == "padded" else 1
    return inputs.keep_count(case["gamma"], (-(-case["H"] // u) * u) * (-(-case["W"] // u) * u))


def _torch_dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _maps(gen, N, C, H, W, dtype, n_sin=16, fmax=8.0):
    """Feature maps as inputs.feature_map describes them, made on the GPU: rectified sums of sinusoids plus 5 % noise."""
    dev, planes = gen.device, N * C
    out = torch.empty((planes, H, W), dtype=dtype, device=dev)
    step = max(1, (1 << 26) // (H * W))

    def rand(*shape):
        return torch.rand(shape, device=dev, generator=gen)

    col = torch.arange(W, device=dev) / W
    row = torch.arange(H, device=dev) / H
    for p0 in range(0, planes, step):
        n = min(planes, p0 + step) - p0
        a = (2 * math.pi * fmax) * rand(n, n_sin, 1) * col + 2 * math.pi * rand(n, n_sin, 1)
        b = (2 * math.pi * fmax) * rand(n, n_sin, 1) * row
        amp = torch.randn((n, n_sin, 1), device=dev, generator=gen)
        left = torch.cat([amp * b.cos(), amp * b.sin()], 1).transpose(1, 2)
        v = torch.matmul(left, torch.cat([a.sin(), a.cos()], 1)).clamp_(min=0)
        out[p0:p0 + n] = v.add_(torch.randn((n, H, W), device=dev, generator=gen), alpha=0.05)
    return out.reshape(N, C, H, W)


def _weights(gen, Cout, Cin):
    return torch.randn((Cout, Cin), device=gen.device, generator=gen) / math.sqrt(Cin)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    op, N, H, W, levels = case["op"], case["N"], case["H"], case["W"], case["levels"]
    dtype, k, bits = _torch_dtype(case), _keep(case), case.get("bits", 8)
    s = dict(op=op, levels=levels, k=k, bits=bits)
    if op in ("layer", "deployed", "padded"):
        Cin, Cout = case["Cin"], case["Cout"]
        s["x"] = _maps(gen, N, Cin, H, W, dtype)
        s["Wt"] = _weights(gen, Cout, Cin)
        if op != "padded":
            s["ws"] = wcc.Workspace.for_problem(s["x"], Cout, levels, k, bits)
            s["y"] = torch.empty((N, Cout, H, W), dtype=dtype, device="cuda")
        if op == "deployed":
            s["residual"] = _maps(gen, N, Cout, H, W, dtype)
            # calibration: the weight codes, and a clipping parameter a little below the largest kept coefficient
            _, t = wcc.forward(s["x"], s["Wt"], levels, k, bits, taps=("Wq", "scale_w", "scale_a"), wbits=4)
            s["Wq"], s["scale_w"] = t["Wq"], t["scale_w"]
            s["alpha"] = 0.75 * float(t["scale_a"]) * ((1 << (bits - 1)) - 1)
            del s["Wt"]
    elif op == "chain":
        width = [case["narrow"] if i % 2 == 0 else case["wide"] for i in range(case["layers"] + 1)]
        s["x"] = _maps(gen, N, width[0], H, W, dtype)
        s["chain"] = wcc.Chain(s["x"], [_weights(gen, width[i + 1], width[i]) for i in range(case["layers"])], levels, k, bits)
        s["y"] = torch.empty((N, width[-1], H, W), dtype=dtype, device="cuda")
    elif op == "block":
        C, E = case["C"], case["E"]
        s["x"] = _maps(gen, N, C, H, W, dtype)
        s["block"] = wcc.Block(s["x"], _weights(gen, E, C), torch.randn((E, 3, 3), device="cuda", generator=gen) / 3,
                               _weights(gen, C, E), levels, k, bits)
        s["y"] = torch.empty_like(s["x"])
    else:
        s["x"] = _maps(gen, N, case["C"], H, W, dtype)
    return s


def run(s):
    op = s["op"]
    if op == "layer":
        return wcc.forward(s["x"], s["Wt"], s["levels"], s["k"], s["bits"], y=s["y"], ws=s["ws"])
    if op == "deployed":
        return wcc.forward(s["x"], None, s["levels"], s["k"], s["bits"], y=s["y"], ws=s["ws"], alpha=s["alpha"], relu=True,
                           residual=s["residual"], Wq=s["Wq"], scale_w=s["scale_w"])
    if op == "padded":
        return wcc.forward_padded(s["x"], s["Wt"], s["levels"], s["k"], s["bits"])
    if op == "chain":
        return s["chain"](s["x"], s["y"])
    if op == "block":
        return s["block"](s["x"], s["y"])
    coef, nrm2 = wcc.haar_fwd(s["x"], s["levels"])
    idx, tau = wcc.select_topk(nrm2, s["k"])
    back = wcc.haar_inv(coef, s["levels"], dtype=s["x"].dtype)
    return dict(coef=coef, nrm2=nrm2, idx=idx, tau=tau, back=back)


def work(case):
    """Input maps and weights read once, output maps written once; the contraction over the kept positions and the
    transforms' additions (about 4 per element and direction)."""
    N, P, k = case["N"], case["H"] * case["W"], _keep(case)
    es = 2 if case["dtype"] == "bf16" else 4
    op = case["op"]
    if op in ("layer", "padded", "deployed"):
        Cin, Cout = case["Cin"], case["Cout"]
        maps = Cin + Cout * (2 if op == "deployed" else 1)
        wbytes = Cin * Cout * (1 if op == "deployed" else 4)
        return {"bytes": es * N * P * maps + wbytes, "flops": 2 * N * k * Cin * Cout + 4 * N * P * (Cin + Cout)}
    if op == "chain":
        width = [case["narrow"] if i % 2 == 0 else case["wide"] for i in range(case["layers"] + 1)]
        pairs = list(zip(width, width[1:]))
        return {"bytes": es * N * P * (width[0] + width[-1]) + 4 * sum(a * b for a, b in pairs),
                "flops": sum(2 * N * k * a * b + 4 * N * P * (a + b) for a, b in pairs)}
    if op == "block":
        C, E = case["C"], case["E"]
        return {"bytes": es * N * P * 2 * C + 4 * (2 * C * E + 9 * E),
                "flops": 2 * (2 * N * k * C * E + 4 * N * P * (C + E)) + 18 * N * P * E}
    C = case["C"]
    # transform: map -> coefficients and norms; norms -> indices; coefficients -> map
    return {"bytes": N * P * C * (2 * es + 8) + 8 * N * P + 4 * N * k + 4 * N, "flops": N * P * C * 10}


def tolerance(case):
    """About four times the distance between the path and an evaluation of it in float64 (same selection rule, same code
    grids, same rounding of stored maps), measured on the listed sizes and on drawn ones.  A coefficient within a rounding
    error of the middle between two codes may land on either, and one near-tie at the threshold may be kept or dropped:
    single values then move by a code step (``max``), the norm hardly (``rel``)."""
    op = case["op"]
    if op == "transform":                       # fp32 sums of a few terms (1e-7 seen); the norms add up to 256 squares
        return {"rel": 5e-7, "max": 1e-5}
    if op == "chain":                           # each layer requantizes what the one before stored: 2.4e-4 seen after 3 layers, 3.2e-2 after 6
        return {"rel": min(0.03, 5e-4 * 2 ** case["layers"]), "max": 0.99}
    if op == "block":
        return {"rel": 1.2e-3, "max": 0.1}      # two layers: 2.8e-4 seen
    if case["bits"] == 0:
        return {"rel": 4e-4, "max": 0.04}       # bf16 operands, fp32 sums: 8.5e-5 seen
    return {"rel": 8e-4, "max": 0.1}            # 2.1e-4 seen

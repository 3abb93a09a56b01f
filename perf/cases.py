"""The calls whose time this repository cares about, as data: what a program that trains with VeLoRA linear layers asks of
the library, through its public entry points, from the smallest layer to the largest.

A case is one of three kinds of pass.

  layer    one training step of a layer: velora_linear_forward (Y and Z), then velora_linear_backward (dX and dW).
  micro    one optimiser step made of several micro-batches: forward, dX and the factored gradient P = beta * P + dY^T Z
           for each, then one velora_expand_p to dW.
  stream   the three operations on their own: velora_init_v, velora_compress and velora_reconstruct.

Sizes are those of ``velora_inputs`` (and of the tests and the benchmark that use it), values follow its recipe: activations
N(0, 1) with a heavy-tailed scale per channel or a few outlier channels, W ~ N(0, 1 / D), gradients N(0, sigma^2).  Buffers
and the workspace are kept between passes as a training program keeps them.
"""
import math

import torch

from paper_2405_17991_b200 import binding as vl

DEV = "cuda"
_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "f8": torch.float8_e4m3fn}
_BYTES = {"f32": 4, "bf16": 2, "f8": 1}


def _layer(name, N, D, O, Dsub, dtype="bf16", z="f32", dw="bf16", rows="padded", scale="lognormal", sigma=0.5, sigma_dy=1.0):
    """``rows``: "padded" keeps every row on a 16-byte boundary, "dense" is what torch.empty gives."""
    c = dict(kind="layer", N=N, D=D, O=O, Dsub=Dsub, dtype=dtype, z=z, dw=dw, rows=rows, scale=scale, sigma=sigma, sigma_dy=sigma_dy)
    if name:
        c["name"] = name
    return c


def _micro(name, N, D, O, Dsub, z, micro_batches):
    c = dict(kind="micro", N=N, D=D, O=O, Dsub=Dsub, dtype="bf16", z=z, dw="bf16", rows="padded", scale="lognormal", sigma=1.0,
             sigma_dy=1.0, micro_batches=micro_batches)
    if name:
        c["name"] = name
    return c


def _stream(name, N, D, Dsub, z="f32", rows="padded", scale="lognormal", sigma=1.0):
    c = dict(kind="stream", N=N, D=D, Dsub=Dsub, dtype="bf16", z=z, rows=rows, scale=scale, sigma=sigma)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest layer there is: fp32, one tile.  Nothing but calls and launches; what a unit-sized model or a
        # debugging run sees.
        _layer("tiny_fp32_layer", 256, 64, 64, 16, dtype="f32", dw="f32", scale="none"),
        # Attention projection of a LLaMA-60M-shaped block in pre-training: a few microseconds per product.
        _layer("llama60m_q_layer", 8192, 512, 512, 64),
        # Its down projection: 1376 columns are 21.5 sub-tokens, the last one ragged.
        _layer("llama60m_down_layer", 8192, 1376, 512, 64),
        # First MLP layer of a ViT-B/16-shaped block in fine-tuning: 64 x 197 tokens (no multiple of a tile), outlier
        # channels, Z kept in the activations' 16 bits.
        _layer("vit_fc1_layer", 64 * 197, 768, 3072, 32, z="bf16", scale="outlier"),
        # The attention output projection of the same block trained in fp32 throughout.
        _layer("vit_proj_fp32_layer", 64 * 197, 768, 768, 32, dtype="f32", dw="f32", scale="outlier"),
        # Up projection of a LLaMA-1B-shaped block, 2048 -> 5461, on tensors as a framework allocates them: rows of 5461
        # elements with no padding, so that Y and dY rows start on odd boundaries.
        _layer("llama1b_up_dense_rows_layer", 16 * 256, 2048, 5461, 128, rows="dense", sigma_dy=0.1),
        # Down projection of that block with the row pitch padded to 5464, gradient kept in fp32 for the optimiser.
        _layer("llama1b_down_layer", 16 * 256, 5461, 2048, 128, dw="f32", sigma_dy=0.1),
        # Attention projection of a LLaMA-7B-shaped block in fine-tuning: the layer that the paper's tables are about.
        _layer("llama7b_q_layer", 4 * 2048, 4096, 4096, 64, sigma=1.0),
        # The largest: its up projection, with the longer sub-token and Z stored in one byte.
        _layer("llama7b_up_layer", 4 * 2048, 4096, 11008, 256, z="f8", sigma=1.0),
        # Down projection of a rank-16 adapter on the same width: tiny output, one pass over X is all there is to do.
        _layer("adapter_rank16_layer", 4 * 2048, 4096, 16, 64, sigma=1.0),
        # Gradient accumulation over four micro-batches of one sequence each, the gradient kept as its factor P.
        _micro("llama7b_q_micro_batches", 2048, 4096, 4096, 64, "bf16", 4),
        # v from a first batch, then compress and reconstruct as separate operations, on the widest activation.
        _stream("llama7b_down_streams", 4 * 2048, 11008, 64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A layer width: mostly multiples of 64, often only of 8, sometimes odd."""
    w = _log_int(rng, lo, hi)
    k = rng.random()
    step = 64 if k < 0.5 else (8 if k < 0.8 else 1)
    return max(lo, w // step * step)


def _dsub(rng, D):
    """Sub-token lengths in use: the fixed 16 .. 256 and D / 8, D / 16, D / 32 of the ablation, 2 .. 256 sub-tokens a row."""
    fixed = [d for d in (16, 32, 64, 128, 256) if 2 <= -(-D // d) <= 256]
    ratio = [D // k for k in (8, 16, 32) if D % (8 * k) == 0 and 2 <= D // k <= 1024]
    return rng.choice(ratio) if ratio and rng.random() < 0.25 else rng.choice(fixed)


def draw(rng):
    while True:
        k = rng.random()
        N = _log_int(rng, 128, 12608)
        scale, sigma = rng.choice([("lognormal", 0.5), ("lognormal", 1.0), ("outlier", 0.5)])
        z = rng.choice(["f32", "f32", "bf16", "f8"])
        if k < 0.50:                                         # layers in bf16, padded or dense
            D, O = _width(rng, 256, 11008), _width(rng, 256, 11008)
            rows = rng.choice(["padded", "dense"])
            cap = 8192 * 4096 * 11008 if rows == "padded" or (D % 8 == 0 and O % 8 == 0) else 4096 * 2048 * 5461
            if N * D * O > cap:
                continue
            return _layer(None, N, D, O, _dsub(rng, D), z=z, dw=rng.choice(["bf16", "bf16", "f32"]), rows=rows, scale=scale, sigma=sigma,
                          sigma_dy=rng.choice([1.0, 0.1]))
        if k < 0.60:                                         # layers in fp32
            D, O = _width(rng, 64, 1376), _width(rng, 64, 3072)
            if N * D * O > 12608 * 768 * 768:
                continue
            return _layer(None, N, D, O, _dsub(rng, D), dtype="f32", dw="f32", rows="dense", scale=scale, sigma=sigma)
        if k < 0.75:                                         # adapters, rank 4 .. 64
            D = _width(rng, 512, 8192)
            return _layer(None, N, D, rng.randint(4, 64), _dsub(rng, D), z=z, scale=scale, sigma=sigma)
        if k < 0.85:                                         # micro-batches
            D, O = _width(rng, 512, 4096) // 8 * 8, _width(rng, 512, 11008) // 8 * 8
            mb = rng.randint(2, 4)
            N = _log_int(rng, 128, 4096)
            if mb * N * D * O > 8192 * 4096 * 11008:
                continue
            return _micro(None, N, D, O, _dsub(rng, D), z if z != "f8" else "bf16", mb)
        D = _width(rng, 256, 11008)
        return _stream(None, N, D, _dsub(rng, D), z=z if z != "f8" else "f32", rows=rng.choice(["padded", "dense"]), scale=scale, sigma=sigma)


def _matrix(case, n_rows, n_cols, dtype):
    ld = n_cols if case["rows"] == "dense" else -(-n_cols // 8) * 8
    return torch.empty((n_rows, ld), dtype=dtype, device=DEV)[:, :n_cols]


def _normal(case, gen, n_rows, n_cols, dtype, scale=None):
    t = torch.randn((n_rows, n_cols), generator=gen, device=DEV)
    if scale is not None:
        t *= scale
    out = _matrix(case, n_rows, n_cols, dtype)
    out.copy_(t)
    return out


def _channel_scale(case, gen):
    D = case["D"]
    if case["scale"] == "lognormal":
        return torch.exp(case["sigma"] * torch.randn(D, generator=gen, device=DEV))
    c = torch.ones(D, device=DEV)
    if case["scale"] == "outlier":
        c[torch.randperm(D, generator=gen, device=DEV)[: max(1, round(0.01 * D))]] = 20.0
    return c


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    N, D, Dsub = case["N"], case["D"], case["Dsub"]
    M = vl.num_subtokens(D, Dsub)
    dt, zt = _TORCH[case["dtype"]], _TORCH[case["z"]]
    scale = _channel_scale(case, gen)
    s = {"kind": case["kind"], "D": D, "Dsub": Dsub}
    if case["kind"] == "stream":
        s["X"] = _normal(case, gen, N, D, dt, scale)
        s["v"] = torch.empty(Dsub, device=DEV)
        s["Z"] = torch.empty((N, M), dtype=zt, device=DEV)
        s["Xhat"] = _matrix(case, N, D, dt)
        s["ws"] = vl.velora_workspace_alloc(vl.velora_workspace_bytes(vl.OP_INIT_V, N, D, 1, Dsub), DEV)
        return s
    O = case["O"]
    batches = case.get("micro_batches", 1)
    s["X"] = [_normal(case, gen, N, D, dt, scale) for _ in range(batches)]
    s["dY"] = [_normal(case, gen, N, O, dt, case["sigma_dy"]) for _ in range(batches)]
    s["W"] = _normal(case, gen, O, D, dt, D ** -0.5)
    s["Y"] = [_matrix(case, N, O, dt) for _ in range(batches)]
    s["dX"] = [_matrix(case, N, D, dt) for _ in range(batches)]
    s["Z"] = [torch.empty((N, M), dtype=zt, device=DEV) for _ in range(batches)]
    s["dW"] = _matrix(case, O, D, _TORCH[case["dw"]])
    need = max(vl.velora_workspace_bytes(op, N, D, O, Dsub) for op in (vl.OP_LINEAR_FORWARD, vl.OP_LINEAR_BACKWARD_FACTORED, vl.OP_WEIGHT_GRAD_FACTORED))
    s["ws"] = vl.velora_workspace_alloc(need, DEV)
    # The vector is fixed on a first batch and kept; the batch stands in for it here as in the tests.
    s["v"] = s["v_load"] = vl.velora_init_v(s["X"][0], Dsub)
    if case["z"] == "f8":                                    # the scale of an 8-bit Z travels in the vector
        _, s["v"], s["v_load"] = vl.velora_z8_calibrate(s["X"][0], s["v"])
    if case["kind"] == "micro":
        s["P"] = torch.empty((O, M), device=DEV)
    return s


def run(s):
    if s["kind"] == "stream":
        v = vl.velora_init_v(s["X"], s["Dsub"], v=s["v"], ws=s["ws"])
        Z = vl.velora_compress(s["X"], v, Z=s["Z"])
        Xhat = vl.velora_reconstruct(Z, v, s["D"], Xhat=s["Xhat"])
        return {"v": v, "Z": Z, "Xhat": Xhat}
    W, ws = s["W"], s["ws"]
    if s["kind"] == "layer":
        X, dY = s["X"][0], s["dY"][0]
        Y, Z = vl.velora_linear_forward(X, W, s["v"], Y=s["Y"][0], Z=s["Z"][0], ws=ws)
        dX, dW = vl.velora_linear_backward(dY, W, Z, s["v_load"], dX=s["dX"][0], dW=s["dW"], ws=ws)
        return {"Y": Y, "Z": Z, "dX": dX, "dW": dW}
    for i, (X, dY) in enumerate(zip(s["X"], s["dY"])):
        _, Z = vl.velora_linear_forward(X, W, s["v"], Y=s["Y"][i], Z=s["Z"][i], ws=ws)
        vl.velora_linear_backward(dY, W, Z, s["v_load"], dX=s["dX"][i], need_dW=False, ws=ws)
        vl.velora_weight_grad_p(dY, Z, s["D"], s["Dsub"], P=s["P"], beta=1 if i else 0, ws=ws)
    dW = vl.velora_expand_p(s["P"], s["v_load"], s["D"], dW=s["dW"])
    return {"Y": s["Y"], "Z": s["Z"], "dX": s["dX"], "P": s["P"], "dW": dW}


def work(case):
    N, D = case["N"], case["D"]
    M = vl.num_subtokens(D, case["Dsub"])
    b, bz = _BYTES[case["dtype"]], _BYTES[case["z"]]
    if case["kind"] == "stream":                             # X in, Z and Xhat out; sums, products, expansion
        return {"bytes": N * D * b * 2 + N * M * bz, "flops": 4 * N * D}
    O, n = case["O"], case.get("micro_batches", 1)
    per_batch = {"bytes": 2 * N * D * b + 2 * N * O * b + N * M * bz, "flops": 4 * N * D * O + 2 * N * D + 2 * N * O * M}
    return {"bytes": n * per_batch["bytes"] + O * D * (b + _BYTES[case["dw"]]), "flops": n * per_batch["flops"] + O * D}


def tolerance(case):
    """About four times what the path shows against the same arithmetic in 64 bits.  fp32: up to 2e-6 in norm and 4.3e-5 for one
    value (dW).  bf16: 2.3e-3 in norm (one rounding of the result, one of Z on its way into the gradient's products) and 0.072
    for one value (a dW column of an outlier channel that nearly cancels).  An 8-bit Z that sits on the border of two codes may
    take either, which are up to an eighth apart."""
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 2e-4}
    return {"rel": 1e-2, "max": 0.25}

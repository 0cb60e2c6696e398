"""The work that users of this library have it do, as timing cases.

``listed()`` names the standing cases, ``draw(rng)`` makes one more of the same ranges, ``prepare`` builds
what a program holds before the call, ``run`` makes one pass through the public entry points, ``work`` counts
what the pass cannot do without, ``tolerance`` says how far two correct implementations may differ and ``exact``
gives the same outputs in binary64.

Kinds of work:

  infer        one linear layer of a serving program: the weights were quantized when the model was loaded, the
               activations are quantized in the call.  ``packed`` is false when the layer keeps its own workspace
               with the tensor-core operand of w in it, true when all layers of a model share one workspace and a
               layer keeps only its packed codes.  Every buffer is kept; no masks (there is no backward pass).
  forward      Algorithm 1 as written: x and w quantized, contracted, everything returned.
  train        forward and backward pass (Algorithm 2) of one linear layer.
  mlp          the MLP block (gate, up, SwiGLU, down) with kept buffers.
  fp4          the forward pass on the FP4 grid.
  weight_only  b-bit weights, bfloat16 activations.
  gemm         the contraction of two packed tensors.
  quantize     codes, scales and masks of one tensor.
"""
import math

import torch

import paper_2502_05003_b200 as quest

_DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
_SIZE = {"bf16": 2, "f32": 4}


def _case(name, kind, M, N, K, bits, g, dtype="bf16", out="bf16", trust=1.0, packed=False):
    return {"name": name, "kind": kind, "M": M, "N": N, "K": K, "bits": bits, "g": g, "dtype": dtype, "out": out,
            "trust": trust, "packed": packed}


def listed():
    return [
        # one token of one sequence through an attention projection of the 1.6B-scale model (hidden size 2048):
        # the smallest call there is, repeated for every layer and token of a generation
        _case("decode_one_token", "infer", 1, 2048, 2048, 4, 128),
        # one step of 24 sequences through the gate or up projection of the MLP (width 5504) in a server that keeps
        # the weights packed and shares one workspace between layers
        _case("decode_batch_packed", "infer", 24, 5504, 2048, 4, 128, packed=True),
        # a prompt of odd length through the down projection of the MLP
        _case("prefill_ragged", "infer", 777, 2048, 5504, 4, 128),
        # single layer in binary32, rotation over the whole row (the small reference configuration)
        _case("forward_f32_small", "forward", 256, 512, 512, 4, 512, dtype="f32", out="f32"),
        # 1-bit weights and activations at 1.6B scale, the trust factor that the paper uses for one bit
        _case("forward_w1a1", "forward", 4096, 2048, 2048, 1, 128, trust=1.3),
        # the headline layer, trained: forward and backward
        _case("train_block128", "train", 4096, 2048, 2048, 4, 128, out="f32"),
        # the same with the full-width rotation, a batch with a ragged last sequence, gradients in bfloat16
        _case("train_full_rotation", "train", 4088, 2048, 2048, 4, 2048),
        # the MLP block of the 1.6B-scale model over a batch of 8192 tokens
        _case("mlp_forward", "mlp", 8192, 5504, 2048, 4, 128),
        # the FP4 grid at 1.6B scale
        _case("forward_fp4", "fp4", 4096, 2048, 2048, 4, 128),
        # weight-only quantization at 1.6B scale
        _case("weight_only", "weight_only", 4096, 2048, 2048, 4, 128),
        # two packed 8-bit tensors, the largest point of the shape sweep
        _case("gemm_codes_w8a8", "gemm", 16384, 4096, 4096, 8, 128),
        # the quantizer alone with the full-width rotation, the largest point of the shape sweep
        _case("quantize_full_rotation", "quantize", 16384, 0, 4096, 3, 4096),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _multiple(rng, lo, hi, step):
    return max(lo, min(hi, int(round(_log_uniform(rng, lo, hi) / step)) * step))


def _largest_block(K):
    g = K & -K
    return min(g, 4096)


def draw(rng):
    kind = rng.choice(["infer", "infer", "infer", "forward", "forward", "train", "train", "mlp", "fp4", "weight_only",
                       "gemm", "quantize"])
    while True:
        # widths: hidden sizes from 512 to 4096 and MLP widths up to 5504, multiples of 128 as models have them, now
        # and then a multiple of 32 only (1376 = 43 x 32)
        K = _multiple(rng, 512, 5504, 128 if rng.random() < 0.85 else 32)
        N = _multiple(rng, 512, 5504, 128 if rng.random() < 0.7 else 8)
        if kind == "infer":
            M = int(_log_uniform(rng, 1, 4096))
        elif kind in ("train", "mlp"):
            M = _multiple(rng, 256, 8192, 8)
        else:
            M = int(_log_uniform(rng, 64, 16384))
        bits = rng.choice([1, 2, 3, 4, 4, 4, 8])
        widest = _largest_block(K)
        g = rng.choice([min(128, widest)] * 3 + [widest, min(64, widest)])
        dtype = "bf16"
        if kind in ("forward", "quantize", "fp4", "weight_only"):
            dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
        out = rng.choice(["bf16", "bf16", "f32"])
        trust = 1.3 if bits == 1 else 1.0
        if kind == "fp4":
            bits = 4
            trust = 1.0
        if kind == "mlp":
            N = _multiple(rng, 512, 5504, 128)
            K = _multiple(rng, 512, 2048, 128)
            g = min(128, _largest_block(K), _largest_block(N))
            out = "bf16"
        if kind == "quantize":
            N = 0
        case = {"kind": kind, "M": M, "N": N, "K": K, "bits": bits, "g": g, "dtype": dtype, "out": out,
                "trust": trust, "packed": kind == "infer" and rng.random() < 0.4}
        w = work(case)
        # no more than the largest listed case: 275 x 2 G multiply-adds on the low-bit paths, 103 x 2 G on the 16-bit ones
        top = 103e9 if kind in ("train", "weight_only") else 550e9
        if w["flops"] <= top and w["bytes"] <= 350e6:
            return case


# ---- inputs ------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _activations(rows, cols, gen, dtype):
    """Student-t with four degrees of freedom, as hidden activations of a trained transformer are heavy-tailed."""
    chi = torch.zeros((rows, cols), device="cuda")
    for _ in range(4):
        chi += torch.randn((rows, cols), generator=gen, device="cuda").square_()
    return torch.randn((rows, cols), generator=gen, device="cuda").mul_(2.0).div_(chi.sqrt_()).to(dtype)


def _weights(rows, cols, gen, dtype):
    return torch.randn((rows, cols), generator=gen, device="cuda").mul_(0.02).to(dtype)


def prepare(case, seed):
    gen = _gen(seed)
    kind, M, N, K, bits, g = (case[k] for k in ("kind", "M", "N", "K", "bits", "g"))
    dt, out = _DTYPES[case["dtype"]], _DTYPES[case["out"]]
    s = {"case": case, "x": _activations(M, K, gen, dt)}
    if kind == "infer":
        # model load: the weights are quantized once, every buffer of the layer is allocated once
        w = _weights(N, K, gen, dt)
        ws = quest.alloc_workspace(M, N, K, bits, bits)
        load = quest.quest_linear_fwd(s["x"], w, bits, g, case["trust"], out_dtype=out, workspace=ws, want_masks=False)
        s["w_cached"] = {"wq": load["wq"], "sw": load["sw"], "operand_in_workspace": not case["packed"]}
        s["saved"] = {"xq": load["xq"], "sx": load["sx"]}
        s["y"], s["workspace"] = load["y"], ws
    elif kind == "forward":
        s["w"] = _weights(N, K, gen, dt)
    elif kind == "train":
        s["w"] = _weights(N, K, gen, dt)
        s["dy"] = torch.randn((M, N), generator=gen, device="cuda").mul_(1e-3).to(torch.bfloat16)
        s["ws_fwd"] = quest.alloc_workspace(M, N, K, bits, bits)
        s["ws_bwd"] = torch.empty(quest.quest_bwd_workspace_bytes(M, N, K), dtype=torch.uint8, device="cuda")
    elif kind == "mlp":
        s["w_gate"], s["w_up"] = _weights(N, K, gen, dt), _weights(N, K, gen, dt)
        s["w_down"] = _weights(K, N, gen, dt)
        s["buffers"] = quest.mlp_buffers(M, K, N, bits, out_dtype=out)
    elif kind == "fp4":
        s["w"] = _weights(N, K, gen, dt)
    elif kind == "weight_only":
        s["w"] = _weights(N, K, gen, dt)
        s["workspace"] = torch.empty(quest.quest_weight_only_workspace_bytes(M, N, K), dtype=torch.uint8, device="cuda")
    elif kind == "gemm":
        s["xq"], s["sx"], _ = quest.quest_quantize(s.pop("x"), bits, g, case["trust"], want_mask=False)
        s["wq"], s["sw"], _ = quest.quest_quantize(_weights(N, K, gen, dt), bits, g, case["trust"], want_mask=False)
        s["workspace"] = quest.alloc_workspace(M, N, K, bits, bits)
    return s


def run(state):
    case = state["case"]
    kind, bits, g, trust, K = case["kind"], case["bits"], case["g"], case["trust"], case["K"]
    out = _DTYPES[case["out"]]
    if kind == "infer":
        r = quest.quest_linear_fwd(state["x"], None, bits, g, trust, y=state["y"], saved=state["saved"],
                                   w_cached=state["w_cached"], workspace=state["workspace"], want_masks=False)
        return {"y": r["y"], "xq": r["xq"], "sx": r["sx"]}
    if kind == "forward":
        return quest.quest_linear_fwd(state["x"], state["w"], bits, g, trust, out_dtype=out)
    if kind == "train":
        r = quest.quest_linear_fwd(state["x"], state["w"], bits, g, trust, workspace=state["ws_fwd"])
        d = quest.quest_linear_bwd(state["dy"], r, bits, g, K, out_dtype=out, workspace=state["ws_bwd"])
        return {**r, **d}
    if kind == "mlp":
        b = quest.quest_mlp_fwd(state["x"], state["w_gate"], state["w_up"], state["w_down"], bits, g, trust,
                                buffers=state["buffers"])
        return {k: v for k, v in b.items() if k not in ("workspace", "launches")}
    if kind == "fp4":
        return quest.quest_linear_fwd_fp4(state["x"], state["w"], g, trust, out_dtype=out)
    if kind == "weight_only":
        return quest.quest_linear_fwd_weight_only(state["x"], state["w"], bits, g, trust, out_dtype=out,
                                                  workspace=state["workspace"])
    if kind == "gemm":
        y, _ = quest.quest_lowbit_gemm(state["xq"], state["sx"], bits, state["wq"], state["sw"], bits, K, out_dtype=out,
                                       workspace=state["workspace"])
        return y
    codes, scales, mask = quest.quest_quantize(state["x"], bits, g, trust)
    return {"codes": codes, "scales": scales, "mask": mask}


# ---- what a pass cannot do without ---------------------------------------------------------------------

def _quantized(rows, cols, bits, masks=True):
    """Bytes of the codes, scales and mask of one tensor."""
    return rows * cols * quest.container_bits(bits) / 8 + rows * 4 + (rows * cols / 8 if masks else 0)


def work(case):
    kind, M, N, K, bits = (case[k] for k in ("kind", "M", "N", "K", "bits"))
    e, o = _SIZE[case["dtype"]], _SIZE[case["out"]]
    flops = 2.0 * M * N * K
    if kind == "infer":
        nbytes = M * K * e + _quantized(M, K, bits, False) + _quantized(N, K, bits, False) + M * N * o
    elif kind in ("forward", "fp4"):
        nbytes = (M + N) * K * e + _quantized(M, K, bits) + _quantized(N, K, bits) + M * N * o
    elif kind == "train":
        nbytes = (M + N) * K * e + _quantized(M, K, bits) + _quantized(N, K, bits) + M * N * e   # y has the type of x
        nbytes += M * N * 2 + (M + N) * K * o
        flops *= 3
    elif kind == "mlp":
        nbytes = M * K * e + 3 * N * K * e + _quantized(M, K, bits) + 2 * _quantized(N, K, bits)
        nbytes += M * N * 2 + _quantized(M, N, bits) + _quantized(K, N, bits) + M * K * o
        flops *= 3
    elif kind == "weight_only":
        nbytes = (M + N) * K * e + M * K * 2 + _quantized(N, K, bits) + M * N * o
    elif kind == "gemm":
        nbytes = _quantized(M, K, bits, False) + _quantized(N, K, bits, False) + M * N * o
    else:
        nbytes = M * K * e + _quantized(M, K, bits)
        flops = float(M * K * (math.log2(case["g"]) + 8))
    return {"bytes": float(nbytes), "flops": flops}


def tolerance(case):
    """About four times the error that each path shows against the same path in binary64 from its own codes."""
    kind, f32 = case["kind"], case["out"] == "f32"
    if kind == "train":
        # the backward products have one operand rounded to bfloat16 (1.6e-3 of the norm), the gradients may be too
        return {"rel": 7e-3 if f32 else 1e-2}
    if kind == "mlp":
        # h is rounded to bfloat16 after an exponential that two implementations evaluate in different ways (one
        # element in a thousand moves by a unit); a code of h next to a rounding boundary can move with it
        return {"rel": 7e-3, "differ": 1e-5}
    if kind == "weight_only":
        # xh is rounded once from exact sums of fixed order; y sums in an order that the hardware chooses
        return {"rel": 1e-6 if f32 else 7e-3}
    if kind == "quantize":
        return {"rel": 4e-7}
    # whole numbers are exact, y is a scale product away from an exact integer: the output type decides
    return {"rel": 4e-7 if f32 else 7e-3}


# ---- the same outputs in binary64 ----------------------------------------------------------------------

# alpha*(b) of the uniform grids and of the FP4 grid (minimisers of the Gaussian quantization error)
_ALPHA = {1: 0.7978846, 2: 1.4935300, 3: 2.0510680, 4: 2.5140045, 5: 2.9161513, 6: 3.2779846, 7: 3.6110970, 8: 3.9222038}
_ALPHA_FP4 = 2.9224751
_E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


def _rotated(t, g):
    """Orthonormal Walsh-Hadamard transform of every block of g consecutive elements of a row (its own inverse)."""
    v = t.double().reshape(t.shape[0], -1, g)
    h = 1
    while h < g:
        v = v.reshape(t.shape[0], -1, g // (2 * h), 2, h)
        v = torch.stack((v[..., 0, :] + v[..., 1, :], v[..., 0, :] - v[..., 1, :]), dim=-2)
        h *= 2
    return (v / math.sqrt(g)).reshape(t.shape[0], -1)


def _projected(t, bits, g, trust):
    """(grid values 2k - (2^b - 1), row scales, trusted elements)."""
    u = _rotated(t, g)
    top = 2.0 ** bits - 1.0
    alpha = _ALPHA[bits]
    rms = u.square().mean(1).sqrt()
    pos = u * (top / (2.0 * alpha)) / rms.clamp_min(1e-300)[:, None] + top / 2.0
    k = pos.clamp(0.0, top).round()
    return 2.0 * k - top, alpha * rms / top, (pos - k).abs() <= trust / 2.0


def _projected_fp4(t, g):
    u = _rotated(t, g)
    rms = u.square().mean(1).sqrt()
    pos = u * (6.0 / _ALPHA_FP4) / rms.clamp_min(1e-300)[:, None]
    mag = pos.abs().clamp_max(6.0)
    step = torch.where(mag < 2.0, 0.5, torch.where(mag < 4.0, 1.0, 2.0))
    return torch.sign(pos) * (mag / step).round() * step, _ALPHA_FP4 * rms / 6.0


def exact(case, seed):
    """What ``run`` returns, in binary64 from the definition; codes and masks are whole numbers and have no such value."""
    gen = _gen(seed)
    kind, M, N, K, bits, g, trust = (case[k] for k in ("kind", "M", "N", "K", "bits", "g", "trust"))
    dt = _DTYPES[case["dtype"]]
    x = _activations(M, K, gen, dt)
    if kind == "quantize":
        return {"codes": None, "scales": _projected(x, bits, g, trust)[1], "mask": None}
    if kind == "mlp":
        wg, wu = _weights(N, K, gen, dt), _weights(N, K, gen, dt)
        wd = _weights(K, N, gen, dt)
        qx, sx, _ = _projected(x, bits, g, trust)
        qg, sg, _ = _projected(wg, bits, g, trust)
        qu, su, _ = _projected(wu, bits, g, trust)
        gate = (qx @ qg.T) * sx[:, None] * sg
        h = (gate / (1.0 + torch.exp(-gate)) * ((qx @ qu.T) * sx[:, None] * su)).to(torch.bfloat16)   # h is a bfloat16 tensor
        qh, sh, _ = _projected(h, bits, g, trust)
        qd, sd, _ = _projected(wd, bits, g, trust)
        out = dict.fromkeys(("xq", "mx", "wgq", "mwg", "wuq", "mwu", "hq", "mh", "wdq", "mwd"))
        return {**out, "h": h.double(), "y": (qh @ qd.T) * sh[:, None] * sd, "sx": sx, "swg": sg, "swu": su, "sh": sh, "swd": sd}
    w = _weights(N, K, gen, dt)
    if kind == "weight_only":
        xh = _rotated(x, g)
        qw, sw, _ = _projected(w, bits, g, trust)
        return {"y": (xh @ qw.T) * sw, "xh": xh, "wq": None, "sw": sw, "mw": None}
    if kind == "fp4":
        (qx, sx), (qw, sw) = _projected_fp4(x, g), _projected_fp4(w, g)
    else:
        (qx, sx, mx), (qw, sw, mw) = _projected(x, bits, g, trust), _projected(w, bits, g, trust)
    y = (qx @ qw.T) * sx[:, None] * sw
    if kind == "gemm":
        return y
    if kind == "infer":
        return {"y": y, "xq": None, "sx": sx}
    out = {"xq": None, "sx": sx, "mx": None, "wq": None, "sw": sw, "mw": None, "y": y}
    if kind == "train":
        dy = torch.randn((M, N), generator=gen, device="cuda").mul_(1e-3).to(torch.bfloat16).double()
        out["dx"] = _rotated((dy @ (qw * sw[:, None])) * mx, g)
        out["dw"] = _rotated((dy.T @ (qx * sx[:, None])) * mw, g)
    return out

"""Measured workloads: the calls that training and inference programs make of this library, over the sizes they use.

Each case names a kind of pass and its sizes.  The kinds:

  train_block   one step of a transformer block's FP8 linears and its penalty (``workload.BlockStep``): per-tensor casts of
                X, W and dY, the three products of every linear, the TWEO loss and gradient on the block output(s).
                "plain" takes each tensor's current amax as its scale; "fused" is the delayed-scaling recipe with the amax
                and the FP8 copies of the outputs from the epilogue.
  train_linear  one linear and its penalty called directly: cast, forward, backward, loss; the weight gradient in bf16, or
                added into a binary32 buffer over micro-batches.
  block_fwd     the MLP half of a block's training forward with given (delayed) scales: norm -> FP8, linear + activation
                -> FP8, linear -> bf16, residual addition with the penalty, its gradient and the next block's FP8 copy.
  w8a8          the static per-tensor W8A8 inference linear on bf16 activations.
  int8_token    the 8-bit residual stream with per-token activation scales and per-channel weight scales: quantise the
                activations, integer linear, quantise its output, add it to the quantised residual.
  w4            the few-token inference linear on packed 4-bit weights, including the cast of its activations.

Inputs are drawn on the GPU from the seed with the distributions of the benchmark's recipe: N(0,1) activations (with the
configuration's outliers), N(0, 0.02) weights, N(0, 1e-3) gradients.
"""
import math

import torch

from paper_2511_23225_b200 import binding as tw
from paper_2511_23225_b200 import synth
from paper_2511_23225_b200.workload import BlockStep

ACTS = {"gelu": tw.ACT_GELU, "gelu_tanh": tw.ACT_GELU_TANH, "swiglu": tw.ACT_SWIGLU}


def listed():
    return [
        # the small linear with extreme outliers, 512 tokens: launches and latency
        {"name": "train_linear_small", "kind": "train_linear", "M": 512, "K": 256, "N": 1024, "dw": "bf16"},
        # GPT-2-small-shaped block, 8 x 1024 tokens, current scaling
        {"name": "train_gpt2_small_block", "kind": "train_block", "cfg": 2, "M": 8192, "variant": "plain"},
        # ViT-B/16-shaped step with all twelve block outputs, 61 images of 197 tokens: the last, smaller batch of an epoch
        {"name": "train_vit_b16_ragged", "kind": "train_block", "cfg": 3, "M": 61 * 197, "variant": "plain"},
        # LLaMA-1B-shaped block, 4 x 4096 tokens, delayed scaling and fused epilogues: the benchmark's step
        {"name": "train_llama_1b_block", "kind": "train_block", "cfg": 4, "M": 16384, "variant": "fused"},
        # MLP half of a ViT-B/16 block's forward, 64 images: GELU (erf form) between two linears
        {"name": "block_fwd_vit_mlp", "kind": "block_fwd", "M": 64 * 197, "d": 768, "ff": 3072, "act": "gelu", "norm": "layer"},
        # decode of one sequence: one token, the up projection of a LLaMA-7B-shaped MLP
        {"name": "w8a8_decode_1", "kind": "w8a8", "M": 1, "K": 4096, "N": 11008},
        # a short prompt, or a large decode batch: a few hundred tokens, an odd count, the attention projections
        {"name": "w8a8_batch_300", "kind": "w8a8", "M": 300, "K": 4096, "N": 4096},
        # prefill of one prompt: 1024 tokens, the down projection
        {"name": "w8a8_prefill_1024", "kind": "w8a8", "M": 1024, "K": 11008, "N": 4096},
        # prefill of a batch of prompts
        {"name": "w8a8_prefill_8192", "kind": "w8a8", "M": 8192, "K": 4096, "N": 11008},
        # a decode batch of 16 sequences on the per-token 8-bit stream
        {"name": "int8_token_decode_16", "kind": "int8_token", "M": 16, "K": 4096, "N": 4096},
        # prefill on the same stream, a prompt of odd length
        {"name": "int8_token_prefill_1999", "kind": "int8_token", "M": 1999, "K": 4096, "N": 4096},
        # decode of 8 sequences with packed 4-bit weights
        {"name": "w4_decode_8", "kind": "w4", "M": 8, "K": 11008, "N": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi, step=16):
    """A layer width: mostly a multiple of 128 as models have them, else any multiple of `step`."""
    s = 128 if rng.random() < 0.6 else step
    return max(lo, min(hi, _log_int(rng, lo, hi) // s * s))


def draw(rng):
    kind = rng.choice(["train_block", "train_linear", "block_fwd", "w8a8", "w8a8", "int8_token", "w4"])
    if kind == "train_block":
        cfg = rng.randint(1, 4)
        top = {1: 8192, 2: 32768, 3: 50432, 4: 16384}[cfg]
        return {"kind": kind, "cfg": cfg, "M": _log_int(rng, 200, top), "variant": rng.choice(["plain", "fused"])}
    if kind == "train_linear":
        return {"kind": kind, "M": _log_int(rng, 64, 16384), "K": _width(rng, 256, 6144), "N": _width(rng, 256, 6144),
                "dw": rng.choice(["bf16", "f32_accumulate"])}
    if kind == "block_fwd":
        d = _width(rng, 256, 4096, 64)
        act = rng.choice(sorted(ACTS))
        ff = int(d * (2.75 if act == "swiglu" else 4)) // 64 * 64
        return {"kind": kind, "M": _log_int(rng, 200, 16384 if d <= 2048 else 8192), "d": d, "ff": ff, "act": act,
                "norm": "rms" if act == "swiglu" else "layer"}
    if kind == "w8a8":
        return {"kind": kind, "M": _log_int(rng, 1, 8192), "K": _width(rng, 1024, 11008), "N": _width(rng, 1024, 11008)}
    if kind == "int8_token":
        return {"kind": kind, "M": _log_int(rng, 1, 8192), "K": _width(rng, 768, 8192), "N": _width(rng, 768, 8192)}
    return {"kind": "w4", "M": _log_int(rng, 1, 128), "K": _width(rng, 1024, 11008, 128), "N": _width(rng, 1024, 11008)}


# ------------------------------------------------------------------------------------------------ inputs

def _normal(gen, shape, std=1.0):
    return (torch.randn(shape, device="cuda", generator=gen) * std).to(torch.bfloat16)


def _activation(gen, shape, kind="normal"):
    x = torch.randn(shape, device="cuda", generator=gen)
    if kind == "student_t":            # + t with three degrees of freedom: N / sqrt(chi2_3 / 3)
        chi = sum(torch.randn(shape, device="cuda", generator=gen).square_() for _ in range(3))
        x = x + torch.randn(shape, device="cuda", generator=gen) * (chi / 3).rsqrt_()
    elif kind == "outlier_channels":   # one channel of ten thousand, at least one, times 500
        k = max(1, round(1e-4 * shape[-1]))
        x[:, torch.randperm(shape[-1], device="cuda", generator=gen)[:k]] *= 500.0
    elif kind == "outlier_entries":    # one entry of a thousand at +-U(1000, 3000)
        at = torch.rand(shape, device="cuda", generator=gen) < 1e-3
        big = 1000.0 + 2000.0 * torch.rand(shape, device="cuda", generator=gen)
        x = torch.where(at, torch.copysign(big, x), x)
    return x.to(torch.bfloat16)


def _scale(amax, top=448.0):
    """A given scale, as calibration or an amax history leaves it."""
    return torch.full((1,), top / amax, dtype=torch.float32, device="cuda")


def _empty(*shape, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda")


# ------------------------------------------------------------------------------------------------ the kinds

def _inputs_train_block(c, gen):
    """X, W and dY of every linear, then the block outputs, in the order of the step's buffers."""
    cfg, M = synth.CONFIGS[c["cfg"]], c["M"]
    for l in cfg.linears:
        yield _activation(gen, (M, l.K), cfg.x_kind)
        yield _normal(gen, (l.N, l.K), 0.02)
        yield _normal(gen, (M, l.N), 1e-3)
    for _ in range(cfg.n_blocks):
        yield _activation(gen, (M, cfg.d), cfg.x_kind)


def _prepare_train_block(c, gen):
    b = BlockStep(c["cfg"], M=c["M"], variant=c["variant"])
    for t, v in zip([t for lb in b.linears for t in (lb.x, lb.w, lb.dy)] + b.a, _inputs_train_block(c, gen)):
        t.copy_(v)
    if c["variant"] == "fused":        # the amax histories of a step that has run before
        b.step()
        b.step()
    return b


def _run_train_block(b):
    b.step()
    out = {"loss": b.loss, "loss_per_block": b.loss_per_block, "grad": b.ga,
           "linears": [(lb.y, lb.dx, lb.dw) for lb in b.linears]}
    if b.variant == "fused":
        out["copies"] = [(lb.yq, lb.dxq) for lb in b.linears]
        out["scales"] = (b.scale_e, b.scale_g, b.hist_e, b.hist_g)
    return out


def _work_train_block(c):
    cfg, M = synth.CONFIGS[c["cfg"]], c["M"]
    byt = 4 * M * cfg.d * cfg.n_blocks
    for l in cfg.linears:
        byt += 4 * (M * l.K + l.N * l.K + M * l.N)
        if c["variant"] == "fused":
            byt += M * l.K + M * l.N
    return {"bytes": byt, "flops": sum(6 * M * l.K * l.N for l in cfg.linears)}


def _inputs_train_linear(c, gen):
    M, K, N = c["M"], c["K"], c["N"]
    return {"x": _activation(gen, (M, K), "outlier_entries"), "w": _normal(gen, (N, K), 0.02), "dy": _normal(gen, (M, N), 1e-3),
            "a": _activation(gen, (M, K), "outlier_entries")}


def _prepare_train_linear(c, gen):
    M, K, N = c["M"], c["K"], c["N"]
    s = {**_inputs_train_linear(c, gen), "y": _empty(M, N), "dx": _empty(M, K), "g": [_empty(M, K)],
         "f32": c["dw"] != "bf16"}
    s["dw"] = torch.zeros((N, K), dtype=torch.float32 if s["f32"] else torch.bfloat16, device="cuda")
    sc = torch.ones(9, dtype=torch.float32, device="cuda")
    s["q"] = [tw.Quantized(_empty(*t.shape, dtype=torch.uint8), sc[3 * i:3 * i + 1], sc[3 * i + 1:3 * i + 2], sc[3 * i + 2:3 * i + 3],
                           None, f) for i, (t, f) in enumerate(((s["x"], tw.E4M3), (s["w"], tw.E4M3), (s["dy"], tw.E5M2)))]
    s["ws_q"], s["ws"] = tw.new_workspace(tw.OP_QUANTIZE), tw.new_workspace(tw.OP_LINEAR_WGRAD)
    s["ws_loss"] = tw.new_workspace(tw.OP_LOSS, M * K, 1)
    return s


def _run_train_linear(s):
    qx, qw, qd = s["q"]
    tw.quantize_per_tensor_batch([s["x"], s["w"], s["dy"]], s["q"], ws=s["ws_q"])
    tw.fp8_linear_fwd(qx.q, qw.q, qx.scale_inv, qw.scale_inv, y=s["y"], ws=s["ws"])
    if s["f32"]:
        tw.fp8_linear_bwd_dgrad(qd.q, qw.q, qd.scale_inv, qw.scale_inv, dx=s["dx"], ws=s["ws"])
        tw.fp8_linear_bwd_wgrad(qx.q, qd.q, qx.scale_inv, qd.scale_inv, dw=s["dw"], dw_dtype=tw.F32, accumulate=True, ws=s["ws"])
    else:
        tw.fp8_linear_bwd(qd.q, qx.q, qw.q, qd.scale_inv, qx.scale_inv, qw.scale_inv, dx=s["dx"], dw=s["dw"], ws=s["ws"])
    loss, _, g = tw.loss_fwd_bwd([s["a"]], 3.0, 1e-6, 4.0, 0.01, grads=s["g"], ws=s["ws_loss"], per_block=False)
    return {"y": s["y"], "dx": s["dx"], "dw": s["dw"], "loss": loss, "grad": g[0],
            "amax": [q.amax for q in s["q"]], "codes": [q.q for q in s["q"]]}


def _work_train_linear(c):
    M, K, N = c["M"], c["K"], c["N"]
    return {"bytes": 5 * (M * K + N * K + M * N) + 2 * (M * N + M * K) + (8 if c["dw"] != "bf16" else 2) * N * K + 4 * M * K,
            "flops": 6 * M * K * N}


def _inputs_block_fwd(c, gen):
    M, d, ff = c["M"], c["d"], c["ff"]
    rows = 2 * ff if c["act"] == "swiglu" else ff
    return {"x": _activation(gen, (M, d)), "gamma": 1.0 + 0.1 * torch.randn(d, device="cuda", generator=gen),
            "beta": None if c["norm"] == "rms" else 0.1 * torch.randn(d, device="cuda", generator=gen),
            "w1": _normal(gen, (rows, d), 0.02), "w2": _normal(gen, (d, ff), 0.02)}


def _prepare_block_fwd(c, gen):
    M, d, ff = c["M"], c["d"], c["ff"]
    i = _inputs_block_fwd(c, gen)
    s = {"x": i["x"], "gamma": i["gamma"], "beta": i["beta"],
         "norm": tw.NORM_RMS if c["norm"] == "rms" else tw.NORM_LAYER, "act": ACTS[c["act"]],
         "w1": tw.quantize_per_tensor(i["w1"]), "w2": tw.quantize_per_tensor(i["w2"]),
         "s_n": _scale(6.0), "s_h": _scale(4.0), "s_a": _scale(8.0), "amax_h": torch.zeros(1, device="cuda"),
         "nq": _empty(M, d, dtype=torch.uint8), "hq": _empty(M, ff, dtype=torch.uint8), "f": _empty(M, d), "a": _empty(M, d),
         "grad": _empty(M, d), "aq": _empty(M, d, dtype=torch.uint8), "ws": tw.new_workspace(tw.OP_LINEAR_FWD),
         "ws_b": tw.new_workspace(tw.OP_BLOCK_OUTPUT)}
    s["i_n"], s["i_h"] = 1.0 / s["s_n"], 1.0 / s["s_h"]
    return s


def _run_block_fwd(s):
    _, nq, amax_n, mean, rstd = tw.layernorm_fp8(s["x"], s["gamma"], s["beta"], 1e-5, s["norm"], want_y=False, q_fmt=tw.E4M3,
                                                 q_scale=s["s_n"], want_stats=True, yq=s["nq"])
    tw.fp8_linear_fwd_act(nq, s["w1"].q, s["i_n"], s["w1"].scale_inv, s["act"], want_y=False, out_amax=s["amax_h"], out_q=s["hq"],
                          q_scale=s["s_h"])
    tw.fp8_linear_fwd(s["hq"], s["w2"].q, s["i_h"], s["w2"].scale_inv, y=s["f"], ws=s["ws"])
    a, loss, amax_a, grad, aq = tw.block_output_fused(s["x"], s["f"], 3.0, 1e-6, 4.0, 0.01, q_fmt=tw.E4M3, q_scale=s["s_a"],
                                                      a=s["a"], grad=s["grad"], aq=s["aq"], ws=s["ws_b"])
    return {"normed": nq, "mean": mean, "rstd": rstd, "hidden": s["hq"], "f": s["f"], "a": a, "loss": loss, "grad": grad, "aq": aq,
            "amax": (amax_n, s["amax_h"], amax_a)}


def _work_block_fwd(c):
    M, d, ff = c["M"], c["d"], c["ff"]
    rows = 2 * ff if c["act"] == "swiglu" else ff
    # x; the two weights; normed, hidden, f, a, grad, aq
    return {"bytes": 2 * M * d + (rows + ff) * d + M * d + M * ff + 7 * M * d, "flops": 2 * M * d * (rows + ff)}


def _inputs_w8a8(c, gen):
    M, K, N = c["M"], c["K"], c["N"]
    w = _normal(gen, (N, K), 0.02)
    sx = _scale(float(_normal(gen, (1024, K)).abs().max()))   # calibration
    return _normal(gen, (M, K)), w, sx


def _prepare_w8a8(c, gen):
    M, K, N = c["M"], c["K"], c["N"]
    x, w, sx = _inputs_w8a8(c, gen)
    wq = tw.quantize_per_tensor(w)
    return {"x": x, "sx": sx, "w": wq.q, "sw_inv": wq.scale_inv, "y": _empty(M, N),
            "ws": tw.new_workspace(tw.OP_W8A8, M, N, K)}


def _run_w8a8(s):
    return tw.w8a8_static_gemm(s["x"], s["sx"], s["w"], s["sw_inv"], y=s["y"], ws=s["ws"])


def _work_w8a8(c):
    M, K, N = c["M"], c["K"], c["N"]
    return {"bytes": 2 * M * K + N * K + 2 * M * N, "flops": 2 * M * K * N}


def _inputs_int8_token(c, gen):
    M, K, N = c["M"], c["K"], c["N"]
    w, r = _normal(gen, (N, K), 0.02), _normal(gen, (M, N))
    return _normal(gen, (M, K)), w, r


def _prepare_int8_token(c, gen):
    M, K, N = c["M"], c["K"], c["N"]
    x, w, r = _inputs_int8_token(c, gen)
    wq, sw = tw.absmax_quantize(w, granularity=tw.GRAN_ROW)
    rq, rs = tw.absmax_quantize(r, granularity=tw.GRAN_ROW)
    return {"x": x, "wq": wq, "sw": sw, "rq": rq, "rs": rs, "y": _empty(M, N),
            "out": _empty(M, N, dtype=torch.int8)}


def _run_int8_token(s):
    xq, sx = tw.absmax_quantize(s["x"], granularity=tw.GRAN_ROW)
    f = tw.int8_linear(xq, sx, s["wq"], s["sw"], y=s["y"])
    fq, sf = tw.absmax_quantize(f, granularity=tw.GRAN_ROW)
    yq, sy = tw.residual_add_q8_rows(s["rq"], s["rs"], fq, sf, yq=s["out"])
    return {"xq": xq, "sx": sx, "f": f, "fq": fq, "sf": sf, "yq": yq, "sy": sy}


def _work_int8_token(c):
    M, K, N = c["M"], c["K"], c["N"]
    return {"bytes": 3 * M * K + N * K + 2 * M * N + 3 * M * N, "flops": 2 * M * K * N}


def _inputs_w4(c, gen):
    M, K, N = c["M"], c["K"], c["N"]
    w, x = _normal(gen, (N, K), 0.02), _normal(gen, (M, K))
    return x, w, _scale(float(_normal(gen, (1024, K)).abs().max()))


def _prepare_w4(c, gen):
    M, K, N = c["M"], c["K"], c["N"]
    x, w, sx = _inputs_w4(c, gen)
    w = tw.fp4_quantize(w, carriers=False)
    sc = torch.empty(2, dtype=torch.float32, device="cuda")
    return {"x": x, "sx": sx, "w4": w.q4.view(N, K // 2), "sw_inv": w.scale_inv, "y": _empty(M, N),
            "q": tw.Quantized(_empty(M, K, dtype=torch.uint8), sx, sc[0:1], sc[1:2], None, tw.E4M3)}


def _run_w4(s):
    q = tw.quantize_per_tensor(s["x"], tw.E4M3, tw.SCALE_GIVEN, out=s["q"])
    return tw.fp4_weight_linear(q.q, q.scale_inv, s["w4"], s["sw_inv"], y=s["y"])


def _work_w4(c):
    M, K, N = c["M"], c["K"], c["N"]
    return {"bytes": 2 * M * K + N * K // 2 + 2 * M * N, "flops": 2 * M * K * N}


# ------------------------------------------------------------------------------------------------ 64-bit results

# The codes, the scales and the roundings to bf16 that a later operation reads are part of what a pass is defined to do
# (a binary32 multiplication by the scale, one rounding); everything between them is taken in binary64.  Codes have no
# value of their own here: None.

_GRID = {tw.E4M3: (448.0, torch.float8_e4m3fn), tw.E5M2: (57344.0, torch.float8_e5m2)}


def _bf16(x):
    return x.to(torch.bfloat16)


def _over(top, x):
    """top / x in binary32, rounded once (a Python number over a tensor is a reciprocal and a product)."""
    return torch.full_like(x, top) / x


def _fp8(x, fmt=tw.E4M3, scale=None):
    """The dequantised FP8 values of a bf16 tensor, and its largest magnitude; `scale`: given, else the current one."""
    top, dtype = _GRID[fmt]
    amax = x.abs().max().float().view(1)
    scale = _over(top, amax) if scale is None else scale
    q = (x.float() * scale).clamp_(-top, top).to(dtype)
    return q.double() * _over(1.0, scale).double(), amax


def _absmax_rows(x):
    """Codes and scales of Eq. 4 with one scale per row; x in binary32 or bf16."""
    s = x.abs().amax(dim=1).float() + 1e-6
    return (x.float() * _over(127.0, s)[:, None]).round_().clamp_(-127, 127).double(), s


def _penalty(a, c, tau=3.0, eps=1e-6, p=4.0):
    a, d = a.double(), tau + eps
    return (a.abs() / d).pow(p).mean().view(1), c * p * a.sign() * a.abs().pow(p - 1) / (a.numel() * d ** p)


def _exact_train_block(c, gen):
    cfg = synth.CONFIGS[c["cfg"]]
    inputs, L = list(_inputs_train_block(c, gen)), cfg.n_blocks
    linears, amax_e, amax_g, n = [], [], [], len(cfg.linears)
    for i in range(n):
        x, w, dy = inputs[3 * i:3 * i + 3]
        (xv, ax), (wv, aw), (dv, ad) = _fp8(x), _fp8(w), _fp8(dy, tw.E5M2)
        y, dx, dw = xv @ wv.T, dv @ wv, dv.T @ xv
        linears.append((y, dx, dw))
        if c["variant"] == "fused":   # of the step before the first scales were known, and of every later one
            one = x.new_ones(1, dtype=torch.float32)
            x1, w1, d1 = _fp8(x, tw.E4M3, one)[0], _fp8(w, tw.E4M3, one)[0], _fp8(dy, tw.E5M2, one)[0]
            y1, dx1 = (float(_bf16(t).abs().max()) for t in (x1 @ w1.T, d1 @ w1))
            amax_e.append([(float(ax),) * 3, (float(aw),) * 3, (float(_bf16(y).abs().max()),) * 2 + (y1,)])
            amax_g.append([(float(ad),) * 3, (float(_bf16(dx).abs().max()),) * 2 + (dx1,)])
    terms = [_penalty(a, 0.01 / L) for a in inputs[3 * n:]]
    per_block = torch.cat([t[0] for t in terms])
    out = {"loss": per_block.mean().view(1), "loss_per_block": per_block, "grad": [t[1] for t in terms], "linears": linears}
    if c["variant"] == "fused":
        groups = []
        for amax, fmt in ((amax_e, tw.E4M3), (amax_g, tw.E5M2)):
            hist = torch.tensor([linear[k] for k in range(len(amax[0])) for linear in amax], dtype=torch.float64, device="cuda")
            groups.append((_GRID[fmt][0] / hist.amax(dim=1), torch.cat([hist, hist.new_zeros(len(hist), 13)], dim=1)))
        out["scales"] = (groups[0][0], groups[1][0], groups[0][1], groups[1][1])
    return out


def _exact_train_linear(c, gen):
    i = _inputs_train_linear(c, gen)
    (xv, ax), (wv, aw), (dv, ad) = _fp8(i["x"]), _fp8(i["w"]), _fp8(i["dy"], tw.E5M2)
    loss, grad = _penalty(i["a"], 0.01)
    return {"y": xv @ wv.T, "dx": dv @ wv, "dw": dv.T @ xv, "loss": loss, "grad": grad, "amax": [ax, aw, ad], "codes": None}


def _exact_block_fwd(c, gen):
    i = _inputs_block_fwd(c, gen)
    x = i["x"].double()
    mean = x.mean(dim=1, keepdim=True) if c["norm"] == "layer" else torch.zeros_like(x[:, :1])
    rstd = ((x - mean).square().mean(dim=1, keepdim=True) + 1e-5).rsqrt()
    n = (x - mean) * rstd * i["gamma"].double() + (0.0 if i["beta"] is None else i["beta"].double())
    nv, amax_n = _fp8(_bf16(n), tw.E4M3, _scale(6.0))
    h = nv @ _fp8(i["w1"])[0].T
    if c["act"] == "swiglu":
        h = torch.nn.functional.silu(h[:, :c["ff"]]) * h[:, c["ff"]:]
    else:
        h = torch.nn.functional.gelu(h, approximate="none" if c["act"] == "gelu" else "tanh")
    hv, amax_h = _fp8(_bf16(h), tw.E4M3, _scale(4.0))
    f = hv @ _fp8(i["w2"])[0].T
    a = x + _bf16(f).double()
    loss, grad = _penalty(_bf16(a), 0.01)
    return {"normed": None, "mean": mean.view(-1), "rstd": rstd.view(-1), "hidden": None, "f": f, "a": a, "loss": loss,
            "grad": grad, "aq": None, "amax": (amax_n, amax_h, _bf16(a).abs().max().view(1))}


def _exact_w8a8(c, gen):
    x, w, sx = _inputs_w8a8(c, gen)
    return _fp8(x, tw.E4M3, sx)[0] @ _fp8(w)[0].T


def _exact_int8_token(c, gen):
    x, w, r = _inputs_int8_token(c, gen)
    (xq, sx), (wq, sw), (rq, sr) = _absmax_rows(x), _absmax_rows(w), _absmax_rows(r)
    f = (xq @ wq.T) * (sx.double()[:, None] / 127) * (sw.double() / 127)
    fq, sf = _absmax_rows(_bf16(f))
    y = fq * (sf.double()[:, None] / 127) + rq * (sr.double()[:, None] / 127)
    return {"xq": None, "sx": x.double().abs().amax(dim=1) + 1e-6, "f": f, "fq": None,
            "sf": _bf16(f).double().abs().amax(dim=1) + 1e-6, "yq": None, "sy": y.abs().amax(dim=1) + 1e-6}


def _exact_w4(c, gen):
    x, w, sx = _inputs_w4(c, gen)
    s = _over(6.0, w.abs().max().float())
    v = (w.float() * s).clamp_(-6.0, 6.0)
    step = torch.where(v.abs() < 2, 0.5, torch.where(v.abs() < 4, 1.0, 2.0))   # E2M1: 0 0.5 1 1.5 2 3 4 6
    return _fp8(x, tw.E4M3, sx)[0] @ (((v / step).round_() * step).double() * _over(1.0, s).double()).T


_KINDS = {"train_block": (_prepare_train_block, _run_train_block, _work_train_block, _exact_train_block),
          "train_linear": (_prepare_train_linear, _run_train_linear, _work_train_linear, _exact_train_linear),
          "block_fwd": (_prepare_block_fwd, _run_block_fwd, _work_block_fwd, _exact_block_fwd),
          "w8a8": (_prepare_w8a8, _run_w8a8, _work_w8a8, _exact_w8a8),
          "int8_token": (_prepare_int8_token, _run_int8_token, _work_int8_token, _exact_int8_token),
          "w4": (_prepare_w4, _run_w4, _work_w4, _exact_w4)}


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    return case["kind"], _KINDS[case["kind"]][0](case, gen)


def run(state):
    return _KINDS[state[0]][1](state[1])


def work(case):
    return _KINDS[case["kind"]][2](case)


def exact(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    return _KINDS[case["kind"]][3](case, gen)


def tolerance(case):
    """Four times what the same passes show with their sums in another order (contractions permuted, or taken in
    binary64): bf16 results then differ by at most one rounding (2^-7 of a value) in up to 4 values of ten thousand, a
    2-norm of up to 9e-5, and FP8 codes in up to 3 of a hundred thousand.  The penalty's gradient is a cube, so one
    rounding of the block output shows up three times as large there."""
    if case["kind"] == "int8_token":   # integer sums, and binary32 scalings in a stated order
        return "exact"
    return {"rel": 4e-4, "max": 0.1 if case["kind"] == "block_fwd" else 0.032, "differ": 1.2e-4}

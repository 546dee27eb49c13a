"""What this framework is timed on: single linear layers and the weight
quantizer, each through the public entry points as a serving or diffusion
program calls them, from one decoded token to a full diffusion transformer
batch.

A layer call quantizes a bf16 activation and multiplies it with a weight
quantized beforehand; its outputs are Y and everything else the calls write
(codes, scales, phi).  The activations are normal draws with outlier channels
and massive-activation tokens, the weights N(0, 0.02^2).
"""
import math

import numpy as np
import torch

from paper_2608_26581_gb300 import rfq

DEV = "cuda"
WAN = 32760 * 5120 * 13824          # multiply-adds of the largest listed layer


def listed():
    return [
        # one decoded token through a gate/up projection (Qwen3-VL-8B, 4096 -> 24576)
        dict(name="decode_gate_up_m1", kind="linear", M=1, K=4096, N=24576, out="bf16"),
        # a decode batch through the down projection of the same model: few output columns, long K
        dict(name="decode_down_m48", kind="linear", M=48, K=12288, N=4096, out="bf16"),
        # the smallest call: a few tokens through a square projection, quantizer and GEMM in one launch
        dict(name="decode_fused_m8", kind="fused", M=8, K=4096, N=4096, out="bf16"),
        # a short, ragged prefill through the down projection, fp32 output for a following reduction
        dict(name="prefill_down_m333", kind="linear", M=333, K=12288, N=4096, out="f32"),
        # a 4096-token prefill through the gate/up projection
        dict(name="prefill_gate_up", kind="linear", M=4096, K=4096, N=24576, out="bf16"),
        # the largest: a whole video batch through the FFN up projection of a Wan2.2-14B DiT block
        dict(name="wan_ffn_up", kind="linear", M=32760, K=5120, N=13824, out="bf16"),
        # the same layer on a ragged piece of it with the residual kept only on tiles above a threshold
        dict(name="selective_phi_m1777", kind="phi", M=1777, K=5120, N=13824, out="bf16", tau=200.0),
        # the FP8 residual (more accurate, slower), on a quarter of the Wan batch
        dict(name="fp8_residual_m8190", kind="mixed", M=8190, K=5120, N=13824, out="bf16"),
        # the HiF4 format, prefill and decode, down projection of Qwen3-VL-8B
        dict(name="hif4_down", kind="hif4", M=4096, K=12288, N=4096, out="bf16"),
        dict(name="hif4_decode_m32", kind="hif4", M=32, K=12288, N=4096, out="bf16"),
        # the expert gate/up projections of Qwen3-VL-30B-A3B, 4096 tokens routed to 8 of 128 experts
        dict(name="moe_gate_up", kind="moe", M=32768, K=2048, N=1536, groups=128, out="bf16"),
        # loading a model: one weight matrix quantized
        dict(name="quantize_weight", kind="weight", M=0, K=5120, N=13824, out="mxfp4"),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["linear"] * 5 + ["fused", "phi", "mixed", "hif4", "hif4", "moe", "weight"])
    while True:
        c = dict(kind=kind, M=_log(rng, 1, 32760), K=128 * _log(rng, 4, 108), N=16 * _log(rng, 32, 1536),
                 out="f32" if rng.random() < 0.2 else "bf16")
        if kind == "fused":
            c["M"] = _log(rng, 1, 256)
        elif kind == "phi":
            c["K"] = 256 * _log(rng, 2, 54)
            c["tau"] = float(rng.choice([100.0, 200.0, 300.0]))
        elif kind == "mixed":
            c["M"] = _log(rng, 128, 8190)
        elif kind == "hif4":
            c["M"], c["K"] = _log(rng, 1, 4096), 64 * _log(rng, 8, 192)
            c["N"] = 16 * _log(rng, 32, 768)
        elif kind == "moe":
            c["groups"] = rng.randrange(8, 129)
            c["M"], c["K"], c["N"] = _log(rng, 2048, 32768), 128 * _log(rng, 4, 16), 128 * _log(rng, 4, 12)
        elif kind == "weight":
            c["M"], c["out"] = 0, rng.choice(["mxfp4", "mxfp4", "hif4", "mxfp8"])
            c["K"] = 128 * _log(rng, 4, 40)
            c["N"] = 16 * _log(rng, 32, 864)
        if c["M"] * c["K"] * c["N"] <= (WAN // 4 if kind == "mixed" else WAN):
            return c


# ------------------------------------------------------------------ inputs

def _counts(case, seed):
    """Rows routed to each expert (uneven; the seed says which expert gets which share) and the padded
    row at which each expert starts."""
    r = np.random.default_rng(17)
    z = r.standard_normal(case["groups"])
    p = np.exp(z - z.max())
    n = np.random.default_rng(seed).permutation(r.multinomial(case["M"], p / p.sum()))
    off = np.concatenate([[0], np.cumsum(-(-n // 128) * 128)])
    return n, off


def _inputs(case, seed):
    """X [rows, K] and W [K, N] ([groups * N] columns for experts) in bf16."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    M, K, N = case["M"], case["K"], case["N"]
    n_w = N * case.get("groups", 1)
    w = torch.empty(K, n_w, dtype=torch.bfloat16, device=DEV)
    w.normal_(0.0, 0.02, generator=g)
    if case["kind"] == "weight":
        return None, w
    x = torch.empty(M, K, dtype=torch.bfloat16, device=DEV)
    x.normal_(0.0, 1.0, generator=g)
    cols = torch.randperm(K, generator=g, device=DEV)[: max(1, K // 100)]
    x[:, cols] *= 64.0
    toks = torch.randperm(M, generator=g, device=DEV)[: -(-M // 1000)]
    x[toks] *= 200.0 if M >= 1000 else 8.0
    if case["kind"] == "moe":
        n, off = _counts(case, seed)
        full = torch.zeros(max(int(off[-1]), 128), K, dtype=torch.bfloat16, device=DEV)
        at = np.concatenate([np.arange(o, o + k) for o, k in zip(off[:-1], n)])
        full[torch.from_numpy(at).to(DEV)] = x
        x = full
    return x, w


def prepare(case, seed):
    x, w = _inputs(case, seed)
    kind, K, N = case["kind"], case["K"], case["N"]
    s = dict(case=case, x=x)
    lay = rfq.RFQ_SCALE_MMA
    hif4 = kind == "hif4"
    if kind == "weight":
        fmt = {"mxfp4": rfq.RFQ_FMT_MXFP4, "hif4": rfq.RFQ_FMT_HIF4, "mxfp8": rfq.RFQ_FMT_MXFP8}[case["out"]]
        s["w"], s["wq"] = w, rfq.empty_qtensor(fmt, lay, N, K)
        return s
    fmt = rfq.RFQ_FMT_HIF4 if hif4 else rfq.RFQ_FMT_MXFP4
    wq = rfq.empty_qtensor(fmt, lay, w.shape[1], K)
    rfq.rfq_quantize_weight(w, wq)
    if hif4:
        wo = rfq.empty_bf16_operand(N, K)
        rfq.rfq_dequant(wq, wo.codes)
        wq = wo
    s["wq"] = wq
    M = x.shape[0]
    bf16 = case["out"] == "bf16"
    s["y"] = torch.empty(M, N, dtype=torch.bfloat16 if bf16 else torch.float32, device=DEV)
    s["out"] = rfq.RFQ_OUT_BF16 if bf16 else rfq.RFQ_OUT_F32
    if kind == "fused":
        s["ws"] = rfq.fused_workspace(M, K)
        return s
    s["ws"] = torch.zeros(rfq.rfq_linear_workspace_bytes() // 4, dtype=torch.int32, device=DEV)
    s["xq"] = rfq.empty_qtensor(fmt, lay, M, K)
    s["xr"] = rfq.empty_qtensor(rfq.RFQ_FMT_MXFP8 if kind == "mixed" else fmt, lay, M, K)
    if hif4:
        s["xo"], s["ro"] = rfq.empty_bf16_operand(M, K), rfq.empty_bf16_operand(M, K)
    if kind == "phi":
        s["phi"] = torch.empty((M + 127) // 128 * ((K + 255) // 256), dtype=torch.uint8, device=DEV)
    if kind == "moe":
        s["off"] = torch.from_numpy(_counts(case, seed)[1].astype(np.int32)).to(DEV)
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "weight":
        rfq.rfq_quantize_weight(s["w"], s["wq"])
        return {"codes": s["wq"].codes, "scales": s["wq"].scales}
    y, ws, wq, out = s["y"], s["ws"], s["wq"], s["out"]
    if kind == "fused":
        rfq.rfq_linear_fused(s["x"], wq, y, out, ws)
        return {"y": y}
    xq, xr = s["xq"], s["xr"]
    got = {"y": y, "codes": xq.codes, "scales": xq.scales, "res_codes": xr.codes, "res_scales": xr.scales}
    if kind == "hif4":
        rfq.rfq_quantize_act_expand(s["x"], xq, xr, s["xo"], s["ro"])
        rfq.rfq_linear(s["xo"], s["ro"], None, 256, wq, y, out, ws)
        got["main_bf16"], got["res_bf16"] = s["xo"].codes, s["ro"].codes
    elif kind == "phi":
        rfq.rfq_quantize_act(s["x"], xq, xr, s["phi"], mode=rfq.RFQ_FALLBACK_AMAX, tau=c["tau"])
        rfq.rfq_linear(xq, xr, s["phi"], 256, wq, y, out, ws)
        got["phi"] = s["phi"]
    else:
        rfq.rfq_quantize_act(s["x"], xq, xr)
        if kind == "mixed":
            rfq.rfq_linear_mixed(xq, xr, None, 256, wq, y, out, ws)
        elif kind == "moe":
            rfq.rfq_linear_grouped(xq, xr, None, 256, s["off"], wq, c["N"], y, out, ws)
        else:
            rfq.rfq_linear(xq, xr, None, 256, wq, y, out, ws)
    return got


def work(case):
    """Bytes: X, the stored weight, and every output once.  Operations: main and residual product."""
    M, K, N, kind = case["M"], case["K"], case["N"], case["kind"]
    q = {"mxfp4": 17 / 32, "mxfp8": 33 / 32, "hif4": 36 / 64}      # bytes per element of each format
    if kind == "weight":
        return {"bytes": K * N * (2 + q[case["out"]]), "flops": 0}
    y = M * N * (2 if case["out"] == "bf16" else 4)
    if kind == "fused":
        return {"bytes": 2 * M * K + N * K * q["mxfp4"] + y, "flops": 4 * M * N * K}
    if kind == "hif4":
        return {"bytes": M * K * (2 + 2 * q["hif4"] + 4) + 2 * N * K + y, "flops": 4 * M * N * K}
    res = q["mxfp8"] if kind == "mixed" else q["mxfp4"]
    w = N * K * q["mxfp4"] * case.get("groups", 1)
    # (a threshold keeps part of the residual: only the main product is sure)
    return {"bytes": M * K * (2 + q["mxfp4"] + res) + w + y, "flops": (2 if kind == "phi" else 4) * M * N * K}


# ------------------------------------------------------------------ the values in 64 bits

def _log2(v):
    return torch.frexp(v)[1] - 1                                   # floor(log2 v), v > 0


def _pow2(e):
    return ((e.to(torch.int64) + 1023) << 52).view(torch.float64)     # 2^e, exactly


def _mx(x, fp8=False):
    """MXFP4 / MXFP8 values of x [rows, K] (blocks of 32 along K)."""
    top, low, man, most = (8, -6, 3, 448.0) if fp8 else (2, 0, 1, 6.0)
    b = x.reshape(x.shape[0], -1, 32)
    am = b.abs().amax(-1, keepdim=True)
    s = _pow2(torch.where(am > 0, _log2(am) - top, -127).clamp(-127, 127))
    v = b / s
    q = _pow2(torch.where(v != 0, _log2(v.abs()), low).clamp(min=low) - man)
    return ((torch.round(v / q) * q).clamp(-most, most) * s).reshape(x.shape)


def _hif4(x):
    """HiF4 values of x [rows, K] (blocks of 64, sub-groups of 4 paired in groups of 8)."""
    b = x.reshape(x.shape[0], -1, 16, 4)
    am = b.abs().amax((-1, -2))
    v = am / 7
    e = _log2(torch.where(am > 0, v, 1.0))
    m = torch.ceil((v / _pow2(e) - 1) * 4).clamp(min=0)
    s = torch.where(am > 0, (1 + m / 4) * _pow2(e), 0.0).clamp(min=2.0 ** -48, max=1.75 * 2.0 ** 15)[..., None]
    sub = b.abs().amax(-1)
    t = (sub > 1.75 * s).to(torch.float64) + (sub > 3.5 * s).to(torch.float64)
    g = (t.reshape(*t.shape[:-1], 8, 2).amax(-1) == 2).to(torch.float64).repeat_interleave(2, -1)
    step = (0.25 * s * torch.exp2(g + (t - g).clamp(min=0)))[..., None]
    return (torch.round(b / step).clamp(-7, 7) * step).reshape(x.shape)


def exact(case, seed):
    kind, N = case["kind"], case["N"]
    if kind == "weight":
        return None
    x, w = _inputs(case, seed)
    quant = _hif4 if kind == "hif4" else _mx
    wt = quant(w.t().contiguous().double())                        # [N, K]
    del w
    y = torch.empty(x.shape[0], N, dtype=torch.float64, device=DEV)
    off = _counts(case, seed)[1] if kind == "moe" else [0, x.shape[0]]
    for g in range(len(off) - 1):
        for r in range(int(off[g]), int(off[g + 1]), 4096):
            end = min(r + 4096, int(off[g + 1]))
            xd = x[r:end].double()
            main = quant(xd)
            res = _mx(xd - main, fp8=True) if kind == "mixed" else quant(xd - main)
            if kind == "phi":
                rows = -(-xd.shape[0] // 128) * 128
                a = torch.zeros(rows, xd.shape[1], dtype=torch.float64, device=DEV)
                a[: xd.shape[0]] = xd.abs()
                on = a.reshape(rows // 128, 128, -1, 256).amax((1, 3)) > case["tau"]
                res *= on.repeat_interleave(128, 0)[: xd.shape[0]].repeat_interleave(256, 1)
            y[r:end] = (main + res) @ wt[g * N : (g + 1) * N].t()
    return {"y": y}

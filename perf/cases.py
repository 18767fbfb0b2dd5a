"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one layer call (or the offline preparation of one layer) through the package's public entry points:

  kind "layer"    SegQuantLinear.forward: quantize -> GEMM -> epilogue, checked and planned on every call
  kind "plan"     the same layer prepared once for its buffers and replayed (SegQuantLinear.plan)
  kind "fused"    the pre-activation in, SiLU / GELU / gated GELU fused into the quantizer, then the GEMM
  kind "token"    W4A8: per-token scales and codes, 4-bit weights unpacked, GEMM with per-(token, channel) factors
  kind "offline"  a new layer: weight scales, weight codes and activation scales from a calibration batch

Sizes are those of the package's workloads (DiT-XL/2, SD3 MMDiT, FLUX, SDXL-like layers) plus a ragged one.
"""
import math

import torch

from paper_2507_14811_b200 import binding as B
from paper_2507_14811_b200.layer import SegQuantLinear

_CAL_ROWS = 256


def _case(name, kind, M, K, N, P=1, Q=1, dual=True, code="int8", x="bf16", y="bf16", pre="normal", mult=False):
    return {"name": name, "kind": kind, "M": M, "K": K, "N": N, "P": P, "Q": Q, "dual": dual, "code": code,
            "x": x, "y": y, "pre": pre, "mult": mult}


def listed():
    return [
        # the smallest layer a caller runs eagerly: fp32 activations, a chunked projection; launches and host work
        _case("tiny_qkv", "layer", 256, 256, 768, Q=3, x="f32", pre="gelu"),
        # adaLN modulation of a batch of 8 samples (one conditioning vector each): the weights are streamed once
        _case("modulation_batch8", "plan", 8, 3072, 18432, Q=6, code="e4m3", pre="silu"),
        # sizes that no tile divides, fp32 in and out, N-segments that end inside a 32-column slab
        _case("ragged_f32", "layer", 1111, 1072, 1000, P=2, Q=3, x="f32", y="f32", pre="gelu"),
        # DiT-XL/2 adaLN projection over the token count, chunked in 6, replayed from a plan
        _case("dit_adaln", "plan", 2048, 1152, 6912, Q=6, pre="silu"),
        # W4A8 on the DiT-XL/2 second MLP layer: dynamic per-token scales, packed weights
        _case("dit_fc2_w4a8", "token", 2048, 4608, 1152, pre="gelu"),
        # gated feed-forward output projection, SDXL-like block of 640 channels, gate fused into the quantizer
        _case("sdxl_geglu", "fused", 8192, 2560, 640, pre="geglu"),
        # attention output projection behind the head merge: one scale per head, 24 K-segments of 64 channels
        _case("sd3_heads", "layer", 8858, 1536, 1536, P=24, dual=False),
        # skip connection: two concatenated streams, many rows, a small projection
        _case("sdxl_skip", "layer", 32768, 1280, 640, P=2, pre="silu"),
        # joint QKV over image and text streams: two K-segments, three N-segments, one activation scale each
        _case("sd3_joint_qkv", "layer", 8858, 3072, 4608, P=2, Q=3, dual=False),
        # second MLP layer with the GELU in front fused into the quantizer
        _case("sd3_fc2_gelu", "fused", 8858, 6144, 1536, pre="gelu"),
        # the largest product: FLUX second MLP layer on FP8 codes
        _case("flux_fc2", "layer", 4608, 12288, 3072, code="e4m3", pre="gelu"),
        # a new layer from fp32 weights: scales per N-segment, codes, activation scales (model load)
        _case("offline_modulation", "offline", 256, 3072, 18432, Q=6, code="e4m3", pre="silu"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    while True:
        kind = rng.choice(["layer", "layer", "plan", "plan", "fused", "fused", "token", "offline"])
        M = int(_log_uniform(rng, 1, 32768)) if kind != "offline" else rng.choice([64, 256])
        K = int(_log_uniform(rng, 256, 12288)) // 16 * 16
        N = int(_log_uniform(rng, 256, 18432)) // 8 * 8
        pre = rng.choice(["silu", "gelu", "geglu"]) if kind == "fused" else rng.choice(["normal", "silu", "gelu"])
        P = rng.choice([1, 1, 1, 2, 2, rng.randint(3, 24)])
        if P > 2:                                         # head merge: equal segments of a multiple of 32 channels
            K = P * (max(32, K // P // 32 * 32))
        Q = 1 if kind == "token" else rng.choice([1, 1, 2, 3, 6])
        if Q > 1 and rng.random() < 0.75:                 # chunks are equal and usually whole 32-column slabs
            N = Q * max(32, N // Q // 32 * 32)
        dual = pre != "normal" and rng.random() < 0.8
        code = "int8" if kind == "token" else rng.choice(["int8", "int8", "e4m3"])
        x = rng.choice(["bf16", "bf16", "bf16", "f32"])
        y = rng.choice(["bf16", "bf16", "bf16", "bf16", "f32"]) if kind != "offline" else "bf16"
        mult = kind == "fused" and rng.random() < 0.3
        if K > 12288 or N > 18432:
            continue
        # no more work than the largest listed cases
        if 2 * M * N * K * (2 if dual else 1) > 4 * 4608 * 12288 * 3072 or M * N > 8858 * 4608 or M * K > 8858 * 6144:
            continue
        c = _case("", kind, M, K, N, P, Q, dual, code, x, y, pre, mult)
        del c["name"]
        return c


# ------------------------------------------------------------------------------------------------ inputs

def _bounds(total, parts, unit):
    """Ascending bounds 0 .. total: equal parts, interior bounds rounded down to multiples of `unit`."""
    return [0] + [total * i // parts // unit * unit for i in range(1, parts)] + [total]


def _bounds_kn(c):
    return _bounds(c["K"], c["P"], 32), _bounds(c["N"], c["Q"], 8)


def _dtype(name):
    return torch.float32 if name == "f32" else torch.bfloat16


def _gelu64(h):
    return h * 0.5 * torch.special.erfc(-h * math.sqrt(0.5))


def _silu64(h):
    return h / (1.0 + torch.exp(-h))


def _draw_pre(c, rows, g, kb):
    """Pre-activations [rows, K] (gated: [rows, 2K]) in fp32; every K-segment has its own range."""
    K = c["K"]
    h = torch.randn((rows, 2 * K if c["pre"] == "geglu" else K), generator=g, device="cuda")
    for p in range(c["P"]):
        h[:, kb[p]:kb[p + 1]] *= 1.0 + 4.0 * p / max(1, c["P"] - 1) if c["P"] > 1 else (1.5 if c["pre"] != "normal" else 1.0)
    return h


def _act(c, h):
    """The activation behind pre-activations h (as stored), rounded once to h's dtype."""
    K, dt = c["K"], h.dtype
    if c["pre"] == "geglu":
        return (h[:, :K].double() * _gelu64(h[:, K:].double())).to(dt)
    if c["pre"] == "normal":
        return h
    return (_gelu64(h.double()) if c["pre"] == "gelu" else _silu64(h.double())).to(dt)


def _inputs(c, seed):
    """Everything that is random: weights, bias, multipliers, the calibration batch and the call's input."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kb, nb = _bounds_kn(c)
    W = torch.randn((c["N"], c["K"]), generator=g, device="cuda") * 0.02
    for q in range(1, c["Q"]):                            # chunked projections have chunks of different ranges
        W[nb[q]:nb[q + 1]] *= 10.0 ** (q / 5.0)
    bias = torch.randn((c["N"],), generator=g, device="cuda") * 0.1
    mult = torch.rand((c["K"],), generator=g, device="cuda") + 0.5 if c["mult"] else None
    dt = _dtype(c["x"])
    X_cal = _act(c, _draw_pre(c, _CAL_ROWS if c["kind"] != "offline" else c["M"], g, kb).to(dt))
    H = _draw_pre(c, c["M"], g, kb).to(dt) if c["kind"] != "offline" else None
    if H is not None and c["kind"] != "fused":
        H = _act(c, H)
    if mult is not None:                                  # scales belong to what the quantizer sees
        X_cal = (X_cal.float() * mult).to(dt)
    return W, bias, mult, X_cal, H


def prepare(case, seed):
    c = case
    kb, nb = _bounds_kn(c)
    W, bias, mult, X_cal, X = _inputs(c, seed)
    M, N, K = c["M"], c["N"], c["K"]
    s = {"case": c, "X": X, "mult": mult}
    if c["kind"] == "offline":
        s.update(W=W, bias=bias, X_cal=X_cal, kb=kb, nb=nb)
        return s
    if c["kind"] == "token":
        seg = B.SegTable(kb, nb)
        s_w, _, w_codes, _ = B.segquant_quantize_per_row(W, seg, False, bits=4)
        s.update(seg=seg, s_w=s_w, W4=B.segquant_pack_w4(w_codes), W8=B.new_codes(N, K, "cuda"), bias=bias,
                 workspace=B.new_workspace())
    else:
        layer = SegQuantLinear(W, bias, kb, nb, c["dual"], c["code"])
        layer.calibrate(X_cal)
        s["layer"] = layer
        if c["kind"] == "fused":
            s["codes"] = B.new_codes(M, K, "cuda"), (B.new_codes(M, K, "cuda") if c["dual"] else None)
    s["Y"] = torch.empty((M, N), dtype=_dtype(c["y"]), device="cuda")
    if c["kind"] == "plan":
        s["plan"] = layer.plan(X, s["Y"])
    return s


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "layer":
        return state["layer"].forward(state["X"], state["Y"])
    if kind == "plan":
        state["plan"].run()
        return state["Y"]
    if kind == "fused":
        l, Y = state["layer"], state["Y"]
        c_pos, c_neg = state["codes"]
        B.segquant_quantize_act_fused(state["X"], l.seg, l.s_pos, l.s_neg, l.code, c["pre"], state["mult"], l.flags, c_pos, c_neg)
        if l.dual:
            return B.segquant_dualscale_gemm(c_pos, c_neg, l.Wq, l.seg, l.code, l.s_pos, l.s_neg, l.s_w, l.bias, l.workspace, Y=Y)
        return B.segquant_seglinear_gemm(c_pos, l.Wq, l.seg, l.code, l.s_pos, l.s_w, l.bias, l.workspace, Y=Y)
    if kind == "token":
        seg = state["seg"]
        s_pos, s_neg, c_pos, c_neg = B.segquant_quantize_per_row(state["X"], seg, c["dual"])
        W8 = B.segquant_unpack_w4(state["W4"], out=state["W8"])
        Y = B.segquant_w4a8_gemm(c_pos, c_neg, W8, seg, s_pos, s_neg, state["s_w"], state["bias"], state["workspace"], Y=state["Y"])
        return (Y, s_pos, s_neg) if c["dual"] else (Y, s_pos)
    layer = SegQuantLinear(state["W"], state["bias"], state["kb"], state["nb"], c["dual"], c["code"])
    layer.calibrate(state["X_cal"])
    return (layer.s_w, layer.Wq, layer.s_pos, layer.s_neg) if c["dual"] else (layer.s_w, layer.Wq, layer.s_pos)


# ------------------------------------------------------------------------------------------------ what is asked of a pass

def work(case):
    c = case
    M, K, N, npol = c["M"], c["K"], c["N"], 2 if c["dual"] else 1
    xs, ys = (4 if c["x"] == "f32" else 2), (4 if c["y"] == "f32" else 2)
    if c["kind"] == "offline":
        return {"bytes": 4 * N * K + N * K + xs * M * K, "flops": 2 * N * K}
    x_bytes = xs * M * K * (2 if c["pre"] == "geglu" and c["kind"] == "fused" else 1)
    w_bytes = N * K // 2 + 4 * N * c["P"] if c["kind"] == "token" else N * K
    return {"bytes": x_bytes + w_bytes + ys * M * N + 4 * N, "flops": 2 * M * N * K * npol}


def tolerance(case):
    c = case
    if c["kind"] == "offline":                            # extrema, one IEEE division each, codes: unique
        return "exact"
    # sums of int8 products are exact and e4m3 ones fp32; the rest is a few fp32 roundings, plus one to the output
    # type.  A fused activation evaluated with other fp32 roundings moves a few values by one step of their code.
    if c["y"] == "f32" and c["kind"] != "fused":
        return {"rel": 1e-5, "max": 1e-4} if c["code"] == "int8" else {"rel": 2e-4, "max": 2e-3}
    return {"rel": 2e-3, "max": 2e-2}


# ------------------------------------------------------------------------------------------------ 64-bit results

def _steps(extremum, q):
    s = extremum.float() / torch.tensor(q, dtype=torch.float32, device=extremum.device)
    return torch.where(extremum > 0, s, torch.ones_like(s))


def _round_codes(q, code, lo, hi):
    """fp32 quotients -> codes as fp64 numbers."""
    if code == "int8":
        return torch.round(q).clamp(lo, hi).double()
    return q.clamp(lo, hi).to(torch.float8_e4m3fn).double()


def _act_scales(X, kb, dual, code):
    q_max, q_min = (127.0, 128.0) if code == "int8" else (448.0, 448.0)
    pos, neg = [], []
    for k0, k1 in zip(kb, kb[1:]):
        x = X[:, k0:k1]
        mx, mn = x.max().float().clamp(min=0), (-x.min().float()).clamp(min=0)
        pos.append(_steps(mx if dual else torch.maximum(mx, mn), q_max))
        neg.append(_steps(mn, q_min))
    return torch.stack(pos), (torch.stack(neg) if dual else None)


def exact(case, seed):
    c = case
    kb, nb = _bounds_kn(c)
    W, bias, mult, X_cal, X = _inputs(c, seed)
    code, dual, P, Q = c["code"], c["dual"], c["P"], c["Q"]
    w_max, lo = (127.0, -128.0) if code == "int8" else (448.0, -448.0)
    if c["kind"] == "token":
        w_max = 7.0
        s_w = torch.stack([_steps(W[:, a:b].abs().amax(1), 7.0) for a, b in zip(kb, kb[1:])], 1)        # [N, P]
        w_scale = s_w
    else:
        s_w = torch.stack([torch.stack([_steps(W[n0:n1, a:b].abs().max(), w_max) for n0, n1 in zip(nb, nb[1:])])
                           for a, b in zip(kb, kb[1:])])                                                # [P, Q]
        rows = torch.repeat_interleave(torch.arange(Q, device="cuda"), torch.tensor([b - a for a, b in zip(nb, nb[1:])], device="cuda"))
        w_scale = s_w.t()[rows]                                                                         # [N, P]
        s_pos, s_neg = _act_scales(X_cal, kb, dual, code)
    Wc = [_round_codes(W[:, a:b] / w_scale[:, p:p + 1], code, -w_max, w_max) for p, (a, b) in enumerate(zip(kb, kb[1:]))]
    if c["kind"] == "offline":
        q = torch.cat(Wc, 1)
        q = q.to(torch.int8).view(torch.uint8) if code == "int8" else (q.float() + 0.0).to(torch.float8_e4m3fn).view(torch.uint8)
        q = torch.where(q == 128, torch.zeros_like(q), q) if code == "e4m3" else q                      # -0 is stored as +0
        return (s_w.reshape(-1), q, s_pos, s_neg) if dual else (s_w.reshape(-1), q, s_pos)
    del W
    M = c["M"]
    Y = torch.empty((M, c["N"]), dtype=torch.float64, device="cuda")
    sp_all, sn_all = [], []
    for r0 in range(0, M, 4096):
        x = X[r0:r0 + 4096]
        if c["kind"] == "fused":
            x = _act(c, x)
        x = x.float()
        if mult is not None:
            x = x * mult
        y = bias.double()[None, :].expand(x.shape[0], -1).clone()
        sp_row, sn_row = [], []
        for p, (a, b) in enumerate(zip(kb, kb[1:])):
            xp = x[:, a:b]
            if c["kind"] == "token":
                mx, mn = xp.amax(1).clamp(min=0), (-xp.amin(1)).clamp(min=0)
                sp = _steps(mx if dual else torch.maximum(mx, mn), 127.0)[:, None]
                sn = _steps(mn, 128.0)[:, None]
                sp_row.append(sp)
                sn_row.append(sn)
            else:
                sp, sn = s_pos[p], (s_neg[p] if dual else None)
            if dual:
                v = _round_codes(torch.where(xp >= 0, xp / sp, torch.zeros_like(xp)), code, 0.0, w_max if c["kind"] != "token" else 127.0) * sp.double()
                v += _round_codes(torch.where(xp < 0, xp / sn, torch.zeros_like(xp)), code, lo, 0.0) * sn.double()
            else:
                top = 127.0 if code == "int8" else 448.0
                v = _round_codes(xp / sp, code, -top, top) * sp.double()
            y += (v @ Wc[p].t()) * w_scale[:, p].double()[None, :]
        Y[r0:r0 + 4096] = y
        if sp_row:
            sp_all.append(torch.cat(sp_row, 1))
            sn_all.append(torch.cat(sn_row, 1))
    if c["kind"] == "token":
        out = (Y, torch.cat(sp_all).double(), torch.cat(sn_all).double())
        return out if dual else out[:2]
    return Y

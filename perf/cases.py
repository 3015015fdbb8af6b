"""Workloads of the library as a user's program runs them, for timing.

Each case is a call (or a short sequence of calls) of paper_2111_13824_gb300.fqvit on inputs with the
shapes and statistics of the DeiT / ViT / Swin layers in paper_2111_13824_gb300.synth, drawn on the GPU
from a seed.  ``listed()`` are the fixed ones, ``draw(rng)`` gives more of the same ranges.

    prepare(case, seed)  inputs, packed weights and scales a program holds before the call
    run(state)           one pass through the public entry points; returns every output
    work(case)           bytes and operations of one pass: each input read once, each output written once
    exact(case, seed)    the computed outputs by plain torch in 64 bits, where they have such a value
"""
from __future__ import annotations

import math

import torch

from paper_2111_13824_gb300 import fqvit

DEV = "cuda:0"
D_HEAD = 64  # head dimension of the ViT models (32 in Swin)


def listed():
    return [
        # one image through one DeiT-T layer (norm1 and the attention core): latency
        dict(name="block_deit_t_b1", kind="block", B=1, L=197, H=3),
        # one layer of ViT-L/16 at 384 px, batch 32: the benchmark's step is 24 of these
        dict(name="block_vit_l384_b32", kind="block", B=32, L=577, H=16),
        # DeiT-S at batch 64, attention output in 8 bits for the projection, V with a zero point
        dict(name="attn_u8_deit_s_b64", kind="attn", B=64, L=197, H=6, d=64, out="u8", zp_v=-9),
        # rows of a ViT-B/16 at 448 px (28 x 28 patches and the class token): above 592 keys
        dict(name="attn_448px_b8", kind="attn", B=8, L=785, H=12, d=64, out="acc", zp_v=0),
        # Swin-S stage 1, shifted 7 x 7 windows: relative-position bias and mask, batch 64
        dict(name="window7_swin_s_b64", kind="window", images=64, side=56, window=7, H=3, shift=True, out="acc"),
        # 12 x 12 windows (384-px inputs), shifted, 8-bit output
        dict(name="window12_b16", kind="window", images=16, side=48, window=12, H=6, shift=True, out="u8"),
        # attention from 8-bit Q, K and V, one ViT-L/384 layer at batch 32
        dict(name="qkv_attn_vit_l384_b32", kind="qkv", B=32, L=577, H=16, zp_q=0, zp_k=0, zp_v=0),
        # norm of Swin-S's first patch merging, batch 64: 4 x 96 channels
        dict(name="ln_merge_swin_s_b64", kind="ln", rows=64 * 28 * 28, C=384),
        # projection of one DeiT-T image: the smallest Linear layer
        dict(name="linear_proj_deit_t_b1", kind="linear", M=197, N=192, K=192),
        # the widest Linear layer: ViT-L/384 fc1 at batch 32
        dict(name="linear_fc1_vit_l384_b32", kind="linear", M=32 * 577, N=4096, K=1024),
        # calibration of one DeiT-S norm on 32 images, then the batch quantized with the result
        dict(name="calibrate_deit_s", kind="calib", rows=32 * 197, C=384, K=3),
        # the whole integer block (norm1, QKV, attention, projection, norm2, MLP) of ViT-B, batch 8
        dict(name="chain_vit_b_b8", kind="chain", B=8, L=197, H=12),
    ]


# ---- drawn cases -------------------------------------------------------------

_MAX_LOGITS = 512 * 577 * 577   # attention logits of the largest listed case
_MAX_MACS = 32 * 577 * 4096 * 1024


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["block", "attn", "attn", "window", "window", "qkv", "ln", "linear", "linear", "calib", "chain"])
    if kind == "block":
        L, H = rng.randint(50, 592), rng.choice([3, 6, 12, 16])
        return dict(kind=kind, B=_log_int(rng, 1, max(1, _MAX_LOGITS // (H * L * L))), L=L, H=H)
    if kind == "attn":
        L, H = rng.randint(65, 1024), rng.choice([3, 6, 12, 16])
        cap = _MAX_LOGITS // (4 * H * L * L)
        return dict(kind=kind, B=_log_int(rng, 1, max(1, min(64, cap))), L=L, H=H, d=64,
                    out=rng.choice(["acc", "u8"]), zp_v=rng.choice([0, rng.randint(-128, 127)]))
    if kind == "window":
        w, H = rng.choice([7, 7, 8, 12]), rng.choice([3, 4, 6, 8, 12, 24])
        side = w * rng.randint(1, 8)
        cap = 12000 * 49 * 49 // ((side // w) ** 2 * H * w ** 4)
        return dict(kind=kind, images=_log_int(rng, 1, max(1, min(64, cap))), side=side, window=w, H=H,
                    shift=rng.random() < 0.5, out=rng.choice(["acc", "u8"]))
    if kind == "qkv":
        L, H = rng.randint(50, 592), rng.choice([3, 6, 12, 16])
        return dict(kind=kind, B=_log_int(rng, 1, max(1, _MAX_LOGITS // (H * L * L))), L=L, H=H,
                    zp_q=rng.choice([0, rng.randint(-40, 40)]), zp_k=rng.choice([0, rng.randint(-40, 40)]),
                    zp_v=rng.choice([0, rng.randint(-40, 40)]))
    if kind == "ln":
        return dict(kind=kind, rows=_log_int(rng, 1, 60000), C=16 * rng.randint(6, 96))
    if kind == "linear":
        N, K = 16 * _log_int(rng, 4, 256), 8 * _log_int(rng, 8, 512)
        return dict(kind=kind, M=_log_int(rng, 1, min(20000, _MAX_MACS // (N * K))), N=N, K=K)
    if kind == "calib":
        return dict(kind=kind, rows=_log_int(rng, 197, 32 * 577), C=16 * rng.randint(6, 64), K=rng.randint(1, 4))
    return dict(kind="chain", B=_log_int(rng, 1, 12), L=rng.randint(50, 577), H=rng.choice([3, 6, 12]))


# ---- inputs ------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _f32(x):
    return float(torch.tensor(x, dtype=torch.float32))


def _channels(g, rows, C):
    """Real activations whose channel ranges spread log-normally, the widest 40 x the median."""
    r = torch.randn(C, generator=g, device=DEV)
    r = torch.exp((r - r.median()) * (math.log(40.0) / (r.max() - r.median()).clamp_min(0.1)))
    m = 0.25 * r * torch.randn(C, generator=g, device=DEV)
    return m + (r / 6.0) * torch.randn(rows, C, generator=g, device=DEV)


def _norm(g, C):
    gamma = 1.0 + 0.1 * torch.randn(C, generator=g, device=DEV)
    beta = 0.1 * torch.randn(C, generator=g, device=DEV)
    return gamma, beta


def _ln_inputs(g, rows, C, K=3):
    """PTF codes of such activations: layer scale from the range, factors from the channels' ranges."""
    x = _channels(g, rows, C)
    lo, hi = float(x.min()), float(x.max())
    s0 = max(hi - lo, 1e-6) / 255.0
    s, zp = s0 / 2 ** K, int(min(255, max(0, round(-lo / s0))))
    need = x.abs().amax(0) / (s * 100.0)
    alpha = torch.clamp(torch.ceil(torch.log2(need.clamp_min(1e-6))), 0, K)
    xq = torch.clamp(torch.round(x / (torch.exp2(alpha) * s)) + zp, 0, 255).to(torch.uint8)
    gamma, beta = _norm(g, C)
    return dict(xq=xq, zp_in=zp, alpha=alpha.to(torch.uint8), gamma=gamma, beta=beta, s_out=_f32(9.2 / 255.0),
                zp_out=128)


def _codes(g, BH, L, d, zp=0):
    """Signed 8-bit codes of N(0, 1) values over +-4.5 sigma, with a zero point, and their scale."""
    s = 4.5 / 127.0
    x = torch.round(torch.randn(BH, L, d, generator=g, device=DEV) / s) + zp
    return torch.clamp(x, -128, 127).to(torch.int8), _f32(s)


def _logit_quantizer(q, k, zp_q, zp_k, s_q, s_k, d):
    """MinMax of the real logits over up to 64 heads: (s_logit in the supported range, zero point)."""
    n = min(64, q.shape[0])
    p = torch.bmm(q[:n].float() - zp_q, (k[:n].float() - zp_k).transpose(1, 2)) * (s_q * s_k / math.sqrt(d))
    lo, hi = float(p.min()), float(p.max())
    s = _f32(min(0.5, max(2.0 ** -7, (hi - lo) / 255.0)))
    return s, int(min(255, max(0, round(-lo / s)))) - 128


def _logits(g, BH, L, d):
    """int8 logits [BH * L, ld] (rows padded to 16 bytes), their scale, and V's codes."""
    q, s_q = _codes(g, BH, L, d)
    k, s_k = _codes(g, BH, L, d)
    s, zp = _logit_quantizer(q, k, 0, 0, s_q, s_k, d)
    out = torch.zeros(BH, L, (L + 15) // 16 * 16, dtype=torch.int8, device=DEV)
    for b in range(0, BH, 256):
        p = torch.bmm(q[b:b + 256].float(), k[b:b + 256].float().transpose(1, 2)) * (s_q * s_k / math.sqrt(d) / s)
        out[b:b + 256, :, :L] = torch.clamp(torch.round(p) + zp, -128, 127).to(torch.int8)
    return out.reshape(BH * L, -1), s


def _regions(side, w):
    """Region ids [windows, w * w] of a map shifted by w // 2: three bands per axis."""
    t = torch.arange(side)
    band = (t >= side - w).long() + (t >= side - w // 2).long()
    ids = (3 * band[:, None] + band[None, :]).reshape(side // w, w, side // w, w).permute(0, 2, 1, 3)
    return ids.reshape(-1, w * w).to(torch.uint8).to(DEV).contiguous()


def _minmax(v):
    lo, hi = min(float(v.min()), 0.0), max(float(v.max()), 0.0)
    s = _f32(max(hi - lo, 1e-6) / 255.0)
    return s, int(min(255, max(0, round(-lo / s))))


def _linear_weights(g, N, K, s_x):
    w = 0.02 * torch.randn(N, K, generator=g, device=DEV) * (0.5 + 1.5 * torch.rand(N, 1, generator=g, device=DEV))
    s_w = w.abs().amax(1) / 127.0
    codes = torch.clamp(torch.round(w / s_w[:, None]), -127, 127).to(torch.int8)
    bias = torch.round(0.02 * torch.randn(N, generator=g, device=DEV) / (s_x * s_w)).to(torch.int32)
    return codes, s_w, bias


def _linear_real(x, zp_x, s_x, codes, s_w, bias):
    return ((x.float() - zp_x) @ codes.float().T + bias.float()) * (s_x * s_w)


def _linear_inputs(g, M, N, K):
    """A layer over N(0, 1) activations (the norm's and the attention's outputs), MinMax quantized."""
    x = torch.randn(M, K, generator=g, device=DEV)
    s_x, zp_x = _minmax(x)
    x = torch.clamp(torch.round(x / s_x) + zp_x, 0, 255).to(torch.uint8)
    codes, s_w, bias = _linear_weights(g, N, K, s_x)
    s_y, zp_y = _minmax(_linear_real(x[:512], zp_x, s_x, codes, s_w, bias))
    return dict(x=x, zp_x=zp_x, s_x=s_x, w=codes, s_w=s_w, bias=bias, s_y=s_y, zp_y=zp_y)


def _chain_inputs(g, B, L, H, d):
    """A block's weights and the MinMax scales of its stages, from the real-valued block on one image."""
    C = H * d
    st = dict(B=B, L=L, H=H, d=d, n1=_ln_inputs(g, B * L, C))
    n1 = st["n1"]
    xi = (n1["xq"][:L].float() - n1["zp_in"]) * torch.exp2(n1["alpha"].float())
    gamma2, beta2 = _norm(g, C)

    def norm(x, gamma, beta):
        return (x - x.mean(1, keepdim=True)) / x.std(1, keepdim=True, unbiased=False).clamp_min(1e-6) * gamma + beta

    def linear(x, s_x, zp_x, N):
        codes, s_w, bias = _linear_weights(g, N, x.shape[1], s_x)
        xq = torch.clamp(torch.round(x / s_x) + zp_x, 0, 255)
        y = _linear_real(xq, zp_x, s_x, codes, s_w, bias)
        s_y, zp_y = _minmax(1.1 * y)
        return y, dict(w_h=fqvit.linear_pack_weight(codes), s_w=s_w, bias=bias, s_x=s_x, zp_x=zp_x, s_y=s_y, zp_y=zp_y)

    y1 = norm(xi, n1["gamma"], n1["beta"])
    qkv, st["qkv"] = linear(y1, n1["s_out"], n1["zp_out"], 3 * C)
    s, zp = st["qkv"]["s_y"], st["qkv"]["zp_y"]
    q, k, v = qkv.reshape(L, 3, H, d).permute(1, 2, 0, 3)
    logits = torch.bmm(q, k.transpose(1, 2)) / math.sqrt(d)
    lo, hi = float(logits.min()), float(logits.max())
    s_l = _f32(min(0.5, max(2.0 ** -7, (hi - lo) / 255.0)))
    st.update(s_qkv=s, zp_s=zp - 128, s_logit=s_l, zp_logit=int(min(255, max(0, round(-lo / s_l)))) - 128)
    att = torch.bmm(torch.softmax(logits, -1), v).permute(1, 0, 2).reshape(L, C)
    st["s_att"], st["zp_att"] = _minmax(1.3 * att)
    p, st["proj"] = linear(att, st["s_att"], st["zp_att"], C)
    st["n2"] = dict(alpha=torch.zeros(C, dtype=torch.uint8, device=DEV), gamma=gamma2, beta=beta2,
                    s_out=_f32(9.2 / 255.0), zp_out=128)
    y2 = norm(p, gamma2, beta2)
    f1, st["fc1"] = linear(y2, st["n2"]["s_out"], 128, 4 * C)
    _, st["fc2"] = linear(f1, st["fc1"]["s_y"], st["fc1"]["zp_y"], C)
    return st


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    st = dict(kind=kind)
    if kind == "block":
        BH, L, C = case["B"] * case["H"], case["L"], case["H"] * D_HEAD
        st.update(_ln_inputs(g, case["B"] * L, C))
        st["logits"], st["s_logit"] = _logits(g, BH, L, D_HEAD)
        st["v"], _ = _codes(g, BH, L, D_HEAD)
        st["yq"] = torch.empty_like(st["xq"])
        st["acc"] = torch.empty(BH, L, D_HEAD, dtype=torch.int32, device=DEV)
    elif kind == "attn":
        BH, L = case["B"] * case["H"], case["L"]
        st["logits"], st["s_logit"] = _logits(g, BH, L, case["d"])
        st["v"], st["s_v"] = _codes(g, BH, L, case["d"], case["zp_v"])
        st.update(zp_v=case["zp_v"], out=case["out"], s_out=_f32(1.5 * st["s_v"]), zp_out=128)
    elif kind == "window":
        w, side, H = case["window"], case["side"], case["H"]
        nw, L = (side // w) ** 2, w * w
        BH = case["images"] * nw * H
        st["logits"], st["s_logit"] = _logits(g, BH, L, 32)
        st["v"], st["s_v"] = _codes(g, BH, L, 32)
        st["bias"] = torch.randint(-16, 17, (H, (2 * w - 1) ** 2), generator=g, device=DEV).to(torch.int8)
        st["region"] = _regions(side, w) if case["shift"] and nw > 1 else None
        st.update(mask=max(-32768, round(-100.0 / st["s_logit"])), heads=H, window=w, out=case["out"],
                  s_out=_f32(1.5 * st["s_v"]), zp_out=128)
    elif kind == "qkv":
        BH, L = case["B"] * case["H"], case["L"]
        st["q"], st["s_q"] = _codes(g, BH, L, D_HEAD, case["zp_q"])
        st["k"], st["s_k"] = _codes(g, BH, L, D_HEAD, case["zp_k"])
        st["v"], _ = _codes(g, BH, L, D_HEAD, case["zp_v"])
        st["s_logit"], st["zp_logit"] = _logit_quantizer(st["q"], st["k"], case["zp_q"], case["zp_k"], st["s_q"],
                                                         st["s_k"], D_HEAD)
        st.update(zp_q=case["zp_q"], zp_k=case["zp_k"], zp_v=case["zp_v"])
        # the logits workspace a program keeps with the layer
        st["workspace"] = torch.empty(fqvit.qk_workspace_size(BH, L), dtype=torch.int8, device=DEV)
    elif kind == "ln":
        st.update(_ln_inputs(g, case["rows"], case["C"]))
    elif kind == "linear":
        st.update(_linear_inputs(g, case["M"], case["N"], case["K"]))
        st["w_h"] = fqvit.linear_pack_weight(st.pop("w"))
    elif kind == "calib":
        st["x"] = _channels(g, case["rows"], case["C"])
        st["K"] = case["K"]
        st["sse"] = torch.empty(case["C"], case["K"] + 1, dtype=torch.float64, device=DEV)
    elif kind == "chain":
        st.update(_chain_inputs(g, case["B"], case["L"], case["H"], D_HEAD))
    else:
        raise ValueError(kind)
    return st


# ---- one pass ----------------------------------------------------------------


def _linear(x, p):
    return fqvit.linear_q(x, p["zp_x"], p["s_x"], p["w_h"], p["s_w"], p["bias"], p["s_y"], p["zp_y"])


def _run_chain(st):
    n1, n2, B, L, H = st["n1"], st["n2"], st["B"], st["L"], st["H"]
    y1 = fqvit.ptf_layernorm(n1["xq"], n1["zp_in"], n1["alpha"], n1["gamma"], n1["beta"], n1["s_out"], n1["zp_out"])
    qkv = _linear(y1, st["qkv"])
    q, k, v = fqvit.split_qkv(qkv, B, L, H, st["d"])
    logits = fqvit.qk_logits(q, k, st["zp_s"], st["zp_s"], st["s_qkv"], st["s_qkv"], st["s_logit"], st["zp_logit"])
    att = fqvit.lis_attention_q(logits, st["s_logit"], v, st["zp_s"], st["s_qkv"], st["s_att"], st["zp_att"])
    merged = fqvit.merge_heads(att, B, L, H)
    proj = _linear(merged, st["proj"])
    y2 = fqvit.ptf_layernorm(proj, st["proj"]["zp_y"], n2["alpha"], n2["gamma"], n2["beta"], n2["s_out"], n2["zp_out"])
    f1 = _linear(y2, st["fc1"])
    return dict(norm1=y1, qkv=qkv, logits=logits, attn=merged, proj=proj, norm2=y2, fc1=f1, fc2=_linear(f1, st["fc2"]))


def run(st):
    kind = st["kind"]
    if kind == "block":
        return fqvit.block_int(st["xq"], st["zp_in"], st["alpha"], st["gamma"], st["beta"], st["s_out"], st["zp_out"],
                               st["yq"], st["logits"], st["logits"].shape[1], st["s_logit"], st["v"], 0, st["acc"])
    if kind == "attn":
        if st["out"] == "u8":
            return fqvit.lis_attention_q(st["logits"], st["s_logit"], st["v"], st["zp_v"], st["s_v"], st["s_out"],
                                         st["zp_out"])
        return fqvit.lis_attention(st["logits"], st["s_logit"], st["v"], st["zp_v"])
    if kind == "window":
        where = dict(bias=st["bias"], heads=st["heads"], window=st["window"])
        if st["out"] == "u8":
            return fqvit.lis_attention_masked_q(st["logits"], st["s_logit"], st["v"], st["region"], st["mask"], 0,
                                                st["s_v"], st["s_out"], st["zp_out"], **where)
        return fqvit.lis_attention_masked(st["logits"], st["s_logit"], st["v"], st["region"], st["mask"], **where)
    if kind == "qkv":
        return fqvit.qk_lis_attention(st["q"], st["k"], st["v"], st["zp_q"], st["zp_k"], st["s_q"], st["s_k"],
                                      st["s_logit"], st["zp_logit"], st["zp_v"], workspace=st["workspace"])
    if kind == "ln":
        return fqvit.ptf_layernorm(st["xq"], st["zp_in"], st["alpha"], st["gamma"], st["beta"], st["s_out"],
                                   st["zp_out"])
    if kind == "linear":
        return _linear(st["x"], st)
    if kind == "calib":
        s, zp, alpha = fqvit.calibrate_ptf(st["x"], K=st["K"], sse=st["sse"])
        xq = fqvit.ptf_quantize(st["x"], float(s.item()), int(zp.item()), alpha)
        return dict(s=s, zp=zp, alpha=alpha, sse=st["sse"], xq=xq)
    return _run_chain(st)


# ---- the work a pass cannot do without ---------------------------------------


def _attn_work(BH, L, d, out_bytes, logits=True):
    n = BH * L
    return (n * L if logits else 0) + n * d * (1 + out_bytes), 2 * n * L * d


def _linear_work(M, N, K):
    return M * K + 2 * N * K + M * N + 8 * N, 2 * M * N * K


def work(case):
    kind = case["kind"]
    if kind == "block":
        rows, C = case["B"] * case["L"], case["H"] * D_HEAD
        b, f = _attn_work(case["B"] * case["H"], case["L"], D_HEAD, 4)
        b, f = b + 2 * rows * C + 9 * C, f + 8 * rows * C
    elif kind == "attn":
        b, f = _attn_work(case["B"] * case["H"], case["L"], case["d"], 1 if case["out"] == "u8" else 4)
    elif kind == "window":
        BH = case["images"] * (case["side"] // case["window"]) ** 2 * case["H"]
        b, f = _attn_work(BH, case["window"] ** 2, 32, 1 if case["out"] == "u8" else 4)
    elif kind == "qkv":
        BH, L = case["B"] * case["H"], case["L"]
        b, f = _attn_work(BH, L, D_HEAD, 4, logits=False)
        b, f = b + 2 * BH * L * D_HEAD, 2 * f
    elif kind == "ln":
        b, f = 2 * case["rows"] * case["C"] + 9 * case["C"], 8 * case["rows"] * case["C"]
    elif kind == "linear":
        b, f = _linear_work(case["M"], case["N"], case["K"])
    elif kind == "calib":
        n = case["rows"] * case["C"]
        b, f = 4 * n + 4 * n + n, n * (case["K"] + 1) * 8
    else:
        M, C, BH, L = case["B"] * case["L"], case["H"] * D_HEAD, case["B"] * case["H"], case["L"]
        b, f = 2 * (2 * M * C + 9 * C), 16 * M * C
        for N, K in ((3 * C, C), (C, C), (4 * C, C), (C, 4 * C)):
            x, y = _linear_work(M, N, K)
            b, f = b + x, f + y
        x, y = _attn_work(BH, L, D_HEAD, 1, logits=False)
        b, f = b + x + 2 * M * C + BH * L * L, f + 2 * y  # the logits are an output of the chain
    return {"bytes": int(b), "flops": int(f)}


# ---- 64-bit values -----------------------------------------------------------


def exact(case, seed):
    """The calibration's scale and error sums and a Linear layer's codes.  The other outputs are integers
    that the paper's integer algorithms define bit for bit; they have no separate real value."""
    g = _gen(seed)
    if case["kind"] == "calib":
        x, K = _channels(g, case["rows"], case["C"]), case["K"]
        s0 = (x.max() - x.min()) / 255.0
        zp = float(torch.clamp(torch.round(-x.min() / s0), 0, 255))
        sse = torch.empty(case["C"], K + 1, dtype=torch.float64, device=DEV)
        for a in range(K + 1):
            step = s0 * 2.0 ** (a - K)
            d = x - torch.clamp(torch.round(x / step), -zp, 255 - zp) * step
            sse[:, a] = d.double().square().sum(0)
        s = (x.max().double() - x.min().double()) / 255.0 / 2 ** K
        return dict(s=s.reshape(1), zp=None, alpha=None, sse=sse, xq=None)
    if case["kind"] == "linear" and case["M"] * case["N"] * case["K"] <= _MAX_MACS:
        p = _linear_inputs(g, case["M"], case["N"], case["K"])
        acc = (p["x"].double() - p["zp_x"]) @ p["w"].double().T + p["bias"].double()
        m = (torch.tensor(p["s_x"], device=DEV) * p["s_w"]) / torch.tensor(p["s_y"], device=DEV)
        n1 = torch.clamp(7 - torch.floor(torch.log2(m.double())), max=31)
        y = torch.floor(torch.floor(m.double() * torch.exp2(n1)) * acc / torch.exp2(n1) + 0.5) + p["zp_y"]
        return torch.clamp(y, 0, 255).to(torch.uint8)
    return None

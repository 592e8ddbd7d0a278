"""Workloads that the library is timed on.

Each case is one pass of a layer (or of an encoder / decoder call, or of one
attention decode step) through the package's public entry points, on inputs
already on the GPU.  Sizes are those of paper_2509_26436_gb300/inputs.py
(FLUX.1-schnell, PixArt-Sigma, SDXL and LLaMA-2-7B layers, the Table 6
attention settings, the encode sweep) and generic ones between them.

exact() restates Eq. 1, Eq. 2 and the layer from their definitions in plain
torch, in 64 bits; it uses nothing of this package.
"""
import math

import torch

import paper_2509_26436_gb300 as Q

_DTYPES = {"float16": torch.float16, "bfloat16": torch.bfloat16, "float32": torch.float32}
_D = 128  # head dimension of the attention step


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _linear(name, path, M, N, K, group_s, out="float16", bias=False, mode="sym", code_bits=8, prepared=True,
            flag_bits=8):
    c = dict(kind="linear", path=path, M=M, N=N, K=K, group_s=group_s, out=out, bias=bias, mode=mode,
             code_bits=code_bits, prepared=prepared, flag_bits=flag_bits)
    return dict(c, name=name) if name else c


def _attention(name, heads, batch, L, L_max, group_s, flag_bits=8, out="float16"):
    c = dict(kind="attention", heads=heads, batch=batch, L=L, L_max=L_max, group_s=group_s, flag_bits=flag_bits,
             out=out)
    return dict(c, name=name) if name else c


def _codec(name, kind, rows, K, group_s, mode="sym", code_bits=8, flag_bits=8):
    c = dict(kind=kind, rows=rows, K=K, group_s=group_s, mode=mode, code_bits=code_bits, flag_bits=flag_bits)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small layer (256 tokens, hidden 1152): launches and latency count
        _linear("small_1152", "f16", 256, 1152, 1152, 16),
        # an LLM's fused qkv projection while decoding, one token for each of 16 sequences
        _linear("llm_decode_qkv", "f16", 16, 12288, 4096, 8, code_bits=16),
        # an LLM's down projection at a 2048-token prefill
        _linear("llm_prefill_down", "f16", 2048, 4096, 11008, 8, code_bits=16),
        # a DiT MLP at 1024 px, encoder and layer called one after the other
        _linear("pixart_fc1", "two_call", 8192, 4608, 1152, 16, bias=True),
        # Eq. 1 with zero points, an odd token count, weights not prepared beforehand, 32-bit results
        _linear("asym_ragged_qkv", "two_call", 4001, 3456, 1152, 32, out="float32", mode="asym", prepared=False),
        # a UNet convolution as im2col GEMM with the latent-diffusion scales: one per tensor, one per channel
        _linear("sdxl_conv_static", "static", 2048, 1280, 11520, 16, bias=True),
        # the largest MLP layers of a DiT block, 18432 tokens: fused call with a bias ...
        _linear("flux_fc1", "f16", 18432, 12288, 3072, 16, out="bfloat16", bias=True),
        # ... and the long reduction, encoder and layer called one after the other
        _linear("flux_fc2", "two_call", 18432, 3072, 12288, 16),
        # one decode step over a long cache: encode the query, append the token, attend
        _attention("attn_32x16_4096", 32, 16, 4096, 4096, 16),
        # the same for one sequence with a short, odd context in a larger cache, FLAGs packed
        _attention("attn_40x1_777", 40, 1, 777, 1024, 8, flag_bits=4),
        # activations to their stored 4-bit form, 128 M elements
        _codec("encode_128m", "encode", 32768, 4096, 16),
        # and back, 16 M elements
        _codec("decode_16m", "decode", 4096, 4096, 32),
    ]


def _log(rng, lo, hi, step=1):
    """A multiple of `step` in [lo, hi], spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    what = rng.choice(["linear"] * 5 + ["attention", "attention", "encode", "decode"])
    gs = rng.choice([8, 16, 16, 32, 64])
    flag_bits = rng.choice([8, 8, 4])
    if what == "linear":
        path = rng.choice(["f16", "f16", "two_call", "two_call", "static"])
        K = _log(rng, 1152, 12288, 64)
        N = _log(rng, 640, 12288, 8)
        most = 18432 * 12288 * 3072 // (N * K)
        M = _log(rng, 1, max(1, min(18432, most)))
        mode, bits = "sym", 8
        if path == "two_call":
            mode = rng.choice(["sym", "sym", "asym"])
        if path != "static" and mode == "sym":
            bits = rng.choice([8, 8, 16])
        return _linear(None, path, M, N, K, gs, out=rng.choice(["float16", "bfloat16", "float32"]),
                       bias=rng.random() < 0.5, mode=mode, code_bits=bits, prepared=rng.random() < 0.75,
                       flag_bits=flag_bits)
    if what == "attention":
        heads, batch = rng.choice([32, 40, 64]), _log(rng, 1, 16)
        L_max = _log(rng, 128, 4096)
        L = max(1, L_max - rng.choice([0, 1, rng.randrange(L_max // 2)]))
        return _attention(None, heads, batch, L, L_max, rng.choice([8, 16, 32]), flag_bits,
                          rng.choice(["float16", "bfloat16", "float32"]))
    K = _log(rng, 1152, 12288, 64)
    rows = _log(rng, 2 ** 17 // K, 2 ** 27 // K)
    mode = rng.choice(["sym", "sym", "asym", "row"])
    bits = rng.choice([8, 8, 16]) if mode == "sym" else 8
    return _codec(None, what, rows, K, gs, mode, bits, flag_bits)


# --------------------------------------------------------------------------
# inputs (the distributions of paper_2509_26436_gb300/inputs.py, drawn on the GPU)
# --------------------------------------------------------------------------
def _activations(g, rows, K, outlier_frac=0.002, outlier_scale=50.0):
    """Laplace(0, 0.05) with a few large channels, fp16."""
    u = torch.rand((rows, K), generator=g, device="cuda")
    s = torch.rand((rows, K), generator=g, device="cuda") - 0.5
    x = (-0.05 * torch.log(u + 1e-9)).copysign_(s)
    ch = torch.randperm(K, generator=g, device="cuda")[:max(1, round(K * outlier_frac))]
    x[:, ch] *= outlier_scale
    return x.half()


def _normal(g, rows, K, std):
    return (torch.randn((rows, K), generator=g, device="cuda") * std).half()


def _inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) + 1)
    if case["kind"] == "linear":
        x = _activations(g, case["M"], case["K"])
        w = _normal(g, case["N"], case["K"], 0.02)
        bias = _normal(g, 1, case["N"], 0.1)[0] if case["bias"] else None
        return x, w, bias
    if case["kind"] == "attention":
        BH, L, L_max = case["heads"] * case["batch"], case["L"], case["L_max"]
        ch = torch.randperm(_D, generator=g, device="cuda")[:3]  # the large key channels

        def kv(rows, scale):
            t = torch.randn((rows, _D), generator=g, device="cuda")
            t[:, ch] *= scale
            return t.half()

        # the query, the caches, the new token's key and value (it goes to position L - 1)
        return kv(BH, 1.0), kv(BH * L_max, 8.0), kv(BH * L_max, 1.0), kv(BH, 8.0), kv(BH, 1.0)
    return _activations(g, case["rows"], case["K"])


def _static_scale(K):
    """The calibrated per-tensor scale: 127 steps up to 2.5 (larger elements saturate)."""
    return 2.5 / 127


# --------------------------------------------------------------------------
# a pass
# --------------------------------------------------------------------------
def _mode(case):
    return Q.ASYMMETRIC if case["mode"] == "asym" else Q.SYMMETRIC


def prepare(case, seed):
    if case["kind"] == "linear":
        x, w, bias = _inputs(case, seed)
        fmt = dict(group_s=case["group_s"], mode=_mode(case), code_bits=case["code_bits"],
                   flag_bits=case["flag_bits"], group_q=case["K"] if case["path"] == "static" else 64)
        ew = Q.encode_weights(w, **fmt)
        wp = Q.prepare_weights(ew) if case["prepared"] else None
        return dict(case=case, x=x, bias=bias, w=ew, wp=wp, fmt=fmt, out=_DTYPES[case["out"]])
    if case["kind"] == "attention":
        q, k, v, k_new, v_new = _inputs(case, seed)
        fmt = dict(group_s=case["group_s"], flag_bits=case["flag_bits"])
        BH = case["heads"] * case["batch"]
        return dict(case=case, q=q, k=Q.quantize(k, **fmt), v=Q.quantize(v, **fmt), k_new=k_new.view(BH, 1, _D),
                    v_new=v_new.view(BH, 1, _D), fmt=fmt, out=_DTYPES[case["out"]])
    x = _inputs(case, seed)
    fmt = dict(group_s=case["group_s"], mode=_mode(case), code_bits=case["code_bits"], flag_bits=case["flag_bits"],
               group_q=case["K"] if case["mode"] == "row" else 64)
    if case["kind"] == "encode":
        return dict(case=case, x=x, fmt=fmt)
    return dict(case=case, e=Q.quantize(x, **fmt))


def run(state):
    case = state["case"]
    if case["kind"] == "linear":
        if case["path"] == "f16":
            return Q.linear_f16(state["x"], state["w"], state["bias"], out_dtype=state["out"],
                                w_prepared=state["wp"])
        if case["path"] == "static":
            a = Q.quantize_static(state["x"], _static_scale(case["K"]), group_s=case["group_s"], group_q=case["K"],
                                  flag_bits=case["flag_bits"])
        else:
            a = Q.quantize(state["x"], **state["fmt"])
        return Q.linear(a, state["w"], state["bias"], out_dtype=state["out"], w_prepared=state["wp"])
    if case["kind"] == "attention":
        L, L_max = case["L"], case["L_max"]
        q = Q.quantize(state["q"], **state["fmt"])
        Q.kv_append(state["k_new"], state["k"], L_max, L - 1)
        Q.kv_append(state["v_new"], state["v"], L_max, L - 1)
        o = Q.attention_decode(q, state["k"], state["v"], L_max, L, _D ** -0.5, out_dtype=state["out"])
        k, v = state["k"], state["v"]
        return dict(o=o, k_codes=k.codes, k_flags=k.flags, k_scales=k.scales, v_codes=v.codes, v_flags=v.flags,
                    v_scales=v.scales)
    if case["kind"] == "encode":
        e = Q.quantize(state["x"], **state["fmt"])
        out = dict(codes=e.codes, flags=e.flags, scales=e.scales)
        if e.zeros is not None:
            out.update(zeros=e.zeros, gsum=e.gsum)
        return out
    return Q.dequantize(state["e"])


def _side_bytes(case, group_q):
    """Bytes per element of one encoded tensor: codes, FLAGs, scales (and zero points, sums)."""
    b = 0.5 + case["flag_bits"] / 8 / case["group_s"] + 2 / group_q
    return b + (5 / group_q if case.get("mode") == "asym" else 0)


def work(case):
    if case["kind"] == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        out = {"float16": 2, "bfloat16": 2, "float32": 4}[case["out"]]
        # fp16 activations and the encoded weights in, the result out
        b = 2 * M * K + _side_bytes(case, K if case["path"] == "static" else 64) * N * K + out * M * N
        return {"bytes": b + (2 * N if case["bias"] else 0), "flops": 2 * M * N * K}
    if case["kind"] == "attention":
        BH, L = case["heads"] * case["batch"], case["L"]
        out = {"float16": 2, "bfloat16": 2, "float32": 4}[case["out"]]
        return {"bytes": 2 * _side_bytes(case, 64) * BH * L * _D + BH * _D * (3 * 2 + out), "flops": 4 * BH * L * _D}
    n = case["rows"] * case["K"]
    return {"bytes": n * (2 + _side_bytes(case, case["K"] if case["mode"] == "row" else 64)), "flops": n}


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------
def _f32(t):
    """Rounded to the nearest 32-bit value, kept in 64 bits."""
    return t.float().double()


def _ints(t, limit):
    return t.round().clamp(-limit, limit)  # round() rounds halves to even


def _encode(x, group_s, mode="sym", code_bits=8, group_q=64, scale=None):
    """Eq. 1 and Eq. 2 on fp16 x [rows, K]: the codes' values v, the 16-bit scales s, the unrounded scales and
    the zero points z, all in 64 bits; v [rows, groups, group_q], the others [rows, groups, 1]."""
    rows, K = x.shape
    xg = x.double().view(rows, K // group_q, group_q)
    top = 32767 if code_bits == 16 else 127
    lo = None
    if scale is not None:
        s = torch.full((rows, K // group_q, 1), scale, dtype=torch.float16, device=x.device)
        full = s.double()
    elif mode == "asym":
        lo = xg.amin(-1, keepdim=True).clamp(max=0)
        hi = xg.amax(-1, keepdim=True).clamp(min=0)
        full = _f32(hi - lo) / 255
        s = full.float().half()
    else:
        full = xg.abs().amax(-1, keepdim=True) / top
        s = full.float().half()
    s = s.double()
    r = torch.where(s > 0, _f32(1 / s), torch.zeros_like(s))
    z = torch.zeros_like(s)
    if lo is not None:
        z = torch.where(s > 0, _f32(-lo * r).round() - 128, z)
    q = _ints(_f32(xg * r).round() + z, top)
    m = q.abs().view(rows, -1, group_s).amax(-1, keepdim=True)
    # FLAG: the bits of the subgroup's largest magnitude above the third
    step = torch.ones_like(m)
    for bit in range(3, 15):
        step = torch.where(m >= 2 ** bit, 2.0 ** (bit - 2), step)
    q = q.view(rows, -1, group_s)
    v = (q.abs() / step).floor() * step * q.sign()
    return v.view(rows, K // group_q, group_q), s, full, z


def _value(e):
    v, s, _, z = e
    return (s * (v - z)).reshape(v.shape[0], -1)


def exact(case, seed):
    if case["kind"] == "linear":
        x, w, bias = _inputs(case, seed)
        gq = case["K"] if case["path"] == "static" else 64
        fmt = dict(group_s=case["group_s"], mode=case["mode"], code_bits=case["code_bits"], group_q=gq)
        wd = _value(_encode(w, **fmt))
        scale = _static_scale(case["K"]) if case["path"] == "static" else None
        y = torch.empty((case["M"], case["N"]), dtype=torch.float64, device="cuda")
        for i in range(0, case["M"], 2048):
            torch.matmul(_value(_encode(x[i:i + 2048], scale=scale, **fmt)), wd.t(), out=y[i:i + 2048])
        return y if bias is None else y.add_(bias.double())
    if case["kind"] == "attention":
        q, k, v, k_new, v_new = _inputs(case, seed)
        BH, L, L_max, gs = case["heads"] * case["batch"], case["L"], case["L_max"], case["group_s"]
        k.view(BH, L_max, _D)[:, L - 1] = k_new
        v.view(BH, L_max, _D)[:, L - 1] = v_new
        qd = _value(_encode(q, gs)).view(BH, 1, _D)
        o = torch.empty((BH, _D), dtype=torch.float64, device="cuda")
        ks = torch.empty((BH * L_max, 2), dtype=torch.float64, device="cuda")
        vs = torch.empty_like(ks)
        for i in range(0, BH, 64):
            n = min(64, BH - i)
            rows = slice(i * L_max, (i + n) * L_max)
            ek, ev = _encode(k[rows], gs), _encode(v[rows], gs)
            ks[rows], vs[rows] = ek[2].view(-1, 2), ev[2].view(-1, 2)
            kd = _value(ek).view(n, L_max, _D)[:, :L]
            vd = _value(ev).view(n, L_max, _D)[:, :L]
            p = torch.softmax(torch.bmm(qd[i:i + n], kd.transpose(1, 2)) * _D ** -0.5, dim=-1)
            o[i:i + n] = torch.bmm(p, vd)[:, 0]
        return dict(o=o, k_codes=None, k_flags=None, k_scales=ks, v_codes=None, v_flags=None, v_scales=vs)
    x = _inputs(case, seed)
    gq = case["K"] if case["mode"] == "row" else 64
    mode = "asym" if case["mode"] == "asym" else "sym"
    step = max(1, 2 ** 24 // case["K"])
    parts = []
    for i in range(0, case["rows"], step):
        e = _encode(x[i:i + step], case["group_s"], mode, case["code_bits"], gq)
        parts.append(e[2].reshape(e[2].shape[0], -1) if case["kind"] == "encode" else _value(e))
    whole = torch.cat(parts)
    if case["kind"] == "decode":
        return whole
    out = dict(codes=None, flags=None, scales=whole)
    if case["mode"] == "asym":
        out.update(zeros=None, gsum=None)
    return out

"""Measured cases of the quantizer: what a program that quantizes attention projections calls.

Four kinds of work, each through the functions of the package:

  chain   one projection from its calibration activations: Hessian, damping, out-channel Hessian,
          both inverse Cholesky factors, then the group loop
  layer   a whole attention layer in one call, activations and weights on the device or in pinned
          host memory
  quant   the group loop alone, on Hessians and factors that the program already has (one Hessian
          serves many settings when bit widths or out-blocks are compared)
  pack    the storage format: codes to the packed bit stream, and back to dequantized weights

Integer weights, scales and zero-points are the product of a layer or a chain; the dequantized
weights (an optional output that says the same again) are asked for by `quant` only.
"""
import torch

import paper_2602_04929_b200 as tb

ADAPT, CD, DYN = 1, 2, 4
DEV = "cuda:0"
SEQ = 2048


def listed():
    return [
        # The smallest call: a 256-wide projection, INT4 per channel, its own SPD out-channel Hessian.
        # 32 dependent group steps on very little data: launches and latency are everything.
        dict(name="chain_256_w4", kind="chain", d=256, heads=1, d_head=256, tokens=2048, bits=4, gq=0, g=8,
             flags=ADAPT | CD, dtype="bf16", hout="spd"),
        # An ordinary query projection, 128 x 2048 tokens, INT2, grid and scale refinement on.
        dict(name="chain_4096_w2", kind="chain", d=4096, heads=32, d_head=128, tokens=262144, bits=2, gq=128, g=32,
             flags=ADAPT | CD, dtype="bf16", hout="proj"),
        # Float activations, ragged token count, a width that is no multiple of the tiles, rows treated as
        # GPTQ does (identity out-channel Hessian) with the grid of a column group searched on arrival.
        dict(name="chain_1920_f32_dyn", kind="chain", d=1920, heads=9, d_head=128, tokens=5003, bits=3, gq=64, g=128,
             flags=DYN, dtype="f32", hout="none"),
        # A grouped-query layer with one input Hessian per value head, INT3, refinement on.
        dict(name="layer_gqa_4096_w3", kind="layer", d=4096, q=32, kv=8, d_head=128, tokens=262144, bits=3, gq=128,
             g=64, flags=ADAPT | CD, with_r=False, per_head_v=True, host=False),
        # A multi-head layer with the propagated-error terms: activations of both paths go in.
        dict(name="layer_mha_4096_r", kind="layer", d=4096, q=32, kv=32, d_head=128, tokens=65536, bits=2, gq=128,
             g=32, flags=ADAPT | CD, with_r=True, per_head_v=False, host=False),
        # The largest: an 8192-wide grouped-query layer, INT2, fixed grid (half the usual 128 sequences).
        dict(name="layer_gqa_8192_w2", kind="layer", d=8192, q=64, kv=8, d_head=128, tokens=131072, bits=2, gq=128,
             g=32, flags=0, with_r=False, per_head_v=True, host=False),
        # A small layer of odd sizes: 13 heads, 3001 tokens, one scale per row, with the propagated error.
        dict(name="layer_1664_odd", kind="layer", d=1664, q=13, kv=13, d_head=128, tokens=3001, bits=4, gq=0, g=16,
             flags=ADAPT, with_r=True, per_head_v=False, host=False),
        # Everything in pinned host memory, as a program with the model on the CPU has it.
        dict(name="layer_host_2048_w4", kind="layer", d=2048, q=32, kv=8, d_head=64, tokens=32768, bits=4, gq=128,
             g=32, flags=ADAPT | CD, with_r=False, per_head_v=True, host=True),
        # The sequential rule (one out-channel at a time) on a key projection: long dependent chains.
        dict(name="quant_1024x4096_g1", kind="quant", d=4096, heads=8, d_head=128, bits=2, gq=128, g=1, flags=0,
             hout="spd", per_head_in=False),
        # A value projection with an input Hessian per head and wide column groups.
        dict(name="quant_1024x2048_perhead", kind="quant", d=2048, heads=8, d_head=128, bits=4, gq=256, g=64,
             flags=ADAPT | CD, hout="spd", per_head_in=True),
        # Rows of an output or feed-forward projection: no out-channel Hessian, all rows at once.
        dict(name="quant_4096x4096_rows", kind="quant", d=4096, heads=1, d_head=4096, bits=4, gq=128, g=4096,
             flags=0, hout="none", per_head_in=False),
        # Packing a weight for storage and unpacking it into dequantized weights.
        dict(name="pack_4096x4096_w3", kind="pack", d=4096, rows=4096, bits=3, gq=128),
    ]


def _log(rng, lo, hi, step):
    """A multiple of `step` between lo and hi, spread over the logarithm."""
    v = lo * (hi / lo) ** rng.random()
    return int(min(hi, max(lo, round(v / step) * step)))


def _settings(rng, d, d_head):
    gqs = [0] + [q for q in (32, 64, 128, 256) if d % q == 0]
    return dict(bits=rng.choice([2, 2, 3, 3, 4, 4, 8]), gq=rng.choice(gqs),
                g=rng.choice([v for v in (4, 8, 16, 32, 64, 128) if d_head % v == 0]),
                flags=rng.choice([0, ADAPT, ADAPT | CD, CD]))


def draw(rng):
    kind = rng.choice(["chain", "chain", "layer", "layer", "quant", "pack"])
    d_head = rng.choice([64, 128])
    if kind == "chain":
        d = _log(rng, 256, 5120, 128)
        c = dict(kind=kind, d=d, heads=rng.randint(1, max(1, min(40, d // d_head))), d_head=d_head,
                 tokens=_log(rng, 1000, 100000, 1), dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]),
                 hout=rng.choice(["proj", "proj", "none"]), **_settings(rng, d, d_head))
        if c["dtype"] == "f32":
            c["tokens"] = min(c["tokens"], 20000)
        return c
    if kind == "layer":
        kv = rng.choice([1, 2, 4, 8])
        rep = rng.choice([1, 2, 4])
        dq = kv * rep * d_head
        d = max(256, dq + 128 * rng.choice([0, 0, 0, 1]))
        with_r = rng.random() < 0.3
        c = dict(kind=kind, d=d, q=kv * rep, kv=kv, d_head=d_head, tokens=_log(rng, 2000, 60000, 1), with_r=with_r,
                 per_head_v=rng.random() < 0.6, host=rng.random() < 0.2, **_settings(rng, d, d_head))
        if dq % 128:                      # the output projection's width is a multiple of 128 too
            c["q"], c["d"] = 2 * c["q"], max(d, 256)
        while c["gq"] and (c["q"] * d_head) % c["gq"]:
            c["gq"] //= 2
        return c
    if kind == "quant":
        d = _log(rng, 256, 6144, 128)
        c = dict(kind=kind, d=d, heads=rng.randint(1, 24), d_head=d_head, hout=rng.choice(["spd", "spd", "none"]),
                 per_head_in=False, **_settings(rng, d, d_head))
        if d <= 2048 and rng.random() < 0.3:
            c["per_head_in"], c["heads"] = True, min(c["heads"], 8)
        return c
    d = _log(rng, 256, 8192, 128)
    return dict(kind="pack", d=d, rows=_log(rng, 64, 8192, 1), bits=rng.randint(2, 8),
                gq=rng.choice([0] + [q for q in (32, 64, 128) if d % q == 0]))


# ------------------------------------------------------------------------------------------ inputs

def _activations(g, n_tok, d, dtype=torch.bfloat16):
    """Heavy-tailed activations: log-normal token scale, a rank-64 common factor, 1 % of the channels x 20."""
    sigma = torch.ones(d, device=DEV)
    sigma[torch.randperm(d, generator=g, device=DEV)[:max(1, d // 100)]] = 20.0
    F = torch.randn((64, d), generator=g, device=DEV) / 8.0
    out = torch.empty((n_tok, d), dtype=dtype, device=DEV)
    for t in range(0, n_tok, 16384):
        n = min(16384, n_tok - t)
        x = torch.randn((n, d), generator=g, device=DEV)
        x.addmm_(torch.randn((n, 64), generator=g, device=DEV), F, alpha=2.0)
        x *= torch.exp(0.5 * torch.randn((n, 1), generator=g, device=DEV))
        out[t:t + n] = x * sigma
    return out


def _deviated(g, x_fp):
    """The quantized path's twin of full-precision activations: a low-rank error and some noise."""
    d = x_fp.shape[1]
    A = torch.randn((d, 32), generator=g, device=DEV) / d ** 0.5
    B = torch.randn((32, d), generator=g, device=DEV) / d ** 0.5
    out = torch.empty_like(x_fp)
    for t in range(0, x_fp.shape[0], 16384):
        x = x_fp[t:t + 16384].float()
        out[t:t + 16384] = x + 0.1 * ((x @ A) @ B) + 0.03 * torch.randn(x.shape, generator=g, device=DEV)
    return out


def _mixed(x, head, out):
    """Attention-weighted inputs of a value head: a causal average with exponential decay inside a sequence."""
    rho = 1.0 - 2.0 ** -(1 + head % 6)
    t = torch.arange(SEQ, device=DEV)
    A = torch.tril(rho ** (t[:, None] - t[None, :]).clamp(min=0).float())
    A = (A / A.sum(1, keepdim=True)).to(torch.bfloat16)
    for s in range(0, x.shape[0], SEQ):
        m = min(SEQ, x.shape[0] - s)
        torch.mm(A[:m, :m], x[s:s + m], out=out[s:s + m])


def _weight(g, rows, d):
    return torch.randn((rows, d), generator=g, device=DEV) * 0.02


def _spd(g, n, k):
    """k symmetric positive definite matrices with eigenvalues from 1 down to 1e-3."""
    q = torch.linalg.qr(torch.randn((k, n, n), generator=g, device=DEV, dtype=torch.float64))[0]
    h = (q * torch.logspace(0, -3, n, device=DEV, dtype=torch.float64)) @ q.transpose(1, 2)
    return (0.5 * (h + h.transpose(1, 2))).float().contiguous()


def _upper_factor(h):
    """U with H^-1 = U^T U, in double, rounded once."""
    low = torch.linalg.cholesky(h.double().flip(-2, -1)).flip(-2, -1)      # H = U' U'^T, U' upper
    eye = torch.eye(h.shape[-1], device=DEV, dtype=torch.float64)
    return torch.linalg.solve_triangular(low, eye.expand_as(low), upper=True).triu().float().contiguous()


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * seed + 17)
    return _PREPARE[case["kind"]](case, g)


def _prepare_chain(c, g):
    d, rows = c["d"], c["heads"] * c["d_head"]
    desc = tb.layer_desc(rows, d, c["heads"], c["d_head"], c["bits"], c["gq"],
                         c["g"] if c["hout"] != "none" else c["d_head"], flags=c["flags"])
    s = dict(kind="chain", case=c, desc=desc, W=_weight(g, rows, d), G=None, Hout=None)
    s["X"] = _activations(g, c["tokens"], d, torch.bfloat16 if c["dtype"] == "bf16" else torch.float32)
    if c["hout"] == "proj":
        s["G"] = _weight(g, rows, d)
    elif c["hout"] == "spd":
        s["Hout"] = _spd(g, c["d_head"], c["heads"])
    s["H"], s["Hsum"] = torch.empty((2, d, d), device=DEV).unbind(0)
    s["out"] = tb.empty_result(desc, DEV)
    s["ws"] = torch.empty(tb.tb_quantize_layer_workspace(desc, False, True), dtype=torch.uint8, device=DEV)
    return s


def _prepare_layer(c, g):
    d, dq, dkv = c["d"], c["q"] * c["d_head"], c["kv"] * c["d_head"]
    W = [_weight(g, dq, d), _weight(g, dkv, d), _weight(g, dkv, d), _weight(g, d, dq)]
    X, Xo, Xfp, Xofp, Xv = _activations(g, c["tokens"], d), _activations(g, c["tokens"], dq), None, None, None
    if c["with_r"]:
        Xfp, Xofp = X, Xo
        X, Xo = _deviated(g, Xfp), _deviated(g, Xofp)
    if c["per_head_v"]:
        Xv = torch.empty((c["kv"],) + X.shape, dtype=X.dtype, device=DEV)
        for h in range(c["kv"]):
            _mixed(X, h, Xv[h])
    desc = tb.attention_desc(d, c["q"], c["kv"], c["d_head"], c["bits"], c["gq"], c["g"], c["tokens"],
                             flags=c["flags"], on_host=c["host"], concurrent=True)
    n_info = tb.tb_attention_layer_info_count(desc, c["per_head_v"])
    info = torch.zeros(n_info, dtype=torch.int32, device="cpu" if c["host"] else DEV)
    if c["host"]:
        X, Xo, Xfp, Xofp, Xv, info = (None if t is None else t.cpu().pin_memory() for t in (X, Xo, Xfp, Xofp, Xv, info))
        W = [w.cpu().pin_memory() for w in W]
        outs = tb.attention_outputs(desc, device=None, pin=True, w_hat=False)
    else:
        outs = tb.attention_outputs(desc, device=DEV, w_hat=False)
    io = tb.attention_io(desc, X, Xo, W, outs, X_fp=Xfp, X_v=Xv, X_o_fp=Xofp, info=info)
    ws = torch.empty(tb.tb_attention_layer_workspace(desc, io), dtype=torch.uint8, device=DEV)
    return dict(kind="layer", desc=desc, io=io, ws=ws, outs=outs, info=info, keep=(X, Xo, Xfp, Xofp, Xv, W))


def _prepare_quant(c, g):
    d, rows = c["d"], c["heads"] * c["d_head"]
    n_hin = c["heads"] if c["per_head_in"] else 1
    g_out = c["g"] if c["hout"] != "none" else c["d_head"]
    desc = tb.layer_desc(rows, d, c["heads"], c["d_head"], c["bits"], c["gq"], g_out, n_hin=n_hin, flags=c["flags"])
    H = torch.empty((n_hin, d, d), device=DEV)
    U = torch.empty_like(H)
    for u in range(n_hin):
        x = _activations(g, 2 * d + 1000, d, torch.float32)
        h = (x.T @ x).div_(x.shape[0])
        h.diagonal().add_(0.01 * h.diagonal().mean())
        H[u], U[u] = h, _upper_factor(h)
    Hout = Uout = None
    if c["hout"] == "spd":
        Hout = _spd(g, c["d_head"], c["heads"])
        Uout = _upper_factor(Hout)
    out = tb.empty_result(desc, DEV)
    ws = torch.empty(tb.tb_quantize_layer_workspace(desc, False, True), dtype=torch.uint8, device=DEV)
    return dict(kind="quant", desc=desc, W=_weight(g, rows, d), H=H, U=U, Hout=Hout, Uout=Uout, out=out, ws=ws)


def _prepare_pack(c, g):
    groups = 1 if c["gq"] == 0 else c["d"] // c["gq"]
    codes = torch.randn((c["rows"], c["d"]), generator=g, device=DEV) * 2 ** c["bits"] / 6 + 2 ** (c["bits"] - 1)
    codes = codes.round().clamp(0, 2 ** c["bits"] - 1).to(torch.uint8)
    scales = 0.01 + 0.01 * torch.rand((c["rows"], groups), generator=g, device=DEV)
    zeros = torch.full((c["rows"], groups), 2 ** (c["bits"] - 1), dtype=torch.int32, device=DEV)
    return dict(kind="pack", case=c, codes=codes, scales=scales, zeros=zeros)


_PREPARE = dict(chain=_prepare_chain, layer=_prepare_layer, quant=_prepare_quant, pack=_prepare_pack)


# ------------------------------------------------------------------------------------------ one pass

def run(state):
    return _RUN[state["kind"]](state)


def _result(out, w_hat):
    r = dict(codes=out.codes, scales=out.scales, zeros=out.zeros, loss=out.loss)
    if w_hat:
        r["w_hat"] = out.w_hat
    return r


def _run_chain(s):
    desc, H = s["desc"], s["H"]
    H.zero_()
    tb.tb_accumulate_hessian(H, s["X"])
    tb.tb_finalize_hessian(H, None, s["X"].shape[0], 0.01, Hsum_out=s["Hsum"])
    Hout = s["Hout"] if s["G"] is None else tb.tb_build_hout(s["G"], s["Hsum"], desc.n_heads, desc.d_head, 0.01)
    Uout = None if Hout is None else tb.tb_factor(Hout)[0]
    U, info = tb.tb_factor(H)
    tb.tb_quantize_layer(desc, s["W"], H, U, Hout, Uout, ws=s["ws"], out=s["out"])
    return dict(_result(s["out"], False), info=info)


def _run_layer(s):
    tb.tb_attention_layer(s["desc"], s["io"], s["ws"])
    return dict(outs=s["outs"], info=s["info"])


def _run_quant(s):
    tb.tb_quantize_layer(s["desc"], s["W"], s["H"], s["U"], s["Hout"], s["Uout"], ws=s["ws"], out=s["out"])
    return _result(s["out"], True)


def _run_pack(s):
    c = s["case"]
    packed = tb.tb_pack_codes(s["codes"], c["bits"])
    _, w_hat, _ = tb.tb_unpack_dequant(packed, s["scales"], s["zeros"], c["d"], c["bits"], c["gq"], want_codes=False)
    return dict(packed=packed, w_hat=w_hat)


_RUN = dict(chain=_run_chain, layer=_run_layer, quant=_run_quant, pack=_run_pack)


# ------------------------------------------------------------------------------------------ work and tolerance

def _hessian_flops(d, tokens):
    return tokens * d * (d + 1.0)


def _factor_flops(d):
    return 2.0 / 3.0 * d ** 3


def _loop_flops(rows, d, d_head, g, gq, with_r, has_hout):
    """Sweep d^2 per row (twice with the propagated error), grid search 16 d (group + 1) and the joint
    compensation (d_head - g) d; with the propagated error W C of every step but the last."""
    f = (2.0 if with_r else 1.0) * d * d + 16.0 * d * ((gq or d) + 1)
    if has_hout:
        f += (d_head - g) * d
        if with_r:
            f += 2.0 * d * d * (d_head // g - 1) / (d_head // g)
    return rows * f


def work(case):
    c = case
    kind, d = c["kind"], c["d"]
    if kind == "pack":
        n = float(c["rows"]) * d
        return {"bytes": n * (1 + 2 * c["bits"] / 8 + 4), "flops": 2.0 * n}
    if kind == "layer":
        dq, dkv, tok = c["q"] * c["d_head"], c["kv"] * c["d_head"], c["tokens"]
        n_v = c["kv"] if c["per_head_v"] else 0
        twins = 2 if c["with_r"] else 1
        weights = float(dq * d + 2 * dkv * d + d * dq)
        flops = _hessian_flops(d, tok) * (1 + n_v) + _hessian_flops(dq, tok)
        flops += _factor_flops(d) * (1 + n_v) + _factor_flops(dq) + _factor_flops(c["d_head"]) * (c["q"] + 2 * c["kv"])
        if c["with_r"]:
            flops += 2.0 * tok * (d * d + dq * dq) + 4.0 * (d ** 3 + dq ** 3)
        for rows, width, hout in ((dq, d, True), (dkv, d, True), (dkv, d, True), (d, dq, False)):
            flops += _loop_flops(rows, width, c["d_head"], c["g"], c["gq"], c["with_r"], hout)
        return {"bytes": 2.0 * tok * (d * (twins + n_v) + dq * twins) + 5.0 * weights, "flops": flops}
    rows = c["heads"] * c["d_head"]
    hout = c["hout"] != "none"
    flops = _loop_flops(rows, d, c["d_head"], c["g"], c["gq"], False, hout)
    if kind == "quant":
        n_hin = c["heads"] if c["per_head_in"] else 1
        return {"bytes": 9.0 * rows * d + 6.0 * n_hin * d * d, "flops": flops}
    size = 2 if c["dtype"] == "bf16" else 4
    flops += _hessian_flops(d, c["tokens"]) + _factor_flops(d)
    if hout:
        flops += _factor_flops(c["d_head"]) * c["heads"]
    return {"bytes": float(size) * c["tokens"] * d + 5.0 * rows * d, "flops": flops}


def tolerance(case):
    """Where Hessians and factors are given, everything that decides a code is carried in double and only the
    float sums of the scale refinement and of the loss differ (scales to 2.5e-7, losses to 1.2e-6).

    From activations on, a code is an integer decision inside an error-feedback chain: where a pre-rounding
    value lies within the rounding of the Hessian's float sums of a boundary, the rest of its row, and through
    the joint compensation the rest of its head, takes another equally valid course.  Measured with the tokens
    in reverse order: up to 1 % of the codes of a projection and 3.3e-2 of its scales (0.9 for one value)."""
    kind = case["kind"]
    if kind == "pack":
        return {"rel": 1e-6, "max": 1e-6, "differ": 0.0}
    if kind == "quant":
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-5}
    return {"rel": 0.03, "max": 0.99, "differ": 0.01}

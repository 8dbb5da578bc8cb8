"""Representative calls of the W4A4KV4 path with their inputs, work, exact results and tolerances.

The shapes are the Llama-3-8B and Llama-3-70B layers of `inputs.py` and the square 4096 layer; token counts run from one
decode token to a 4096-token prefill. Decode steps (up to 128 tokens, one CUDA graph per step, as a decode loop keeps one)
are replayed; prefill, attention and offline calls are issued directly.

    listed()  the fixed cases          draw(rng)  one more case of the same ranges
    prepare   inputs, weights, caches, output buffers (and the graph of a decode step)
    run       one pass; the outputs are the state's own buffers
    exact     the same results in 64 bits with plain torch, rounded to bf16 only where the interface stores bf16
"""
from __future__ import annotations

import functools
import math

import torch

from paper_2410_05265_b200 import binding, inputs
from paper_2410_05265_b200.block import Block, BlockShape

ARCH = {"8b": inputs.LLAMA3_8B, "70b": inputs.LLAMA3_70B}
LAYERS = {"8b": 32, "70b": 80}
D = 128
DEV = "cuda"
THETA = 500000.0
EPS = 1e-5
N_PREFIX = 4  # prefixed outlier tokens
CAL_ROWS = 64  # rows of the calibration batch behind a static step


def listed():
    return [
        # one token of one sequence through a whole layer: the latency of interactive decoding
        dict(name="decode_layer_8b_1021", kind="decode_layer", arch="8b", T=1021),
        # the linear layers of a batched decode step, one token for each of 33 sequences
        dict(name="decode_linears_8b_33", kind="decode_linears", arch="8b", M=33, mode="w4a4"),
        # a small batch on the 70B layer: weight streaming
        dict(name="decode_linears_70b_16", kind="decode_linears", arch="70b", M=16, mode="w4a4"),
        # a full decode batch at the 8-bit activation precision
        dict(name="decode_linears_w4a8_96", kind="decode_linears", arch="8b", M=96, mode="w4a8"),
        # one linear layer on a short prompt: launch latency and a chip that the tiles do not fill
        dict(name="linear_256", kind="prefill_linears", arch="one", M=256, mode="w4a4", row_begin=0),
        # the linear layers of a 2048-token prefill whose first four rows are prefixed tokens
        dict(name="prefill_linears_8b_2048", kind="prefill_linears", arch="8b", M=2048, mode="w4a4", row_begin=4),
        # the same at a length that fills no tile, with per-token dynamic steps
        dict(name="prefill_linears_dyn_1000", kind="prefill_linears", arch="8b", M=1000, mode="dyn", row_begin=0),
        # a short prompt through a whole block
        dict(name="block_8b_515", kind="block", arch="8b", T=515, r3=True),
        # the long prefill of the large model
        dict(name="block_70b_4096", kind="block", arch="70b", T=4096, r3=False),
        # decode attention of a batch with full caches
        dict(name="decode_attn_8x4092", kind="decode_attn", arch="8b", B=8, T=4092, dyn=False, ragged=False),
        # decode attention over ragged sequences whose cached vectors carry their own steps
        dict(name="decode_attn_dyn_6x1500", kind="decode_attn", arch="8b", B=6, T=1500, dyn=True, ragged=True),
        # offline: the layer's weights quantized and its static steps calibrated
        dict(name="quantize_layer_8b", kind="quantize", arch="8b", M=512),
    ]


def draw(rng):
    log = lambda lo, hi: min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))
    kind = rng.choice(["decode_layer", "decode_linears", "decode_linears", "prefill_linears", "prefill_linears", "block", "decode_attn",
                       "decode_attn", "quantize"])
    arch = rng.choice(["8b", "8b", "70b"])
    if kind == "decode_layer":
        return dict(kind=kind, arch=arch, T=log(16, 8192))
    if kind == "decode_linears":
        return dict(kind=kind, arch=arch, M=log(1, 128), mode=rng.choice(["w4a4", "w4a4", "w4a8", "dyn", "asym"]))
    if kind == "prefill_linears":
        M = log(17, 4096)
        arch = rng.choice([arch, arch, "one"])
        return dict(kind=kind, arch=arch, M=M, mode=rng.choice(["w4a4", "w4a4", "w4a8", "dyn", "asym"]), row_begin=rng.choice([0, N_PREFIX]))
    if kind == "block":
        return dict(kind=kind, arch=arch, T=log(17, 4096 if arch == "8b" else 3500), r3=rng.random() < 0.5)
    if kind == "decode_attn":
        B = log(1, 64)
        return dict(kind=kind, arch=arch, B=B, T=log(16, 131072 // B if B > 4 else 32768), dyn=rng.random() < 0.3, ragged=rng.random() < 0.5)
    return dict(kind=kind, arch="8b", M=log(64, 2048))


# ---- inputs -----------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=1)
def _ctx():
    return binding.Context()


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1000003 + 17)


def _randn(g, *shape, scale=1.0, dtype=torch.bfloat16):
    out = torch.empty(shape, dtype=dtype, device=DEV)
    flat = out.view(-1)
    for lo in range(0, flat.numel(), 1 << 27):  # bounded fp32 temporaries
        part = flat[lo: lo + (1 << 27)]
        part.copy_(torch.randn(part.numel(), generator=g, device=DEV).mul_(scale))
    return out


def _activations(g, M, K, row_begin):
    """Layer input: normal values with a log-normal spread over the channels; prefixed rows carry four channels near 1000."""
    sigma = torch.exp(0.5 * torch.randn(K, generator=g, device=DEV))
    x = _randn(g, M + CAL_ROWS, K, dtype=torch.float32).mul_(sigma)
    cal, x = x[M:].to(torch.bfloat16), x[:M].to(torch.bfloat16)
    for t in range(min(row_begin, M)):
        for i, c in enumerate(inputs.outlier_channels(K)):
            x[t, c] = 1000.0 if (t + i) % 2 == 0 else -1000.0
    return x, cal


def _shapes(arch):
    """(N, K, width of the rotation) of the layer's GEMMs, q|k|v and gate|up concatenated."""
    if arch == "one":
        return [(4096, 4096, 4096)]
    a = ARCH[arch]
    h, f = a["hidden"], a["ffn"]
    return [(h + 2 * a["kv_dim"], h, h), (h, h, h), (2 * f, h, h), (h, f, 2048)]


# ---- the path in 64 bits ----------------------------------------------------------------------------------
def _fwht(x, block):
    """Rows of x times the normalised Sylvester matrix on contiguous blocks, float64."""
    M, K = x.shape
    y = x.to(torch.float64).reshape(-1, block)
    h = 1
    while h < block:
        y = y.view(-1, block // (2 * h), 2, h)
        y = torch.stack((y[:, :, 0] + y[:, :, 1], y[:, :, 0] - y[:, :, 1]), 2).reshape(-1, block)
        h *= 2
    return (y / math.sqrt(block)).reshape(M, K)


def _seventh(top):
    """top / 7 in fp32 as a true division (dividing by a Python number multiplies by its reciprocal)."""
    return top / torch.full_like(top, 7.0)


def _weight_codes(W):
    s = _seventh(W.float().abs().amax(1))
    return torch.clamp(torch.round(W.float() / s[:, None]), -8, 7), s


def _codes(y, s, lo, hi):
    return torch.clamp(torch.round(y / s), lo, hi)


def _bf16(x):
    return x.to(torch.bfloat16).to(torch.float64)


def _matmul_codes(a, w):
    """a f64 [M, K] times codes w [N, K] transposed, exact, a few thousand output channels at a time."""
    out = torch.empty((a.shape[0], w.shape[0]), dtype=torch.float64, device=a.device)
    for lo in range(0, w.shape[0], 8192):
        out[:, lo: lo + 8192] = a @ w[lo: lo + 8192].to(torch.float64).T
    return out


def _static_step(y, top):
    return (y.abs().amax() / top).to(torch.float32).reshape(1)


def _asym_step(y):
    mx, mn = float(y.max()), float(y.min())
    s = torch.tensor([(mx - mn) / 15.0], dtype=torch.float32, device=DEV)
    z = torch.tensor([-math.floor(mn / float(s))], dtype=torch.int32, device=DEV)
    return s, z


def _rope(x, pos0, rotate):
    """x f64 [T, H, 128] at positions pos0 .., bf16 result."""
    T = x.shape[0]
    i = torch.arange(D // 2, device=DEV, dtype=torch.float64)
    ang = (pos0 + torch.arange(T, device=DEV, dtype=torch.float64))[:, None] * (THETA ** (-2.0 * i / D))[None]
    c, s = torch.cos(ang)[:, None], torch.sin(ang)[:, None]
    a, b = x[..., : D // 2], x[..., D // 2:]
    y = torch.cat((a * c - b * s, b * c + a * s), -1)
    if rotate:
        y = _fwht(y.reshape(-1, D), D).reshape(y.shape)
    return _bf16(y)


def _attend(q, k, v, visible):
    """q f64 [T, Hq, D], k, v f64 [Hkv, n, D]; query t sees the first visible[t] keys."""
    T, Hq, _ = q.shape
    out = torch.empty_like(q)
    mask = torch.arange(k.shape[1], device=DEV)[None] >= visible[:, None]
    for h in range(Hq):
        kv = h // (Hq // k.shape[0])
        s = (q[:, h] @ k[kv].T) / math.sqrt(D)
        out[:, h] = torch.softmax(s.masked_fill_(mask, -math.inf), -1) @ v[kv]
    return out


def _kv_codes(x, s):
    """x bf16-valued f64 [T, Hkv, D]; the decision is one fp32 division, as the interface states."""
    return torch.clamp(torch.round(x.float() / s.view(1, -1, 1)), -8, 7)


def _layer_exact(x, w, g_attn, g_mlp, a, pk, pv, past_k, past_v, r3, steps=None):
    """One layer in 64 bits. `w`: (codes, s_w) of the four GEMMs; past_k, past_v: codes [Hkv, n, D] of the cache so far.
    With steps=None every static step is taken from this batch (the calibration) and returned."""
    Hq, Hkv = a["n_q_heads"], a["n_kv_heads"]
    qd, kd = Hq * D, Hkv * D
    cal = steps is None
    st = dict(s_a=[]) if cal else steps

    def linear(i, y_in, block):
        y = _fwht(y_in, block)
        if cal:
            st["s_a"].append(_static_step(y, 7.0))
        s = st["s_a"][i].double()
        return _bf16(_matmul_codes(_codes(y, s, -8, 7), w[i][0]) * s * w[i][1].double())

    def norm(v, g):
        return _bf16(v / torch.sqrt((v * v).mean(1, keepdim=True) + EPS) * g.double())

    x = x.double()
    T, n_past = x.shape[0], past_k.shape[1]
    qkv = linear(0, norm(x, g_attn), a["hidden"])
    pos0 = N_PREFIX + n_past
    qk = _rope(qkv[:, : qd + kd].reshape(T, Hq + Hkv, D), pos0, r3)
    q, k, v = qk[:, :Hq], qk[:, Hq:], qkv[:, qd + kd:].reshape(T, Hkv, D)
    if cal:
        st["s_k"], st["s_v"] = (_seventh(t.float().abs().amax((0, 2))) for t in (k, v))
    kc, vc = _kv_codes(k, st["s_k"]), _kv_codes(v, st["s_v"])
    keys = torch.cat((pk.double(), torch.cat((past_k, kc.transpose(0, 1)), 1).double() * st["s_k"].double().view(-1, 1, 1)), 1)
    vals = torch.cat((pv.double(), torch.cat((past_v, vc.transpose(0, 1)), 1).double() * st["s_v"].double().view(-1, 1, 1)), 1)
    att = _bf16(_attend(q, keys, vals, N_PREFIX + n_past + 1 + torch.arange(T, device=DEV)))
    x2 = _bf16(x + linear(1, att.reshape(T, qd), a["hidden"]))
    gu = linear(2, norm(x2, g_mlp), a["hidden"])
    gate, up = gu[:, : a["ffn"]], gu[:, a["ffn"]:]
    y = _bf16(x2 + linear(3, _bf16(gate / (1 + torch.exp(-gate)) * up), 2048))
    return st if cal else y


# ---- prepare / run ----------------------------------------------------------------------------------------
def _graph(call):
    """The step as a decode loop keeps it: one captured graph."""
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        call()
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g


def _linear_inputs(case, seed):
    g = _gen(seed)
    for N, K, block in _shapes(case["arch"]):
        x, cal = _activations(g, case["M"], K, case.get("row_begin", 0))
        W = _randn(g, N, K, scale=0.02)
        y = _fwht(cal, block)
        if case["mode"] == "asym":
            yield x, W, block, _asym_step(y)
        else:
            yield x, W, block, (None if case["mode"] == "dyn" else _static_step(y, 127.0 if case["mode"] == "w4a8" else 7.0))


def _prepare_linears(case, seed):
    ctx, M, mode = _ctx(), case["M"], case["mode"]
    layers = []
    for x, W, block, step in _linear_inputs(case, seed):
        N, K = W.shape
        wq, s_w = ctx.quant_weights(W)
        lay = dict(x=x, block=block, step=step, wq=wq, s_w=s_w, out=torch.zeros((M, N), dtype=torch.bfloat16, device=DEV))
        if mode == "w4a8":
            lay["xq"] = torch.zeros((M, K), dtype=torch.int8, device=DEV)
        else:
            lay["xq"] = torch.zeros((M, K // 2), dtype=torch.uint8, device=DEV)
        if mode == "dyn":
            lay["s_tok"] = torch.zeros(M, device=DEV)
        if mode == "asym":
            lay["wsum"] = ctx.weight_code_sums(wq)
        layers.append(lay)
    st = dict(kind=case["kind"], mode=mode, row_begin=case.get("row_begin", 0), layers=layers)
    if case["kind"] == "decode_linears":
        st["graph"] = _graph(lambda: _run_linears(st))
    return st


def _run_linears(st):
    ctx, mode, rb = _ctx(), st["mode"], st["row_begin"]
    outs = []
    for lay in st["layers"]:
        x, block, step, wq, s_w, xq, out = (lay[n] for n in ("x", "block", "step", "wq", "s_w", "xq", "out"))
        if mode == "w4a4":
            ctx.hadamard_quant_act(x, block, step, rb, out=xq)
            ctx.w4a4_gemm(xq, wq, step, s_w, rb, out=out)
        elif mode == "w4a8":
            ctx.hadamard_quant_act8(x, block, step, rb, out=xq)
            ctx.w4a8_gemm(xq, wq, step, s_w, rb, out=out)
        elif mode == "dyn":
            ctx.dyn_hadamard_quant_act(x, block, 1.0, rb, s_tok=lay["s_tok"], out=xq)
            ctx.w4a4_gemm_rows(xq, wq, lay["s_tok"], s_w, rb, out=out)
            outs.append(lay["s_tok"])
        else:
            ctx.hadamard_quant_act_asym(x, block, step[0], step[1], rb, out=xq)
            ctx.w4a4_gemm_asym(xq, wq, step[0], step[1], s_w, lay["wsum"], rb, out=out)
        outs += [xq, out]
    return outs


def _exact_linears(case, seed):
    outs, rb, mode = [], case.get("row_begin", 0), case["mode"]
    for x, W, block, step in _linear_inputs(case, seed):
        y = _fwht(x, block)
        w, s_w = _weight_codes(W)
        if mode == "dyn":
            s = y.abs().amax(1) / 7.0
            a, scale = _codes(y, s[:, None], -8, 7), s[:, None]
            s_out = s.clone()
            s_out[:rb] = 0
            outs.append(s_out)
        elif mode == "asym":
            s, z = step[0].double(), step[1].double()
            a, scale = torch.clamp(torch.round(y / s) + z, 0, 15) - z, s
        else:
            top = 128 if mode == "w4a8" else 8
            scale = step.double()
            a = _codes(y, scale, -top, top - 1)
        out = _matmul_codes(a, w) * scale * s_w.double()
        out[:rb] = 0
        outs += [None, out]
    return outs


def _layer_inputs(case, seed, T):
    a, g = ARCH[case["arch"]], _gen(seed)
    # o and down are drawn smaller by sqrt(2 x layers) and x has the spread of a residual stream that many layers have added to:
    # a block's update is small beside what it is added to, so a code that a different rounding flips stays a small error
    into_stream = 0.02 / math.sqrt(2 * LAYERS[case["arch"]])
    W = [_randn(g, N, K, scale=s) for (N, K, _), s in zip(_shapes(case["arch"]), (0.02, into_stream, 0.02, into_stream))]
    g_attn, g_mlp = ((1.0 + 0.1 * torch.randn(a["hidden"], generator=g, device=DEV)).to(torch.bfloat16) for _ in range(2))
    pk, pv = (_randn(g, a["n_kv_heads"], N_PREFIX, D, dtype=torch.float16) for _ in range(2))
    x, cal = (t * 8 for t in _activations(g, T, a["hidden"], 0))
    none = torch.zeros((a["n_kv_heads"], 0, D), device=DEV)
    steps = _layer_exact(cal, [_weight_codes(w) for w in W], g_attn, g_mlp, a, pk, pv, none, none, case.get("r3", False))
    return a, g, W, g_attn, g_mlp, pk, pv, x, steps


def _layer_state(case, seed, T, t_max):
    a, g, W, g_attn, g_mlp, pk, pv, x, steps = _layer_inputs(case, seed, T)
    shape = BlockShape(a["hidden"], a["n_q_heads"], a["n_kv_heads"], a["ffn"], rope_theta=THETA, eps=EPS, r3=case.get("r3", False))
    blk = Block(_ctx(), shape, *W, g_attn, g_mlp, pk, pv, t_max)
    for dst, src in zip(blk.s_a, steps["s_a"]):
        dst.copy_(src)
    blk.s_k.copy_(steps["s_k"])
    blk.s_v.copy_(steps["s_v"])
    return g, blk, x


def _past(g, a, T):
    """Codes of a cache of T tokens as bf16 keys and values of spread 2.6 steps leave them, [Hkv, T, D]."""
    return [torch.clamp(torch.round(2.6 * torch.randn((a["n_kv_heads"], T, D), generator=g, device=DEV)), -8, 7) for _ in range(2)]


def _pack(c):
    c = c.to(torch.int16)
    return ((c[..., 0::2] & 15) | ((c[..., 1::2] & 15) << 4)).to(torch.uint8)


def _prepare_decode_layer(case, seed):
    T = case["T"]
    g, blk, x = _layer_state(case, seed, 1, T + 64)
    for dst, c in zip((blk.kq, blk.vq), _past(g, ARCH[case["arch"]], T)):
        dst[0, :, :T] = _pack(c)
    blk._buffers(1, x.device)
    cache = blk._cache()
    st = dict(kind="decode_layer", blk=blk, x=x, T=T, start=torch.full((1,), T, dtype=torch.int32, device=DEV),
              ws=_ctx().decode_attn_workspace(cache), cache=cache)
    st["graph"] = _graph(lambda: _run_decode_layer(st))
    return st


def _run_decode_layer(st):
    ctx, blk, x, cache = _ctx(), st["blk"], st["x"], st["cache"]
    s, b, a = blk.shape, blk.buf, blk.s_a
    blk.length.copy_(st["start"])  # the step can be repeated: it always appends at the same place
    ctx.rmsnorm_hadamard_quant_act(x, blk.g_attn, s.eps, a[0], out=b["xq_h"])
    ctx.w4a4_gemm(b["xq_h"], blk.wq_qkv, a[0], blk.sw_qkv, out=b["qkv"])
    qk = b["qkv"][:, : s.q_dim + s.kv_dim].unflatten(1, (s.n_q_heads + s.n_kv_heads, s.head_dim))
    ctx.rope(qk, blk.n_prefix + st["T"], s.rope_theta, out=qk)
    k = b["qkv"][:, s.q_dim: s.q_dim + s.kv_dim].view(1, 1, s.n_kv_heads, s.head_dim)
    v = b["qkv"][:, s.q_dim + s.kv_dim:].view(1, 1, s.n_kv_heads, s.head_dim)
    ctx.kv4_append_decode_attn(cache, k, v, qk[:, : s.n_q_heads], 1.0 / math.sqrt(s.head_dim), st["ws"], out=b["attn"])
    ctx.hadamard_quant_act(b["attn"].view(1, s.q_dim), s.had_block(s.q_dim), a[1], out=b["xq_a"])
    ctx.w4a4_gemm(b["xq_a"], blk.wq_o, a[1], blk.sw_o, out=b["o"])
    ctx.residual_add(x, b["o"], out=b["x2"])
    ctx.rmsnorm_hadamard_quant_act(b["x2"], blk.g_mlp, s.eps, a[2], out=b["xq_h"])
    ctx.w4a4_gemm(b["xq_h"], blk.wq_gu, a[2], blk.sw_gu, out=b["gu"])
    ctx.swiglu_hadamard_quant_act(b["gu"][:, : s.ffn], b["gu"][:, s.ffn:], s.had_block(s.ffn), a[3], out=b["xq_f"])
    ctx.w4a4_gemm(b["xq_f"], blk.wq_down, a[3], blk.sw_down, out=b["d"])
    ctx.residual_add(b["x2"], b["d"], out=b["y"])
    return _outputs(st)


def _attn_inputs(case, seed):
    a, g = ARCH[case["arch"]], _gen(seed)
    B, T, Hkv = case["B"], case["T"], a["n_kv_heads"]
    k, v = (_randn(g, B, T, Hkv, D) for _ in range(2))
    if case["dyn"]:  # vectors of different magnitudes, which is what their own steps are for
        for t in (k, v):
            t.mul_(torch.exp2(torch.randint(-1, 2, (B, T, Hkv, 1), generator=g, device=DEV).to(torch.bfloat16)))
    q = _randn(g, B, a["n_q_heads"], D)
    pk, pv = (_randn(g, Hkv, N_PREFIX, D, dtype=torch.float16) for _ in range(2))
    n = torch.randint(max(1, T // 2), T + 1, (B,), generator=g, device=DEV) if case["ragged"] else torch.full((B,), T, device=DEV)
    return a, k, v, q, pk, pv, n.to(torch.int32)


def _prepare_attn(case, seed):
    a, k, v, q, pk, pv, n = _attn_inputs(case, seed)
    ctx, B, T, Hkv = _ctx(), case["B"], case["T"], a["n_kv_heads"]
    kq = torch.zeros((B, Hkv, T, D // 2), dtype=torch.uint8, device=DEV)
    vq = torch.zeros_like(kq)
    length = torch.zeros(B, dtype=torch.int32, device=DEV)
    steps = {}
    if case["dyn"]:
        steps = dict(sk_tok=torch.ones((B, Hkv, T), device=DEV), sv_tok=torch.ones((B, Hkv, T), device=DEV))
    s_k, s_v = (None, None) if case["dyn"] else (_seventh(t.float().abs().amax((0, 1, 3))) for t in (k, v))
    cache = binding.KV4Cache(pk, pv, kq, vq, s_k, s_v, length, a["n_q_heads"], **steps)
    ctx.kv4_append(cache, k, v)
    length.copy_(n)
    return dict(kind="decode_attn", cache=cache, q=q, ws=ctx.decode_attn_workspace(cache), out=torch.empty_like(q))


def _exact_attn(case, seed):
    a, k, v, q, pk, pv, n = _attn_inputs(case, seed)
    out = torch.empty(q.shape, dtype=torch.float64, device=DEV)
    if not case["dyn"]:
        s_k, s_v = (_seventh(t.float().abs().amax((0, 1, 3))).view(1, -1, 1) for t in (k, v))
    for b in range(case["B"]):
        kb, vb = k[b, : int(n[b])].float(), v[b, : int(n[b])].float()
        if case["dyn"]:
            s_k, s_v = (_seventh(t.abs().amax(2, keepdim=True)) for t in (kb, vb))
        kd, vd = (torch.clamp(torch.round(t / s), -8, 7).double() * s.double() for t, s in ((kb, s_k), (vb, s_v)))
        keys, vals = torch.cat((pk.double(), kd.transpose(0, 1)), 1), torch.cat((pv.double(), vd.transpose(0, 1)), 1)
        out[b] = _attend(q[b: b + 1].double(), keys, vals, torch.tensor([keys.shape[1]], device=DEV))[0]
    return [out]


def _quantize_inputs(case, seed):
    g = _gen(seed)
    for N, K, block in _shapes(case["arch"]):
        yield _randn(g, N, K, scale=0.02), _activations(g, case["M"], K, N_PREFIX)[0], block


def _prepare_quantize(case, seed):
    layers = []
    for W, x, block in _quantize_inputs(case, seed):
        N, K = W.shape
        layers.append(dict(W=W, x=x, block=block, out=(torch.empty((N, K // 2), dtype=torch.uint8, device=DEV), torch.empty(N, device=DEV)),
                           s_a=torch.zeros(1, device=DEV)))
    return dict(kind="quantize", layers=layers)


def _run_quantize(st):
    ctx, outs = _ctx(), []
    for lay in st["layers"]:
        ctx.quant_weights(lay["W"], out=lay["out"])
        ctx.calib_act_scale(lay["x"], lay["block"], N_PREFIX, s_a=lay["s_a"].zero_())
        outs += [*lay["out"], lay["s_a"]]
    return outs


def _exact_quantize(case, seed):
    outs = []
    for W, x, block in _quantize_inputs(case, seed):
        outs += [None, W.double().abs().amax(1) / 7.0, (_fwht(x[N_PREFIX:], block).abs().amax() / 7.0).reshape(1)]
    return outs


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("decode_linears", "prefill_linears"):
        return _prepare_linears(case, seed)
    if kind == "decode_layer":
        return _prepare_decode_layer(case, seed)
    if kind == "block":
        _, blk, x = _layer_state(case, seed, case["T"], case["T"])
        return dict(kind=kind, blk=blk, x=x)
    return _prepare_attn(case, seed) if kind == "decode_attn" else _prepare_quantize(case, seed)


def _outputs(st):
    if st["kind"] == "decode_layer":
        blk = st["blk"]
        return [blk.buf["y"], blk.kq, blk.vq, blk.length]
    return [t for lay in st["layers"] for t in (([lay["s_tok"]] if st["mode"] == "dyn" else []) + [lay["xq"], lay["out"]])]


def run(st):
    kind = st["kind"]
    if "graph" in st:
        st["graph"].replay()
        return _outputs(st)
    if kind == "prefill_linears":
        return _run_linears(st)
    if kind == "block":
        blk = st["blk"]
        y = blk.forward(st["x"])
        return [y, blk.kq, blk.vq, blk.length]
    if kind == "decode_attn":
        return [_ctx().decode_attn(st["cache"], st["q"], 1.0 / math.sqrt(D), st["ws"], out=st["out"])]
    return _run_quantize(st)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("decode_linears", "prefill_linears"):
        return _exact_linears(case, seed)
    if kind in ("block", "decode_layer"):
        T = case["T"] if kind == "block" else 1
        a, g, W, g_attn, g_mlp, pk, pv, x, steps = _layer_inputs(case, seed, T)
        past = _past(g, a, 0 if kind == "block" else case["T"])
        y = _layer_exact(x, [_weight_codes(w) for w in W], g_attn, g_mlp, a, pk, pv, *past, case.get("r3", False), steps)
        return [y, None, None, None]
    return _exact_attn(case, seed) if kind == "decode_attn" else _exact_quantize(case, seed)


# ---- work and tolerances ----------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind in ("decode_linears", "prefill_linears", "quantize"):
        n_bytes = flops = 0
        M = case["M"] - case.get("row_begin", 0)
        for N, K, block in _shapes(case["arch"]):
            if kind == "quantize":
                n_bytes += 2 * N * K + N * K // 2 + 4 * N + 2 * (M - N_PREFIX) * K
                flops += (M - N_PREFIX) * K * math.log2(block)
            else:
                code = K if case["mode"] == "w4a8" else K // 2
                n_bytes += 2 * M * K + M * code + N * K // 2 + 4 * N + 2 * M * N
                flops += 2 * M * N * K + M * K * math.log2(block)
        return {"bytes": n_bytes, "flops": flops}
    a = ARCH[case["arch"]]
    Hq, Hkv = a["n_q_heads"], a["n_kv_heads"]
    if kind == "decode_attn":
        keys = case["B"] * case["T"] * (0.75 if case["ragged"] else 1.0)
        return {"bytes": keys * Hkv * (D + (8 if case["dyn"] else 0)) + 4 * Hkv * N_PREFIX * D + 4 * case["B"] * Hq * D,
                "flops": 4 * (keys + case["B"] * N_PREFIX) * Hq * D}
    T = case["T"] if kind == "block" else 1
    n_bytes = 4 * T * a["hidden"] + sum(N * K // 2 + 4 * N for N, K, _ in _shapes(case["arch"])) + 4 * Hkv * N_PREFIX * D
    flops = sum(2 * T * N * K for N, K, _ in _shapes(case["arch"]))
    if kind == "block":
        n_bytes += T * Hkv * D
        flops += 4 * D * Hq * (T * (T + 1) // 2 + T * N_PREFIX)
    else:
        n_bytes += case["T"] * Hkv * D
        flops += 4 * D * Hq * (case["T"] + N_PREFIX)
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "quantize":
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}  # fp32 maxima; the codes are one IEEE division each
    if kind == "decode_attn":
        return {"rel": 7e-3, "max": 2e-2}  # bf16 outputs
    if kind in ("block", "decode_layer"):
        return {"rel": 2.5e-2, "max": 0.4, "differ": 2e-3}  # codes next to a tie flip, and what follows carries it
    return {"rel": 7e-3, "max": 0.2, "differ": 2e-4}  # bf16 outputs; a code next to a tie may flip

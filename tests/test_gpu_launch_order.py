"""Stream order of the calls under programmatic dependent launch: calls enqueued back to back give bit for bit what the same
calls give with a synchronisation between them."""
import math

import numpy as np
import pytest
import torch

from oracle import pq_oracle as orc
from helpers import to_np
from paper_2410_05265_b200 import inputs

pytestmark = pytest.mark.gpu
D = 128


@pytest.fixture(scope="module")
def ctx():
    from paper_2410_05265_b200 import binding

    c = binding.Context()
    yield c
    c.check()
    c.close()


@pytest.mark.parametrize("T", [1, 17, 64])
@pytest.mark.parametrize("rows", [1, 24])
@pytest.mark.parametrize("writer", ["rope_kv4_append", "kv4_append_decode_attn"])
def test_cache_written_three_launches_back_is_seen_by_the_decode_step(ctx, T, rows, writer):
    """writer -> rotate + quantize -> GEMM of few rows -> one-launch decode step on the same sequence. The two calls between let
    their successors start early (1 row: streaming GEMM, 24 rows: split-K GEMM), the decode step reads lengths and cache rows ahead of its
    wait. Every pass writes other contents over the rows of the pass before."""
    from paper_2410_05265_b200 import binding

    Hq, Hkv, P, Tmax, K, N = 8, 2, 4, 256, 4096, 4096
    pk, pv = inputs.prefix_kv(Hkv, P, D, 0, "k", 1.0).cuda(), inputs.prefix_kv(Hkv, P, D, 0, "v", 1.0).cuda()
    s = torch.full((Hkv,), 0.4, device="cuda")
    s_a = torch.full((1,), 0.3, device="cuda")
    wq, s_w = ctx.quant_weights(inputs.weights(N, K, seed=2).cuda())
    x = inputs.activations(rows, K, seed=0).cuda()
    g = torch.Generator(device="cuda").manual_seed(T * 100 + rows)
    rand = lambda *sh: torch.randn(sh, generator=g, device="cuda").to(torch.bfloat16)
    passes = [dict(qkv=rand(T, (Hq + 2 * Hkv) * D), k=rand(2, 1, 1, Hkv, D), v=rand(2, 1, 1, Hkv, D), q=rand(2, 1, Hq, D)) for _ in range(8)]

    def run(sync):
        cache = binding.KV4Cache(pk, pv, torch.zeros((1, Hkv, Tmax, D // 2), dtype=torch.uint8, device="cuda"),
                                 torch.zeros((1, Hkv, Tmax, D // 2), dtype=torch.uint8, device="cuda"), s, s,
                                 torch.zeros(1, dtype=torch.int32, device="cuda"), Hq)
        ws = ctx.decode_attn_workspace(cache)
        xq = torch.empty((rows, K // 2), dtype=torch.uint8, device="cuda")
        out = torch.empty((rows, N), dtype=torch.bfloat16, device="cuda")
        attn = torch.empty((len(passes), 2, 1, Hq, D), dtype=torch.bfloat16, device="cuda")
        qkv = [p["qkv"].clone() for p in passes]
        torch.cuda.synchronize()
        step = torch.cuda.synchronize if sync else (lambda: None)
        for i, p in enumerate(passes):
            if writer == "rope_kv4_append":
                cache.length.zero_()
                step()
                ctx.rope_kv4_append(cache, 0, qkv[i], P, 500000.0)
            else:
                if i == 0:
                    cache.length.fill_(T)
                    step()
                ctx.kv4_append_decode_attn(cache, p["k"][0], p["v"][0], p["q"][0], 1 / math.sqrt(D), ws, out=attn[i, 0])
            step()
            ctx.hadamard_quant_act(x, K, s_a, out=xq)
            step()
            ctx.w4a4_gemm(xq, wq, s_a, s_w, out=out)
            step()
            ctx.kv4_append_decode_attn(cache, p["k"][1], p["v"][1], p["q"][1], 1 / math.sqrt(D), ws, out=attn[i, 1])
            step()
        ctx.check()
        first = 1 if writer == "rope_kv4_append" else 0  # attn[:, 0] is written by the other writer only
        return cache.kq, cache.vq, cache.length, out, attn[:, first:].contiguous()

    want, got = run(True), run(False)
    for name, a, b in zip(("keys", "values", "lengths", "GEMM", "attention"), want, got):
        assert torch.equal(a, b), f"{name} differ from the synchronised calls"
    assert int(got[2]) == (T + 1 if writer == "rope_kv4_append" else T + 16)


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M,N,K", [(1, 4096, 4096), (16, 5120, 4096), (24, 4096, 4096), (96, 4096, 4096), (200, 4096, 4096),
                                   (140, 8448, 1024), (300, 4200, 1024)])
def test_weights_written_just_before_reach_two_gemms_in_a_row(ctx, mode, M, N, K):
    """quantize weights (and sum their codes) -> rotate + quantize -> GEMM -> GEMM on other weights of the same quantizer call, back
    to back: the streaming, split-K and tensor-memory pair kernels request weights ahead of the wait for their predecessor, the first two let
    their successors start early (up to 32 tokens). The buffers are overwritten in every pass: stale weights, sums or tokens would show."""
    x = [inputs.activations(M, K, seed=s).cuda() for s in range(3)]
    W = [inputs.weights(2 * N, K, seed=2 + s).cuda() for s in range(3)]
    wq = torch.zeros((2 * N, K // 2), dtype=torch.uint8, device="cuda")
    s_w, wsum = torch.zeros(2 * N, device="cuda"), torch.zeros(2 * N, dtype=torch.int32, device="cuda")
    xq = torch.zeros((M, K if mode == "w4a8" else K // 2), dtype=torch.int8 if mode == "w4a8" else torch.uint8, device="cuda")
    s_a, s_tok = torch.full((1,), 0.02 if mode == "w4a8" else 0.3, device="cuda"), torch.full((M,), 0.3, device="cuda")
    z = torch.full((1,), 5, dtype=torch.int32, device="cuda")
    out = torch.zeros((2, M, N), dtype=torch.bfloat16, device="cuda")
    acc = torch.zeros((3, 2, M, N), dtype=torch.int32, device="cuda")
    seen = []
    torch.cuda.synchronize()
    for i in range(3):
        ctx.quant_weights(W[i], out=(wq, s_w))
        if mode == "asym":
            assert ctx.lib.pq_weight_code_sums(ctx.h, wq.data_ptr(), 2 * N, K, wsum.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
            ctx.hadamard_quant_act_asym(x[i], K, s_a, z, out=xq)
        elif mode == "w4a8":
            ctx.hadamard_quant_act8(x[i], K, s_a, out=xq)
        elif mode == "rows":
            ctx.hadamard_quant_act_rows(x[i], K, s_tok, out=xq)
        else:
            ctx.hadamard_quant_act(x[i], K, s_a, out=xq)
        for h in range(2):
            rows = slice(h * N, (h + 1) * N)
            kw = dict(out=out[h], acc_dbg=acc[i, h])
            if mode == "asym":
                ctx.w4a4_gemm_asym(xq, wq[rows], s_a, z, s_w[rows], wsum[rows], **kw)
            elif mode == "w4a8":
                ctx.w4a8_gemm(xq, wq[rows], s_a, s_w[rows], **kw)
            elif mode == "rows":
                ctx.w4a4_gemm_rows(xq, wq[rows], s_tok, s_w[rows], **kw)
            else:
                ctx.w4a4_gemm(xq, wq[rows], s_a, s_w[rows], **kw)
        seen.append((xq.clone(), wq.clone(), wsum.clone()))
    ctx.check()
    for i, (xc, wc, sums) in enumerate(seen):
        ref = (orc.gemm_i8i4 if mode == "w4a8" else orc.gemm_i4)(to_np(xc), to_np(wc))
        if mode == "asym":
            codes = orc.unpack_int4(to_np(wc)).astype(np.int64).sum(1)
            assert np.array_equal(to_np(sums), codes)
            ref = ref - (5 - 8) * codes[None]
        got = to_np(acc[i])
        assert np.array_equal(np.concatenate([got[0], got[1]], 1), ref), f"pass {i}"


@pytest.mark.parametrize("how", ["dynamic, two launches", "dynamic, one launch", "dynamic, a row per CTA", "calibrated", "calibrated, 8 bits", "zero point"])
@pytest.mark.parametrize("M,N", [(1, 4096), (2, 4096), (3, 4096), (4, 1024), (8, 4096), (12, 1024), (16, 4096), (24, 1024), (96, 4096), (200, 1024), (140, 8264)])
def test_steps_and_codes_written_just_before_are_the_ones_used(ctx, how, M, N):
    """step -> codes -> GEMM, every one reading what the launch before it wrote, replayed as one graph and called back to back, against
    the calls with a synchronisation between them: steps, codes, sums and outputs bit for bit, with other activations every time."""
    K = 4096 if how == "dynamic, one launch" else 6144
    # one block of 4096 or three of 2048: steps and codes from one launch; blocks of 1024: from two
    block = K if K == 4096 else 1024 if how == "dynamic, two launches" else 2048
    bits8 = how == "calibrated, 8 bits"
    g = torch.Generator(device="cuda").manual_seed(M)
    wq = torch.randint(0, 256, (N, K // 2), dtype=torch.uint8, device="cuda", generator=g)
    s_w, wsum = torch.full((N,), 1e-3, device="cuda"), ctx.weight_code_sums(wq)
    xs = [(torch.randn((M, K), generator=g, device="cuda") * 3.0**i).to(torch.bfloat16) for i in range(5)]
    x, s_tok, s_a = torch.zeros_like(xs[0]), torch.zeros(M, device="cuda"), torch.zeros(1, device="cuda")
    z = torch.full((1,), 6, dtype=torch.int32, device="cuda")
    xq = torch.zeros((M, K if bits8 else K // 2), dtype=torch.int8 if bits8 else torch.uint8, device="cuda")
    out, acc = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda"), torch.zeros((M, N), dtype=torch.int32, device="cuda")

    def chain(step):
        kw = dict(out=out, acc_dbg=acc)
        if how.startswith("dynamic"):
            if step is not None and how != "dynamic, one launch":  # two launches, apart
                ctx.dyn_act_scale(x, block, out=s_tok)
                step()
                ctx.hadamard_quant_act_rows(x, block, s_tok, out=xq)
            else:
                ctx.dyn_hadamard_quant_act(x, block, 1.0, 0, s_tok=s_tok, out=xq)
            if step is not None:
                step()
            ctx.w4a4_gemm_rows(xq, wq, s_tok, s_w, **kw)
            return
        s_a.zero_()
        calib, quant, gemm = ((ctx.calib_act_scale8, ctx.hadamard_quant_act8, ctx.w4a8_gemm) if bits8 else
                              (ctx.calib_act_scale, ctx.hadamard_quant_act, ctx.w4a4_gemm))
        calib(x, block, 0, s_a=s_a)
        if step is not None:
            step()
        if how == "zero point":
            ctx.hadamard_quant_act_asym(x, block, s_a, z, out=xq)
        else:
            quant(x, block, s_a, out=xq)
        if step is not None:
            step()
        if how == "zero point":
            ctx.w4a4_gemm_asym(xq, wq, s_a, z, s_w, wsum, **kw)
        else:
            gemm(xq, wq, s_a, s_w, **kw)

    state = lambda: [t.clone() for t in (s_tok, s_a, xq, acc, out)]
    want = []
    for v in xs:
        x.copy_(v)
        torch.cuda.synchronize()
        chain(torch.cuda.synchronize)
        torch.cuda.synchronize()
        want.append(state())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(None)
    for name, call in (("graph", graph.replay), ("stream", lambda: chain(None))):
        for i in (0, 1, 2, 3, 4, 0, 3, 1):
            x.copy_(xs[i])
            torch.cuda.synchronize()
            call()
            torch.cuda.synchronize()
            for what, a, b in zip(("per-token steps", "step", "codes", "sums", "outputs"), state(), want[i]):
                assert torch.equal(a, b), f"{what}, {name}, input {i}"
    ctx.check()


@pytest.mark.parametrize("T", [1, 200])
def test_query_and_token_written_just_before_reach_the_decode_step(ctx, T):
    """residual add (writes q, k, v of the step) -> one-launch decode step, in a graph, against the calls apart."""
    from paper_2410_05265_b200 import binding

    Hq, Hkv, Tmax = 8, 2, 256
    n = (Hq + 2 * Hkv) * D
    g = torch.Generator(device="cuda").manual_seed(T)
    rand = lambda *sh: torch.randn(sh, generator=g, device="cuda").to(torch.bfloat16)
    kq = torch.randint(0, 256, (1, Hkv, Tmax, D // 2), dtype=torch.uint8, device="cuda", generator=g)
    s = torch.full((Hkv,), 0.3, device="cuda")
    cache = binding.KV4Cache(rand(Hkv, 4, D).half(), rand(Hkv, 4, D).half(), kq, kq.clone(), s, s, torch.zeros(1, dtype=torch.int32, device="cuda"), Hq)
    ws = ctx.decode_attn_workspace(cache)
    base, a, y, out = rand(n), torch.zeros(n, dtype=torch.bfloat16, device="cuda"), torch.zeros(n, dtype=torch.bfloat16, device="cuda"), rand(1, Hq, D)
    steps = [rand(n) for _ in range(5)]

    def chain(sync):
        ctx.residual_add(a, base, out=y)
        if sync:
            torch.cuda.synchronize()
        ctx.kv4_append_decode_attn(cache, y[Hq * D: (Hq + Hkv) * D].view(1, 1, Hkv, D), y[(Hq + Hkv) * D:].view(1, 1, Hkv, D), y[: Hq * D].view(1, Hq, D),
                                   1 / math.sqrt(D), ws, out=out)

    def run(call):
        res = []
        for v in steps:
            a.copy_(v)
            cache.length.fill_(T)
            torch.cuda.synchronize()
            call()
            torch.cuda.synchronize()
            res.append((out.clone(), cache.kq.clone(), cache.vq.clone(), cache.length.clone()))
        return res

    want = run(lambda: chain(True))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(False)
    for call in (graph.replay, lambda: chain(False)):
        for w, r in zip(want, run(call)):
            assert all(torch.equal(p, q) for p, q in zip(w, r))
    ctx.check()


@pytest.mark.parametrize("dyn", [False, True])
@pytest.mark.parametrize("B,Tmax", [(1, 256), (8, 256), (1, 9000)])
def test_plain_decode_attention_straight_behind_the_append(ctx, dyn, B, Tmax):
    """residual add (writes the step's k and v) -> append -> plain decode attention -> residual add over its output, in a graph and called
    back to back, against the calls apart: lengths, cache rows and (with steps per vector) the steps are the ones just written. One
    cluster per (sequence, head) pair and, in the long cache, several."""
    from paper_2410_05265_b200 import binding

    Hq, Hkv, P, T0 = 8, 2, 4, 130
    g = torch.Generator(device="cuda").manual_seed(B + Tmax)
    rand = lambda *sh: torch.randn(sh, generator=g, device="cuda").to(torch.bfloat16)
    pk, pv = rand(Hkv, P, D).half(), rand(Hkv, P, D).half()
    codes = torch.randint(0, 256, (2, B, Hkv, Tmax, D // 2), dtype=torch.uint8, device="cuda", generator=g)
    s = torch.full((Hkv,), 0.3, device="cuda")
    steps = dict(sk_tok=torch.full((B, Hkv, Tmax), 0.3, device="cuda"), sv_tok=torch.full((B, Hkv, Tmax), 0.2, device="cuda")) if dyn else {}
    cache = binding.KV4Cache(pk, pv, codes[0], codes[1], None if dyn else s, None if dyn else s, torch.zeros(B, dtype=torch.int32, device="cuda"), Hq, **steps)
    ws = ctx.decode_attn_workspace(cache)
    n = B * Hkv * D
    base, kv, new = rand(2 * n), torch.zeros(2 * n, dtype=torch.bfloat16, device="cuda"), torch.zeros(2 * n, dtype=torch.bfloat16, device="cuda")
    q, out, after = rand(B, Hq, D), rand(B, Hq, D), rand(B, Hq, D)
    inputs_ = [rand(2 * n) * 2.0**i for i in range(4)]

    def chain(step):
        for _ in range(3):
            ctx.residual_add(kv, base, out=new)
            step()
            ctx.kv4_append(cache, new[:n].view(B, 1, Hkv, D), new[n:].view(B, 1, Hkv, D))
            step()
            ctx.decode_attn(cache, q, 1 / math.sqrt(D), ws, out=out)
            step()
            ctx.residual_add(out, q, out=after)
            step()
            ctx.residual_add(new, base, out=kv)
            step()

    def run(call):
        res = []
        for v in inputs_:
            kv.copy_(v)
            cache.length.fill_(T0)
            torch.cuda.synchronize()
            call()
            torch.cuda.synchronize()
            res.append([t.clone() for t in (out, after, cache.kq, cache.vq, cache.length, *steps.values())])
        return res

    want = run(lambda: chain(torch.cuda.synchronize))
    assert int(want[0][4][0]) == T0 + 3
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(lambda: None)
    for call in (graph.replay, lambda: chain(lambda: None)):
        for w, r in zip(want, run(call)):
            assert all(torch.equal(a, b) for a, b in zip(w, r))
    ctx.check()


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M", [33, 64, 96, 97, 128])
@pytest.mark.parametrize("N", [4096, 28672])
def test_what_follows_a_captured_gemm_reads_its_output_and_overwrites_its_tokens(ctx, mode, M, N):
    """rotate + quantize -> GEMM -> residual add -> rotate + quantize over the sum, into the buffer the GEMM took its tokens from -> GEMM back
    to the width of the start -> residual add, twice, replayed as one graph with other inputs, against the calls apart. In a graph the split-K GEMM of 33 to
    96 rows (to 128 with a step per token) lets its successor be placed while it still adds and stores; 4096 channels are split along K, 28672 are not."""
    K = 4096
    g = torch.Generator(device="cuda").manual_seed(M + N)
    rand = lambda *sh: torch.randn(sh, generator=g, device="cuda").to(torch.bfloat16)
    wq = [torch.randint(0, 256, sh, dtype=torch.uint8, device="cuda", generator=g) for sh in ((N, K // 2), (K, N // 2))]
    s_w = [torch.full((n,), 4e-3, device="cuda") for n in (N, K)]
    wsum = [ctx.weight_code_sums(w) for w in wq]
    s_a, s_tok = torch.full((1,), 0.02 if mode == "w4a8" else 0.3, device="cuda"), torch.full((M,), 0.3, device="cuda")
    z = torch.full((1,), 6, dtype=torch.int32, device="cuda")
    flat = torch.zeros(M * max(N, K), dtype=torch.int8 if mode == "w4a8" else torch.uint8, device="cuda")
    x, base, out, mid = rand(M, K), rand(M, N), torch.zeros((M, N), dtype=torch.bfloat16, device="cuda"), torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    back = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda")
    xs = [rand(M, K) * 2.0**i for i in range(4)]

    def linear(src, i, dst, step):
        k = src.shape[1]
        xq = flat[: M * (k if mode == "w4a8" else k // 2)].view(M, -1)
        if mode == "w4a8":
            ctx.hadamard_quant_act8(src, 4096, s_a, out=xq)
        elif mode == "rows":
            ctx.hadamard_quant_act_rows(src, 4096, s_tok, out=xq)
        elif mode == "asym":
            ctx.hadamard_quant_act_asym(src, 4096, s_a, z, out=xq)
        else:
            ctx.hadamard_quant_act(src, 4096, s_a, out=xq)
        step()
        if mode == "w4a8":
            ctx.w4a8_gemm(xq, wq[i], s_a, s_w[i], out=dst)
        elif mode == "rows":
            ctx.w4a4_gemm_rows(xq, wq[i], s_tok, s_w[i], out=dst)
        elif mode == "asym":
            ctx.w4a4_gemm_asym(xq, wq[i], s_a, z, s_w[i], wsum[i], out=dst)
        else:
            ctx.w4a4_gemm(xq, wq[i], s_a, s_w[i], out=dst)
        step()

    def chain(step):
        for _ in range(2):
            linear(x, 0, out, step)
            ctx.residual_add(out, base, out=mid)
            step()
            linear(mid, 1, back, step)
            ctx.residual_add(back, x, out=x)
            step()

    def run(call):
        res = []
        for v in xs:
            x.copy_(v)
            torch.cuda.synchronize()
            call()
            torch.cuda.synchronize()
            res.append([t.clone() for t in (x, out, mid, back, flat)])
        return res

    want = run(lambda: chain(torch.cuda.synchronize))
    assert all(len(torch.unique(t)) > 12 for t in want[0]) and bool(torch.isfinite(want[-1][0].float()).all())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(lambda: None)
    for call in (graph.replay, lambda: chain(lambda: None), graph.replay):
        for i, (w, r) in enumerate(zip(want, run(call))):
            assert all(torch.equal(a, b) for a, b in zip(w, r)), f"input {i}"
    ctx.check()


@pytest.mark.parametrize("M", [1, 24, 64, 96, 300, 1030])
@pytest.mark.parametrize("N,K", [(4096, 4096), (8448, 1024)])
def test_weights_are_not_overwritten_under_the_gemm_that_reads_them(ctx, M, N, K):
    """GEMM -> weight quantizer into the codes and steps that GEMM reads -> GEMM on the new ones, and on, in a graph and called back to back:
    the quantizer is placed while the GEMM drains and writes only when it has ended. Sums and outputs as by the calls apart."""
    g = torch.Generator(device="cuda").manual_seed(M)
    W = [inputs.weights(N, K, seed=2 + s).cuda() * 2.0**s for s in range(3)]
    wq, s_w = torch.zeros((N, K // 2), dtype=torch.uint8, device="cuda"), torch.zeros(N, device="cuda")
    xq = torch.randint(0, 256, (M, K // 2), dtype=torch.uint8, device="cuda", generator=g)
    s_a = torch.full((1,), 0.3, device="cuda")
    out = torch.zeros((4, M, N), dtype=torch.bfloat16, device="cuda")
    acc = torch.zeros((4, M, N), dtype=torch.int32, device="cuda")

    def chain(step):
        for i in range(4):
            ctx.quant_weights(W[i % 3], out=(wq, s_w))
            step()
            ctx.w4a4_gemm(xq, wq, s_a, s_w, out=out[i], acc_dbg=acc[i])
            step()

    def run(call):
        out.zero_(), acc.zero_()
        torch.cuda.synchronize()
        call()
        torch.cuda.synchronize()
        return out.clone(), acc.clone()

    want = run(lambda: chain(torch.cuda.synchronize))
    assert not torch.equal(want[1][0], want[1][1])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(lambda: None)
    for call in (graph.replay, lambda: chain(lambda: None)) * 3:
        for a, b in zip(want, run(call)):
            assert torch.equal(a, b)
    ctx.check()

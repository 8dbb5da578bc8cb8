"""Stream order of the calls under programmatic dependent launch: calls enqueued back to back give bit for bit what the same
calls give with a synchronisation between them."""
import math

import pytest
import torch

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

"""Failure detection on the device: every wait inside a kernel is bounded, and a wait that runs out is reported
through the status word while the kernel winds down in order (copies in flight awaited, tensor memory released).
Nothing is made to fault or hang: a self-test kernel waits, with a short bound, on a barrier nothing completes; and
the bound of the real kernels is lowered to a few clocks, so that an ordinary first wait (for a copy that needs a
microsecond) may legitimately run out. Whether it does depends on how long one hardware try_wait suspends, so each
such call may report a timeout or succeed; either way the same context, with the default bound back, must then give
exact results."""
import math

import numpy as np
import pytest
import torch

import gemm_plan
from oracle import pq_oracle as orc
from paper_2410_05265_b200 import inputs
from helpers import assert_attn_close, rand_codes, to_np

pytestmark = pytest.mark.gpu
PQ_ERR_TIMEOUT = 6


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def test_selftest_wait_runs_out_after_the_limit_and_is_reported():
    from paper_2410_05265_b200 import binding

    ctx = binding.Context()
    ctx.set_wait_limit(200_000)                 # a tenth of a millisecond
    waited = ctx.selftest_wait()
    assert ctx.check_status() == PQ_ERR_TIMEOUT
    assert 200_000 < int(waited) < 50_000_000, "the wait ends soon after its bound"
    assert ctx.check_status() == 0
    ctx.set_wait_limit(0)
    x = torch.zeros((4, 128), dtype=torch.bfloat16, device="cuda")
    ctx.hadamard_quant_act(x, 128, torch.ones(1, device="cuda"))
    assert ctx.check_status() == 0              # the context works on
    ctx.close()


def test_a_wait_that_runs_out_is_reported_and_the_context_stays_usable():
    from paper_2410_05265_b200 import binding

    ctx = binding.Context()
    rng = np.random.default_rng(0)
    D = 128
    # split-K GEMM with a few and with many K blocks per CTA; CTA-pair GEMM with weights in tensor memory (more than 128 rows and 64
    # channel tiles), short and long K and with 8-bit tokens (a producer of their own); the one with both operands in shared memory
    gemms = []
    for M, N, K, a8 in [(128, 256, 512, False), (128, 256, 32768, False), (96, 256, 32768, True), (129, 8448, 4096, False), (129, 8448, 8192, False),
                        (129, 8448, 4096, True), (1216, 11304, 2048, True)]:
        wq = rand_codes(rng, N, K)
        xq = rng.integers(-128, 128, (M, K)).astype(np.int8) if a8 else rand_codes(rng, M, K)
        gemms.append((ctx.w4a8_gemm if a8 else ctx.w4a4_gemm, dev(xq), dev(wq), orc.gemm_i8i4(xq, wq) if a8 else orc.gemm_i4(xq, wq)))
    s_a, s_w_all = torch.full((1,), 0.02, device="cuda"), torch.full((11304,), 0.003, device="cuda")
    # a small KV4 cache for the decode and the prefill attention
    B, Hq, Hkv, T, Tmax, P = 2, 8, 2, 300, 320, 4
    kq_np, vq_np = rng.integers(0, 256, (B, Hkv, Tmax, D // 2)).astype(np.uint8), rng.integers(0, 256, (B, Hkv, Tmax, D // 2)).astype(np.uint8)
    s_k, s_v = np.full(Hkv, 0.3, np.float32), np.full(Hkv, 0.5, np.float32)
    pk, pv = inputs.prefix_kv(Hkv, P, D, 0, "k", 1.0), inputs.prefix_kv(Hkv, P, D, 0, "v", 1.0)
    length = np.full(B, T, np.int32)
    cache = binding.KV4Cache(pk.cuda(), pv.cuda(), dev(kq_np), dev(vq_np), dev(s_k), dev(s_v), dev(length), Hq)
    q = inputs.queries(B, Hq, D, 0)
    qp = inputs.kv_tensor(1, T, Hq, D, 3, "k")[0].contiguous()
    ws = ctx.decode_attn_workspace(cache)
    sm = 1 / math.sqrt(D)

    ctx.set_wait_limit(16)                      # a few clocks: no copy from memory is that fast
    seen = []
    for gemm, xq, wq, _ in gemms:
        gemm(xq, wq, s_a, s_w_all[: wq.shape[0]])
        seen.append(ctx.check_status())
        assert ctx.check_status() == 0          # reading the status word clears it
    ctx.decode_attn(cache, q.cuda(), sm, ws)
    seen.append(ctx.check_status())
    ctx.prefill_attn(cache, 1, qp.cuda(), sm)
    seen.append(ctx.check_status())
    torch.cuda.synchronize()                    # the process and the CUDA context are alive
    assert all(st in (0, PQ_ERR_TIMEOUT) for st in seen), seen
    print("statuses under a 16-clock bound (seven GEMMs, decode attention, prefill attention):", seen)

    ctx.set_wait_limit(0)                       # the default bound again: exact results from the same context
    for gemm, xq, wq, acc_ref in gemms:
        acc = torch.zeros(acc_ref.shape, dtype=torch.int32, device="cuda")
        gemm(xq, wq, s_a, s_w_all[: wq.shape[0]], acc_dbg=acc)
        assert ctx.check_status() == 0 and np.array_equal(to_np(acc), acc_ref)
    out = ctx.decode_attn(cache, q.cuda(), sm, ws)
    assert ctx.check_status() == 0
    _, ref = orc.decode_attn(inputs.bits(q), inputs.bits(pk), inputs.bits(pv), kq_np, vq_np, s_k, s_v, length, sm, want_f64=True)
    assert_attn_close(inputs.bits(out), ref, "decode attention after a timed-out call")
    outp = ctx.prefill_attn(cache, 1, qp.cuda(), sm)
    assert ctx.check_status() == 0
    _, refp = orc.prefill_attn(inputs.bits(qp), inputs.bits(pk), inputs.bits(pv), kq_np[1], vq_np[1], s_k, s_v, sm, want_f64=True)
    assert_attn_close(inputs.bits(outp), refp, "prefill attention after a timed-out call")
    ctx.close()


@pytest.mark.parametrize("mode", ["w4a4", "w4a8"])
@pytest.mark.parametrize("M", [16, 40, 96, 128, 200, 130])
def test_a_slow_predecessor_does_not_count_against_the_bounded_waits(mode, M):
    """A GEMM placed early (split-K kernel, many K blocks per CTA; CTA-pair kernel) behind a kernel that runs several times longer than the wait
    limit, though each of its own waits is short (causal attention, 128 key tiles in sequence): nothing is stuck, no timeout."""
    from paper_2410_05265_b200 import binding

    ctx = binding.Context()
    rng = np.random.default_rng(M)
    N, K, T, D = 640, 4096 if M == 130 else 16384, 16384, 128
    wq = rand_codes(rng, N, K)
    if M == 130:  # a layer wide enough for the CTA-pair kernel, which requests its first weights early, too
        wq = np.tile(wq, (14, 1))[:8448]
        assert gemm_plan.route(M, len(wq), K, mode == "w4a8") == "pair_ts"
    if M == 16:  # up to 16 tokens only large layers take that kernel
        wq = np.concatenate([wq, wq, wq])[:1408]
    if mode == "w4a8":
        x8 = rng.integers(-128, 128, (M, K)).astype(np.int8)
        ref, call, xq = orc.gemm_i8i4(x8, wq), ctx.w4a8_gemm, dev(x8)
    else:
        x4 = rand_codes(rng, M, K)
        ref, call, xq = orc.gemm_i4(x4, wq), ctx.w4a4_gemm, dev(x4)
    kq = torch.randint(0, 256, (1, 1, T, D // 2), dtype=torch.uint8, device="cuda")
    s = torch.full((1,), 0.3, device="cuda")
    cache = binding.KV4Cache(None, None, kq, kq.clone(), s, s, torch.full((1,), T, dtype=torch.int32, device="cuda"), 1)
    q = torch.randn((T, 1, D), device="cuda").to(torch.bfloat16)
    s_a, s_w = torch.full((1,), 0.02, device="cuda"), torch.full((wq.shape[0],), 0.003, device="cuda")
    acc, wq = torch.zeros(ref.shape, dtype=torch.int32, device="cuda"), dev(wq)
    out, attn = torch.empty(ref.shape, dtype=torch.bfloat16, device="cuda"), torch.empty_like(q)
    for limit in (0, 60_000):                   # the first pass loads the kernels
        ctx.set_wait_limit(limit)
        for _ in range(3):
            acc.zero_()
            torch.cuda.synchronize()
            ctx.prefill_attn(cache, 0, q, 1 / math.sqrt(D), out=attn)
            call(xq, wq, s_a, s_w, out=out, acc_dbg=acc)
            assert ctx.check_status() == 0
            assert np.array_equal(to_np(acc), ref)
    ctx.close()

"""Prefill attention of short prompts (one 128-row tile per CTA, its key tiles dealt to two softmax groups) and the border to the form with two
row tiles: one key tile to several with and without a prefix tile, ragged ends, both settings of the KV steps."""
import math

import numpy as np
import pytest
import torch

from oracle import pq_oracle as orc
from helpers import assert_attn_close, to_np
from paper_2410_05265_b200 import inputs

pytestmark = pytest.mark.gpu
D = 128


@pytest.mark.parametrize("dyn", [False, True])
@pytest.mark.parametrize("T,Hq,Hkv,P", [
    (17, 4, 1, 0), (128, 2, 1, 0), (129, 2, 1, 0), (128, 4, 2, 1), (256, 8, 1, 64), (257, 4, 4, 4), (385, 2, 2, 3), (515, 8, 2, 4),
    # 128-row CTAs that still have an SM each on 148 SMs, and one token more
    (384, 48, 48, 4), (385, 48, 48, 0), (288, 64, 16, 3), (289, 64, 16, 4),
])
def test_prefill_attention_of_short_prompts(dyn, T, Hq, Hkv, P):
    from paper_2410_05265_b200 import binding

    ctx = binding.Context()
    Tmax = T + 5
    k, v = (inputs.kv_tensor(1, T, Hkv, D, 0, w) for w in "kv")
    s_k, s_v = (orc.calib_kv_scale(inputs.bits(t)) for t in (k, v))
    pk, pv = (inputs.prefix_kv(Hkv, max(P, 1), D, 0, w, 1.0)[:, :P].contiguous() for w in "kv")
    q = inputs.kv_tensor(1, T, Hq, D, 3, "k")[0].contiguous()
    kq = torch.zeros((1, Hkv, Tmax, D // 2), dtype=torch.uint8, device="cuda")
    vq, length = torch.zeros_like(kq), torch.zeros(1, dtype=torch.int32, device="cuda")
    steps = dict(sk_tok=torch.ones((1, Hkv, Tmax), device="cuda"), sv_tok=torch.ones((1, Hkv, Tmax), device="cuda")) if dyn else {}
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    cache = binding.KV4Cache(pk.cuda() if P else None, pv.cuda() if P else None, kq, vq, None if dyn else dev(s_k), None if dyn else dev(s_v),
                             length, Hq, **steps)
    ctx.kv4_append(cache, k.cuda(), v.cuda())
    out = torch.full((T, Hq, D), 7.0, dtype=torch.bfloat16, device="cuda")
    ctx.prefill_attn(cache, 0, q.cuda(), 1 / math.sqrt(D), out=out)
    ctx.check()
    args = (inputs.bits(q), inputs.bits(pk), inputs.bits(pv), to_np(kq)[0], to_np(vq)[0])
    if dyn:
        _, ref = orc.prefill_attn_dyn(*args, to_np(steps["sk_tok"])[0], to_np(steps["sv_tok"])[0], 1 / math.sqrt(D))
    else:
        _, ref = orc.prefill_attn(*args, s_k, s_v, 1 / math.sqrt(D), want_f64=True)
    assert_attn_close(inputs.bits(out), ref, f"prefill attention T{T} Hq{Hq} Hkv{Hkv} P{P} dyn{dyn}")
    ctx.close()

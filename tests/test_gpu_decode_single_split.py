"""Decode attention where a (sequence, KV head) has a single split (caches below 128 rows, many pairs): one CTA then merges all
query heads of the group, more (head, dims) items than it has threads when the group has more than four heads."""
import math

import numpy as np
import pytest
import torch

from oracle import pq_oracle as orc
from paper_2410_05265_b200 import inputs
from helpers import assert_attn_close, to_np

pytestmark = pytest.mark.gpu
D = 128


@pytest.mark.parametrize("B,Hq,Hkv,P,T", [(40, 8, 1, 2, 90), (10, 48, 8, 0, 100), (5, 64, 8, 4, 17), (38, 4, 1, 1, 64)])
def test_single_split_writes_every_query_head(B, Hq, Hkv, P, T):
    from paper_2410_05265_b200 import binding

    ctx = binding.Context()
    rng = np.random.default_rng(B + Hq)
    Tmax = T + 1
    kq = rng.integers(0, 256, (B, Hkv, Tmax, D // 2)).astype(np.uint8)
    vq = rng.integers(0, 256, (B, Hkv, Tmax, D // 2)).astype(np.uint8)
    s_k, s_v, length = np.full(Hkv, 0.1, np.float32), np.full(Hkv, 0.2, np.float32), np.full(B, T, np.int32)
    pk, pv = (inputs.prefix_kv(Hkv, max(P, 1), D, 0, w, 1.0)[:, :P].contiguous() for w in "kv")
    q = inputs.queries(B, Hq, D, 0)
    dev = lambda a: torch.from_numpy(a.copy()).cuda()
    cache = binding.KV4Cache(pk.cuda() if P else None, pv.cuda() if P else None, dev(kq), dev(vq), dev(s_k), dev(s_v), dev(length), Hq)
    sm = 1 / math.sqrt(D)
    ws = ctx.decode_attn_workspace(cache)
    ref = lambda n: orc.decode_attn(inputs.bits(q), inputs.bits(pk), inputs.bits(pv), kq, vq, s_k, s_v, n, sm, want_f64=True)[1]
    out = ctx.decode_attn(cache, q.cuda(), sm, ws, out=torch.full((B, Hq, D), 3.0, dtype=torch.bfloat16, device="cuda"))
    ctx.check()
    assert_attn_close(inputs.bits(out), ref(length), f"single split B{B} Hq{Hq} Hkv{Hkv}")
    k, v = (inputs.kv_tensor(B, 1, Hkv, D, 0, w) for w in "kv")  # the one-launch step over the same cache
    out = ctx.kv4_append_decode_attn(cache, k.cuda(), v.cuda(), q.cuda(), sm, ws, out=torch.full((B, Hq, D), 3.0, dtype=torch.bfloat16, device="cuda"))
    ctx.check()
    assert orc.kv4_append(inputs.bits(k), inputs.bits(v), s_k, s_v, kq, vq, length) == 0
    assert np.array_equal(to_np(cache.length), length) and np.array_equal(to_np(cache.kq), kq)
    assert_attn_close(inputs.bits(out), ref(length), f"single split, one launch, B{B} Hq{Hq} Hkv{Hkv}")
    ctx.close()

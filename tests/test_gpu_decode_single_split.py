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


@pytest.mark.parametrize("B,Hq,Hkv,P,Tmax,lengths", [
    (1, 8, 2, 4, 127, [100]), (1, 8, 2, 4, 129, [128]), (2, 4, 1, 0, 385, [0, 383]), (1, 32, 8, 4, 1024, [1021]), (2, 8, 1, 1, 1153, [1150, 896]),
    (1, 16, 2, 4, 3072, [3069]), (1, 8, 2, 3, 3201, [3073]), (3, 8, 1, 4, 4096, [4093, 1, 2049]), (1, 8, 1, 2, 4224, [4200]),
])
def test_few_pairs_at_the_borders_of_their_splits(B, Hq, Hkv, P, Tmax, lengths):
    """One (sequence, KV head) pair to a few: fewer rounds of 128 keys than splits, one cluster, the lengths up to which it is one (for the plain
    call and for the one-launch step), several clusters. The step runs twice: its counter starts from zero again."""
    from paper_2410_05265_b200 import binding

    ctx = binding.Context()
    rng = np.random.default_rng(Tmax)
    kq = rng.integers(0, 256, (B, Hkv, Tmax, D // 2)).astype(np.uint8)
    vq = rng.integers(0, 256, (B, Hkv, Tmax, D // 2)).astype(np.uint8)
    s_k, s_v, length = np.full(Hkv, 0.1, np.float32), np.full(Hkv, 0.2, np.float32), np.array(lengths, np.int32)
    pk, pv = (inputs.prefix_kv(Hkv, max(P, 1), D, 0, w, 1.0)[:, :P].contiguous() for w in "kv")
    q = inputs.queries(B, Hq, D, 0)
    dev = lambda a: torch.from_numpy(a.copy()).cuda()
    cache = binding.KV4Cache(pk.cuda() if P else None, pv.cuda() if P else None, dev(kq), dev(vq), dev(s_k), dev(s_v), dev(length), Hq)
    sm = 1 / math.sqrt(D)
    ws = ctx.decode_attn_workspace(cache)
    ref = lambda n: orc.decode_attn(inputs.bits(q), inputs.bits(pk), inputs.bits(pv), kq, vq, s_k, s_v, n, sm, want_f64=True)[1]
    out = torch.full((B, Hq, D), 3.0, dtype=torch.bfloat16, device="cuda")
    if P or min(lengths) > 0:
        ctx.decode_attn(cache, q.cuda(), sm, ws, out=out)
        ctx.check()
        assert_attn_close(inputs.bits(out), ref(length), f"few pairs B{B} Tmax{Tmax}")
    for step in range(2):
        if length.max() >= Tmax:
            break
        k, v = (inputs.kv_tensor(B, 1, Hkv, D, step, w) for w in "kv")
        ctx.kv4_append_decode_attn(cache, k.cuda(), v.cuda(), q.cuda(), sm, ws, out=out.fill_(3.0))
        ctx.check()
        assert orc.kv4_append(inputs.bits(k), inputs.bits(v), s_k, s_v, kq, vq, length) == 0
        assert np.array_equal(to_np(cache.length), length) and np.array_equal(to_np(cache.kq), kq)
        assert_attn_close(inputs.bits(out), ref(length), f"few pairs, one launch, B{B} Tmax{Tmax} step {step}")
    ctx.close()

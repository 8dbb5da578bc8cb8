"""GPU parity of the tensor-core GEMMs against the CPU oracle. Split-K kernel (a few tens to a few hundred tokens): every
token-tile width and its edges, ragged channel counts and K tails, the four settings of the call, and the border to the CTA-pair
kernels. CTA-pair kernels at shapes above that border: ragged tiles, both kinds of output store, skipped rows, the ends of int32."""
import numpy as np
import pytest
import torch

import gemm_plan
from oracle import pq_oracle as orc
from helpers import assert_bf16_close, rand_codes, to_np
from paper_2410_05265_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2410_05265_b200 import binding

    c = binding.Context()
    yield c
    c.check()
    c.close()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def check(ctx, mode, M, N, K, ldo_pad=0, row_begin=0):
    rng = np.random.default_rng(M * 1009 + N * 31 + K)
    wq, s_w = rand_codes(rng, N, K), rng.uniform(0.5, 2.0, N).astype(np.float32) * 1e-3
    s_a, s_tok = np.float32(0.02), rng.uniform(0.01, 0.03, M).astype(np.float32)
    out = torch.full((M, N + ldo_pad), 7.0, dtype=torch.bfloat16, device="cuda")
    view = out[:, :N]
    acc = torch.full((M, N), -77, dtype=torch.int32, device="cuda")
    kw = dict(out=view, acc_dbg=acc, row_begin=row_begin)
    sa = torch.full((1,), float(s_a), device="cuda")
    if mode == "w4a8":
        x8 = rng.integers(-128, 128, (M, K)).astype(np.int8)
        ref = orc.gemm_i8i4(x8, wq)
        ctx.w4a8_gemm(dev(x8), dev(wq), sa, dev(s_w), **kw)
    else:
        xq = rand_codes(rng, M, K)
        ref = orc.gemm_i4(xq, wq)
        if mode == "rows":
            ctx.w4a4_gemm_rows(dev(xq), dev(wq), dev(s_tok), dev(s_w), **kw)
        elif mode == "asym":
            wsum = ctx.weight_code_sums(dev(wq))
            ref = ref - (5 - 8) * to_np(wsum).astype(ref.dtype)[None]
            ctx.w4a4_gemm_asym(dev(xq), dev(wq), sa, torch.full((1,), 5, dtype=torch.int32, device="cuda"), dev(s_w), wsum, **kw)
        else:
            ctx.w4a4_gemm(dev(xq), dev(wq), sa, dev(s_w), **kw)
    ctx.check()
    assert np.array_equal(to_np(acc)[row_begin:], ref[row_begin:]), "accumulators differ"
    assert np.all(to_np(acc)[:row_begin] == -77) and bool((out[:row_begin] == 7.0).all()), "rows below row_begin must not be written"
    want = ref.astype(np.float64) * (s_tok.astype(np.float64)[:, None] if mode == "rows" else float(s_a)) * s_w.astype(np.float64)
    want = torch.from_numpy(want).to(torch.bfloat16)
    assert_bf16_close(inputs.bits(view[row_begin:]), inputs.bits(want[row_begin:]), f"{mode} GEMM {M} x {N} x {K}")
    if ldo_pad:
        assert bool((out[:, N:] == 7.0).all()), "columns past N must not be written"


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M,N,K", [
    (17, 1, 32), (32, 127, 160), (33, 129, 416), (48, 130, 1152), (49, 257, 640), (64, 128, 2048), (65, 100, 1280),
    (96, 260, 672), (97, 128, 256), (128, 300, 1280), (129, 128, 4128), (256, 132, 1280), (257, 640, 512), (600, 130, 96), (300, 4000, 640),
])
def test_split_gemm_matches_oracle(ctx, mode, M, N, K):
    check(ctx, mode, M, N, K)


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M", [17, 33, 49, 64, 96, 128])
def test_split_gemm_ends_of_the_k_blocks_and_rings(ctx, mode, M):
    """K around whole K blocks of 128 and 256 elements (a part of one, one and a half, a ring's length and one more, with and without a K split),
    at each width of the token tiles."""
    for N, K in [(130, 96), (128, 224), (129, 256), (64, 288), (130, 1536), (130, 1664), (70, 1824), (200, 7168 + 160)]:
        check(ctx, mode, M, N, K)


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M,N,K,width", [
    (129, 5000, 1280, 64), (192, 6001, 1536, 64), (191, 6144, 96, 64), (136, 6100, 4128, 64), (250, 3000, 416, 64),
    (210, 3900, 2592, 128), (255, 2600, 2080, 128), (256, 3000, 3232, 128),
])
def test_narrow_tiles_above_128_tokens(ctx, mode, M, N, K, width):
    """The forms that take an SM alone, 64 and 128 tokens wide: ragged last tiles, one K block to more than the rings hold, one K split and two."""
    assert gemm_plan.width_whole(M, N, K, mode == "w4a8") == width
    check(ctx, mode, M, N, K)


def test_few_tokens_of_a_long_k(ctx):
    for mode, M, N, K in [("w4a4", 1, 136, 16416), ("w4a8", 8, 130, 20480), ("rows", 3, 264, 28672), ("asym", 5, 100, 16512)]:
        check(ctx, mode, M, N, K)


@pytest.mark.parametrize("M,N,K,pad", [(40, 131, 1536, 5), (100, 260, 5120, 4), (24, 3000, 10240, 1)])
def test_split_gemm_with_a_padded_output(ctx, M, N, K, pad):
    """Row pitches that allow 8-byte stores and that do not; up to eight K splits, two and more K blocks per expansion group."""
    check(ctx, "w4a4", M, N, K, pad)


@pytest.mark.parametrize("mode", ["w4a4", "w4a8"])
def test_large_layers_with_nine_to_sixteen_tokens(ctx, mode):
    for M, N, K in [(9, 5128, 4128), (16, 5120, 4096)]:  # just inside the rule for 9 to 16 tokens
        check(ctx, mode, M, N, K)


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M,N,K", [(129, 8200, 160), (300, 4104, 416), (130, 8328, 8224)])
def test_pair_kernels_just_above_the_border(ctx, mode, M, N, K):
    """Problems just too large for two K splits go to the CTA-pair kernel: ragged edges, short and long K."""
    check(ctx, mode, M, N, K)


# ---- above the border: more than 128 rows and N > 8192 (65 and more channel tiles of 128) always go to the CTA-pair kernels
@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M,N,K,pad,row_begin", [
    (200, 8264, 416, 0, 4),        # dense rows, channels a multiple of 8: bulk-tensor stores; skipped rows
    (141, 8203, 512, 0, 5),        # channels not a multiple of 8: element-wise stores
    (150, 8264, 1152, 4, 0),       # rows too far apart for the bulk stores' 16-byte pitch
    (137, 8203, 8224, 3, 1),       # the same with a long K
    (290, 10241, 8192, 0, 7),      # more tiles than CTA pairs, element-wise stores
    (260, 20000, 160, 0, 0),       # more tiles than CTA pairs, two K blocks
])
def test_pair_kernels_match_oracle(ctx, mode, M, N, K, pad, row_begin):
    check(ctx, mode, M, N, K, pad, row_begin)


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows"])
@pytest.mark.parametrize("K", [4096, 28672, 65536])
def test_pair_kernels_extreme_codes_fit_int32(ctx, mode, K):
    """Every code at its lowest: the largest sums, and with the factors 16 of the expanded codes 2^30 at K = 65536."""
    M, N = 130, 8208
    wq = torch.full((N, K // 2), 0x88, dtype=torch.uint8, device="cuda")
    one, s_w = torch.ones(1, device="cuda"), torch.ones(N, device="cuda")
    acc = torch.zeros((M, N), dtype=torch.int32, device="cuda")
    if mode == "w4a8":
        ctx.w4a8_gemm(torch.full((M, K), -128, dtype=torch.int8, device="cuda"), wq, one, s_w, acc_dbg=acc)
    else:
        xq = torch.full((M, K // 2), 0x88, dtype=torch.uint8, device="cuda")
        if mode == "rows":
            ctx.w4a4_gemm_rows(xq, wq, torch.ones(M, device="cuda"), s_w, acc_dbg=acc)
        else:
            ctx.w4a4_gemm(xq, wq, one, s_w, acc_dbg=acc)
    ctx.check()
    assert int(acc.min()) == int(acc.max()) == 8 * K * (128 if mode == "w4a8" else 8)

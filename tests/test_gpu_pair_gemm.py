"""GPU parity of the CTA-pair GEMMs against the CPU oracle where their tiles can go wrong: every width of a token tile, tiles of two
widths in one launch, a second half narrower than the first, one K block and K tails, more K blocks than any ring holds, several tiles
per pair, ragged channels, both kinds of output store; and 8-bit tokens on whole tiles of 256 (the kernel with both
operands in shared memory). Which kernel and which tiles a shape takes is asked of the launch rules themselves."""
import pytest

import gemm_plan
from test_gpu_split_gemm import check, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M,N,K,ldo_pad", [
    (129, 8448, 32, 0), (161, 8300, 416, 0), (193, 8448, 1152, 3), (256, 8300, 160, 0), (100, 19000, 96, 0),  # one tile per channel tile, or two
    (257, 4250, 1312, 5), (300, 6144, 1152, 0),
    (333, 9500, 256, 0),                                                                                     # several tiles per pair
    (515, 2250, 640, 0), (700, 1500, 2080, 8), (1000, 770, 128, 0), (1500, 264, 992, 0),                     # the split kernel's side
])
def test_pair_gemm_matches_oracle(ctx, mode, M, N, K, ldo_pad):  # noqa: F811
    check(ctx, mode, M, N, K, ldo_pad)


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M,N,K,widths", [
    (273, 12500, 384, (3,)), (849, 5300, 384, (4, 3)), (97, 57100, 128, (4,)), (129, 57344, 384, (5,)), (160, 57100, 128, (5,)), (160, 57100, 1152, (5,)), (192, 57000, 384, (6,)), (192, 57344, 1056, (6,)),
    (193, 57100, 640, (7,)), (224, 57344, 1152, (7,)), (256, 57100, 128, (8,)), (256, 57000, 1152, (8,)), (515, 28700, 384, (6, 5)),
    (515, 28672, 1152, (6, 5)), (600, 28700, 256, (7, 6)), (700, 28700, 1152, (8, 7)),
])
def test_several_tiles_per_pair_at_every_width(ctx, mode, M, N, K, widths):  # noqa: F811
    """Two, three and four accumulator slots that come round again, one K block and more than the rings hold."""
    p = gemm_plan.pair_plan(M, N, K, mode == "w4a8")
    assert gemm_plan.route(M, N, K, mode == "w4a8") == "pair_ts" and p.c_tiles * p.t_tiles > 3 * (gemm_plan.SMS // 2) / 2
    assert widths == tuple(sorted({p.widest, p.base_units}, reverse=True)) and p.n_acc == {2: 4, 3: 3, 4: 2}[p.half_units]
    check(ctx, mode, M, N, K)


@pytest.mark.parametrize("M,N,K,row_begin", [(130, 57100, 32, 0), (300, 28700, 416, 4)])
def test_many_tiles_of_8bit_tokens_match_oracle(ctx, M, N, K, row_begin):  # noqa: F811
    check(ctx, "w4a8", M, N, K, row_begin=row_begin)


@pytest.mark.parametrize("M,N,K,ldo_pad,row_begin", [
    (1216, 11304, 2048, 8, 0), (1280, 11521, 2080, 3, 0), (1250, 11400, 2176, 0, 5), (2033, 7424, 4128, 0, 0), (1500, 9600, 8192, 0, 0),
])
def test_8bit_tokens_on_whole_tiles_match_oracle(ctx, M, N, K, ldo_pad, row_begin):  # noqa: F811
    """The kernel with both operands in shared memory: three rounds of tiles and more, token, channel and K tails, both kinds of store."""
    assert gemm_plan.route(M - row_begin, N, K, True) == "pair"
    check(ctx, "w4a8", M, N, K, ldo_pad, row_begin)


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M", [129, 192, 193, 257, 384, 385])
def test_split_gemm_at_the_edges_of_its_192_token_tiles(ctx, mode, M):  # noqa: F811
    check(ctx, mode, M, 300, 1312)


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M,N,K,ldo_pad", [(129, 8444, 160, 4), (257, 8301, 96, 3), (150, 8266, 416, 14), (129, 19007, 64, 1)])
def test_columns_past_a_ragged_width_stay_as_they_are(ctx, mode, M, N, K, ldo_pad):  # noqa: F811
    """A width that is no multiple of eight inside rows whose pitch is one: bulk stores are cut at 16 bytes, not at the last channel."""
    assert (N + ldo_pad) % 8 == 0 and N % 8 and gemm_plan.route(M, N, K, mode == "w4a8") == "pair_ts"
    check(ctx, mode, M, N, K, ldo_pad)


def test_columns_past_a_ragged_width_stay_as_they_are_on_whole_tiles(ctx):  # noqa: F811
    M, N, K, ldo_pad = 1216, 11300, 2048, 4
    assert gemm_plan.route(M, N, K, True) == "pair"
    check(ctx, "w4a8", M, N, K, ldo_pad)

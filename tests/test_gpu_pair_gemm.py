"""GPU parity of the CTA-pair GEMMs against the CPU oracle where their tiles can go wrong: every width of a token tile, tiles of two
widths in one launch, a second half narrower than the first, one K block and K tails, more K blocks than any ring holds, several tiles
per pair, ragged channels, both kinds of output store; and 8-bit tokens on more than three rounds of tiles (the kernel with both
operands in shared memory)."""
import pytest

import gemm_plan
from test_gpu_split_gemm import check, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["w4a4", "w4a8", "rows", "asym"])
@pytest.mark.parametrize("M,N,K,ldo_pad", [
    (129, 8448, 32, 0), (161, 8300, 416, 0), (193, 8448, 1152, 3), (256, 8300, 160, 0), (100, 19000, 96, 0),  # one tile per channel tile, or two
    (257, 4250, 1312, 5), (300, 6144, 1152, 0), (515, 2250, 640, 0), (700, 1500, 2080, 8), (1000, 770, 128, 0), (1500, 264, 992, 0),
    (333, 9500, 256, 0),                                                                                     # several tiles per pair
])
def test_pair_gemm_matches_oracle(ctx, mode, M, N, K, ldo_pad):  # noqa: F811
    check(ctx, mode, M, N, K, ldo_pad)


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

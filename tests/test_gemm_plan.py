"""The launch rules of the tensor-core GEMMs, compiled for the host: tiles that cover every token once, rings that fit, the kernel
a call takes."""
import functools

import pytest

import gemm_plan as gp

SIZES = [97, 128, 129, 150, 160, 192, 193, 224, 256, 257, 300, 384, 400, 515, 576, 700, 768, 1000, 1152, 1500, 2044, 4096]
WIDTHS = [256, 1500, 4096, 6144, 8192, 10240, 19000, 28672, 57344, 128256]


@functools.lru_cache(None)
def plans():
    """One shape for every distinct launch of a few K blocks or many: rings, widths and the halves of a pair's first tiles."""
    seen = {}
    for M in SIZES:
        for N in WIDTHS:
            for K in (128, 384, 640, 4096, 16384):
                for a8 in (False, True):
                    p = gp.pair_plan(M, N, K, a8)
                    tiles, _ = gp.pair_tiles(p)
                    seen.setdefault((p.half_units, p.n_land, p.n_a, p.n_b, p.n_acc, tuple((t.u0, t.u1) for t in tiles[:8])), (M, N, K, a8))
    return sorted(seen.values())


def test_tiles_cover_the_tokens_and_rings_fit():
    for M, N, K, a8 in plans():
        p = gp.pair_plan(M, N, K, a8)
        assert p.n_land >= p.n_a >= 4 and p.n_b >= p.n_a and p.n_land * p.stage + p.n_b * p.slot <= 192 * 1024
        assert p.n_acc * p.acc_cols + 32 * p.n_a <= 512 and p.n_acc >= (2 if p.widest > p.half_units else 1)
        done = 0
        for i in range(p.t_tiles):
            t = gp.tile_at(p, i)
            assert (t.n0, t.t0) == (0, done) and 1 <= t.u0 <= 4 and 0 <= t.u1 <= t.u0 and (t.u1 == 0 or t.u0 == p.half_units)
            done += 32 * (t.u0 + t.u1)
        assert done - 32 < M <= done


@pytest.mark.parametrize("M,N,K,a8,want", [
    (8, 57344, 8192, False, "stream"), (16, 4096, 4096, False, "stream"), (9, 5120, 4096, False, "split"), (96, 57344, 8192, True, "split"),
    (128, 18944, 4096, False, "split"), (128, 18945, 4096, False, "pair_ts"), (256, 8192, 8192, False, "split"), (257, 8192, 8192, False, "pair_ts"),
    (4096, 57344, 8192, True, "pair"), (4096, 57344, 8192, False, "pair_ts"), (2044, 28672, 16384, True, "pair_ts"),
])
def test_route(M, N, K, a8, want):
    assert gp.route(M, N, K, a8) == want

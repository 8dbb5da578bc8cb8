"""The library's rules for a GEMM launch (csrc/pq_gemm_plan.cuh) compiled for the host with g++, for the tests that check them or choose
their shapes by them."""
import ctypes
import functools
import os
import subprocess
import tempfile

import paper_2410_05265_b200

CSRC = os.path.join(os.path.dirname(paper_2410_05265_b200.__file__), "csrc")
SMS = 148
ROUTES = ("stream", "split", "pair_ts", "pair")
FIELDS = ("c_tiles", "t_tiles", "base_units", "rem_units", "half_units", "box", "n_land", "n_a", "n_b", "n_acc", "stage", "slot", "acc_cols")
SHIM = r"""
#include "pq_gemm_plan.cuh"
using namespace pq_plan;
extern "C" {
int route(long long m, long long n, long long k, int a8, int sms) { return gemm_route(m, n, k, a8 != 0, sms); }
int plan(int m, int n, int n_kb, int a8, int sms, PairPlan* p) { return pair_plan(*p, m, n, n_kb, a8 != 0, sms); }
void tile(const PairPlan* p, int idx, Tile* t) { *t = tile_at(*p, idx); }
// of half h in the tiles first, first + step, ...: accumulator slot and parity of its round, or -1 where the tile has no such half
void acc_slots(const PairPlan* p, int h, int first, int step, int count, int* out) {
  AccRing u;
  for (int i = 0; i < count; ++i) {
    const Tile t = tile_at(*p, first + i * step);
    const Pos s = u.slot(h, *p);
    const bool on = (h ? t.u1 : t.u0) > 0;
    out[2 * i] = on ? s.i : -1, out[2 * i + 1] = s.ph;
    u.advance(h, t, *p);
  }
}
int width(int m) { return split_width(m); }
int splits_pairs(int tiles, int k, int m, int a8) { return split_count_pairs(tiles, k, 148, m, a8 != 0); }
int alone(int m, int ctas, int splits) { return split_alone(m, ctas, splits, 148); }
int alone_smem() { return SPLIT_ALONE_SMEM; }
int splits_whole(int tiles, int k) { return split_count(tiles, k, 148, 1); }
int width_whole(int m, int n, int k, int a8) { return split_width_whole(m, n, k, a8 != 0, 148); }
#define ROW(NT, A8) {NT, A8, SplitCfg<NT, A8>::TMEM_COLS, (int)split_smem<NT, A8>()}
int split_rows(int (*out)[4]) {
  const int rows[][4] = {ROW(16, 0), ROW(32, 0), ROW(48, 0), ROW(64, 0), ROW(96, 0), ROW(128, 0), ROW(192, 0), ROW(256, 0),
                         ROW(16, 1), ROW(32, 1), ROW(48, 1), ROW(64, 1), ROW(96, 1), ROW(128, 1), ROW(192, 1), ROW(256, 1)};
  for (int i = 0; i < 16; ++i)
    for (int j = 0; j < 4; ++j) out[i][j] = rows[i][j];
  return 16;
}
#define WHOLE_ROW(NT, A8) {NT, A8, SplitCfg<NT, A8, true>::TMEM_COLS, (int)split_smem<NT, A8, true>()}
int whole_rows(int (*out)[4]) {
  const int rows[][4] = {WHOLE_ROW(64, 0), WHOLE_ROW(128, 0), WHOLE_ROW(64, 1), WHOLE_ROW(128, 1)};
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) out[i][j] = rows[i][j];
  return 4;
}
}
"""


class Plan(ctypes.Structure):
    _fields_ = [(f, ctypes.c_int) for f in FIELDS]

    @property
    def widest(self):
        return self.base_units + (self.rem_units > 0)


class Tile(ctypes.Structure):
    _fields_ = [(f, ctypes.c_int) for f in ("n0", "t0", "u0", "u1")]


@functools.lru_cache(None)
def lib():
    with tempfile.TemporaryDirectory() as d:
        src, so = os.path.join(d, "plan.cpp"), os.path.join(d, "plan.so")
        with open(src, "w") as f:
            f.write(SHIM)
        subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", CSRC, src, "-o", so])
        dll = ctypes.CDLL(so)
    dll.route.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int] * 2
    return dll


def route(M, N, K, a8=False):
    return ROUTES[lib().route(M, N, K, int(a8), SMS)]


def pair_plan(M, N, K, a8=False):
    p = Plan()
    assert lib().plan(M, N, -(-K // 128), int(a8), SMS, ctypes.byref(p)), f"no rings for {M} x {N} x {K}"
    return p


def tile_at(p, idx):
    t = Tile()
    lib().tile(ctypes.byref(p), idx, ctypes.byref(t))
    return t


def pair_tiles(p, pair=0):
    """The tiles of one CTA pair, in its order, and for both halves the (slot, parity) of each."""
    n, pairs = p.c_tiles * p.t_tiles, min(p.c_tiles * p.t_tiles, SMS // 2)
    ids = list(range(pair, n, pairs))
    slots = []
    for h in range(2):
        out = (ctypes.c_int * (2 * len(ids)))()
        lib().acc_slots(ctypes.byref(p), h, pair, pairs, len(ids), out)
        slots.append([(out[2 * i], out[2 * i + 1]) for i in range(len(ids))])
    return [tile_at(p, i) for i in ids], slots


def split_shapes():
    """(tokens a tile, 8-bit tokens, tensor-memory columns, shared memory) of every form of the split-K kernel."""
    out = ((ctypes.c_int * 4) * 16)()
    n = lib().split_rows(out)
    return [tuple(out[i]) for i in range(n)]


def whole_shapes():
    """The same of the narrow forms that take an SM alone."""
    out = ((ctypes.c_int * 4) * 4)()
    n = lib().whole_rows(out)
    return [tuple(out[i]) for i in range(n)]


def width_whole(M, N, K, a8):
    """Width of the split-K kernel's token tiles above 128 tokens."""
    return lib().width_whole(M, N, K, int(a8))


def splits_pairs(tiles, K, M, a8):
    """K splits of a launch of the split-K kernel's forms of two CTAs to an SM."""
    return lib().splits_pairs(tiles, K, M, int(a8))


def alone(M, ctas, splits):
    """Is such a launch kept to one CTA to an SM?"""
    return bool(lib().alone(M, ctas, splits))


def alone_smem():
    return lib().alone_smem()


def splits_whole(tiles, K):
    """K splits of a launch of the split-K kernel's forms that take an SM alone."""
    return lib().splits_whole(tiles, K)

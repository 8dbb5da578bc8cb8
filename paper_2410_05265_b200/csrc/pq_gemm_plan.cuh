// What a GEMM call runs and in which shape: the kernel, its tiles, its rings and what they take of shared and tensor memory. Plain C++
// without a CUDA header, so that the rules are compiled for the host, too, and walked over all sizes by tests/test_gemm_plan.py.
#pragma once

#include <math.h>
#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define PQ_HD __host__ __device__ __forceinline__
#else
#define PQ_HD inline
#endif

namespace pq_plan {

constexpr int BK = 128;                     // K elements per stage
constexpr int PK_ROW = BK / 2;              // packed bytes per row per stage
constexpr int A_SLOT_COLS = BK / 4;         // 32 columns of tensor memory = 128 K bytes per lane

// ---- which kernel ---------------------------------------------------------------------------------
enum Route { STREAM, SPLIT, PAIR_TS, PAIR };

// The kernel for m rows.
// Weight-streaming kernel or split-K tensor-core kernel (figures: rotate+quantize and GEMM in a graph, us, streaming against
// split). The streaming kernel has the shorter chain, but expands the tokens again for every 16 channels and has no K split:
//   up to 8 tokens   streaming; the other one for a long K, where a CTA of the streaming kernel walks rows alone (8192 x 28672, 1 token: 29 / 24;
//                    whole 70B decode layer 117.8 / 114.1). On 8192 x 8192 it is faster alone (11.4 / 10.4), but inside a decode layer the streaming
//                    kernel's shorter chain and earlier weight requests win (124 / 132 with every layer on the other)
//   9 to 16 tokens   only layers below 20 M weights (16 tokens, 4096 x 4096: 5.6 / 7.1; 6144 x 4096: 8.1 / 7.8,
//                    28672 x 4096: 21.3 / 15.7, 8192 x 28672: 33.9 / 26.0)
//   up to 96         always split (CTA pairs: 40 tokens, 28672 x 4096: 23.0 / 19.8; 8192 x 28672: 59.5 / 31.6)
//   97 to 128        while every channel tile has an SM at once (128 tokens, pairs against split, 57344 x 8192: 74.6 / 85.7,
//                    28672 x 4096: 25.1 / 27.0; but 10240 x 8192: 25.3 / 23.5); 8-bit tokens, whose expansion is shorter, while every
//                    channel tile has one of the two CTAs of an SM (28672 x 4096 22.8 / 23.0, 28672 x 8192 39.6 / 38.1, 20480 x 4096
//                    21.8 / 21.0; but 38912 x 4096 30.6 / 36.2, 45056 x 8192 54 / 64, 57344 x 8192 66.0 / 68.8, 128256 x 8192 122 / 136)
//   above            while the 256-token tiles leave room for two K splits (pairs against split at 256 tokens: 8192 x 8192 26.0 / 23.5,
//                    4096 x 14336 35.7 / 24.2, 6144 x 4096 17.4 / 17.2; at 400, 4096 x 14336 37.8 / 31.9, 4096 x 4096 17.7 / 17.3). With a single
//                    split the pairs win: 57344 x 8192 at 200 tokens 91 / 129, 28672 x 4096 30.1 / 39.3, 10240 x 8192 31.5 / 35.8, 6144 x 4096
//                    at 300 17.9 / 21.7, 4096 x 14336 at 515 39.2 / 49.4.
// CTA pairs: weights in tensor memory, tiles as wide as fit the chip (pq_gemm_tc3.cu), or for 8-bit tokens both operands in shared
// memory, whole tiles of 256 tokens and two whole accumulators (pq_gemm_tc2.cu). The second takes launches of more than three rounds, 2048 <= K <= 8192
// and 1024 tokens and more, of which its whole tiles pad at most a twentieth: it is up to a tenth faster per padded token, and as much
// slower where it pads more or where its longer start-up shows. With the rotation, us, first / second kernel: 28672 x 4096 at 300 tokens 39.5 / 57,
// 515 52 / 67, 800 75 / 85, 1024 89 / 89, 1100 92 / 101, 1500 126 / 121, 1664 131 / 137, 2044 164 / 154, 2100 165 / 170, 3000 231 / 223,
// 4096 315 / 296; 57344 x 8192 at 129 82 / 108, 515 180 / 224, 1024 305 / 308, 1100 330 / 368, 1280 380 / 372, 2044 619 / 564, 2100 601 / 621,
// 4096 1204 / 1083; 28672 x 1024 at 4096 109 / 127, 28672 x 2048 181 / 166; 10240 x 8192 at 1500 98 / 101, 3000 173 / 170, 4096 229 / 222; 128256 x 4096 at 1024 357 / 340.
inline Route gemm_route(int64_t m, int64_t N, int64_t K, bool a8, int sm_count) {
  const int64_t ctiles = (N + 127) / 128, weights = N * K;
  const bool split = m <= 8     ? K > 16384
                     : m <= 16  ? weights >= (int64_t{20} << 20)
                     : m <= 96  ? true
                     : m <= 128 ? ctiles <= (a8 ? 2 : 1) * sm_count
                                : 2 * ((m + 255) / 256) * ctiles <= sm_count * 7 / 8;
  if (split) return SPLIT;
  if (m <= 16) return STREAM;
  const int64_t t_tiles = (m + 255) / 256, tiles = t_tiles * ((N + 255) / 256);
  return a8 && K >= 2048 && K <= 8192 && m >= 1024 && 20 * m >= 19 * 256 * t_tiles && tiles > 3 * (sm_count / 2) ? PAIR : PAIR_TS;
}

// A position in a ring of n slots and the parity of its current round.
struct Pos {
  int i = 0, ph = 0;
  PQ_HD void advance(int k, int n) {  // k <= n
    i += k;
    if (i >= n) i -= n, ph ^= 1;
  }
};

// ---- CTA pairs, weights in tensor memory (pq_gemm_tc3.cu) --------------------------------------------
constexpr int UNIT = 32;                    // tokens: granularity of a tile's width (N of a 256-row pair MMA comes in steps of 32)
constexpr int MAX_UNITS = 8;
constexpr int CH_CTA = 128;                 // output channels per CTA (256 per pair)
constexpr int W_STAGE = CH_CTA * PK_ROW;    // 8 KB of packed weights per K block
constexpr int MAX_LAND = 8, MAX_A = 8, MAX_B = 8, MAX_ACC = 4;  // rings: landing stages, operand slots, accumulator halves
constexpr int N_GROUPS = 4;                 // expansion groups
constexpr int PAIR_TMEM_COLS = 512;
constexpr int RING_BYTES = 192 * 1024;      // landing stages and token operands

struct PairPlan {
  int c_tiles, t_tiles;    // tiles along the channels and along the tokens
  int base_units, rem_units;  // token tile i is base_units + (i < rem_units) units wide
  int half_units;          // units of a tile's first half (as far as it has so many): half of the widest tile's
  int box;                 // token rows per TMA box and of a CTA's share of a first half
  int n_land, n_a, n_b, n_acc;  // ring lengths (4-bit tokens: n_b = n_a, the two operand rings turn together)
  int stage, slot, acc_cols;    // bytes of a landing stage and of a token operand slot, columns of an accumulator half
};

struct Tile {
  int n0, t0;  // first channel, first token
  int u0, u1;  // units of the two halves (u1 = 0: one half)
};
PQ_HD Tile tile_at(const PairPlan& p, int idx) {
  const int c = idx / p.t_tiles, i = idx - c * p.t_tiles;  // the token tiles of a channel tile are neighbours: its weights are in L2
  const int units = p.base_units + (i < p.rem_units ? 1 : 0);
  Tile t;
  t.n0 = c * 2 * CH_CTA;
  t.t0 = (i * p.base_units + (i < p.rem_units ? i : p.rem_units)) * UNIT;
  t.u0 = units < p.half_units ? units : p.half_units;
  t.u1 = units - t.u0;
  return t;
}

// The accumulator slots one half of a pair's tiles takes in turn: half 0 the even ones, half 1 the odd ones. A slot has one issuer and
// one group of epilogue warps, which wait for every phase of its barriers in order, so that the parity they wait for cannot be
// that of two rounds back. (Slots that both halves took in turn, as three did, were waited on by warps that had not seen the phase
// before: a half could be read before it was written, in principle.) Three slots of up to 96 columns, two for the first half and one for the
// second, against one each and against two each with four A slots (us, with the rotation): 300 x 28672 x 4096 42.9 / 44.1 / 45.8,
// 515 x 28672 x 4096 54.1 / 54.8 / 56.7, 515 x 57344 x 8192 179 / 179 / 189.
struct AccRing {
  Pos u;
  PQ_HD Pos slot(int h, const PairPlan&) const {
    Pos s = u;
    s.i = 2 * u.i + h;
    return s;
  }
  PQ_HD void advance(int h, const Tile& t, const PairPlan& p) {
    if ((h ? t.u1 : t.u0) > 0) u.advance(1, (p.n_acc + 1 - h) / 2);
  }
};

// The number of token tiles per channel tile: the one with the shortest estimate for the launch, in whole rounds of the chip's pairs.
// Clocks of a K block, measured on one round of tiles of 64, 128, 192 and 256 tokens (K = 4096 and 8192): 458, 472, 497, 578 (8-bit tokens
// 397, 416, 452, 578): wide tiles take their MMAs' time (64 clocks per unit) and a little, narrow ones that of the expansion and of
// the issue, which hardly depend on the width. A tile adds about 1800 clocks of its own. Gains, narrower tiles against the widest (us,
// with the rotation): 1000 x 6144 x 4096 34.2 / 41, 1000 x 4096 x 4096 21.5 / 24.6, 1500 x 4096 x 14336 76 / 86.
// With more than three rounds of the widest tiles those stay: the ragged round weighs less there, the chip runs at its power limit, and
// narrower tiles expand the weights more often (2044 x 28672 x 4096: 169 with nine tiles, 156 with eight).
inline int tile_rule(int units, int c_tiles, int n_pairs, int n_kb) {
  int best = 0;
  double best_clocks = 0.0;
  const int t_min = (units + MAX_UNITS - 1) / MAX_UNITS;
  if (c_tiles * t_min > 3 * n_pairs) return t_min;
  for (int t = t_min; t <= units && t <= t_min + 8; ++t) {
    const int rounds = (c_tiles * t + n_pairs - 1) / n_pairs;
    auto tile = [n_kb](double w) { return n_kb * fmax(72.0 * w, 440.0 + 9.0 * w) + 1800.0; };
    const double mean = static_cast<double>(units) / t, widest = (units + t - 1) / t;
    const double clocks = (rounds - 1) * tile(mean) + tile(widest);
    if (best == 0 || clocks < best_clocks) best = t, best_clocks = clocks;
  }
  return best;
}

// False when the rings do not fit (no size known).
inline bool pair_plan(PairPlan& p, int M, int N, int n_kb, bool a8, int sm_count) {
  const int units = (M + UNIT - 1) / UNIT;
  p.c_tiles = (N + 2 * CH_CTA - 1) / (2 * CH_CTA);
  p.t_tiles = tile_rule(units, p.c_tiles, sm_count / 2, n_kb);
  p.base_units = units / p.t_tiles;
  p.rem_units = units % p.t_tiles;
  const int widest = p.base_units + (p.rem_units > 0 ? 1 : 0);
  p.half_units = (widest + 1) / 2;
  p.box = p.half_units * (UNIT / 2);
  const bool two = widest > p.half_units;
  p.acc_cols = p.half_units * UNIT;
  p.n_acc = (PAIR_TMEM_COLS - 7 * A_SLOT_COLS) / p.acc_cols;  // what seven A slots leave
  if (p.n_acc > MAX_ACC) p.n_acc = MAX_ACC;
  p.n_a = (PAIR_TMEM_COLS - p.n_acc * p.acc_cols) / A_SLOT_COLS;
  if (p.n_a > MAX_A) p.n_a = MAX_A;
  p.slot = (two ? 2 : 1) * p.box * BK;
  p.stage = W_STAGE + (a8 ? 0 : (two ? 2 : 1) * p.box * PK_ROW);
  p.n_b = MAX_B;
  if (!a8) {
    while (p.n_a > 6 && p.n_a * p.slot + 7 * p.stage > RING_BYTES) --p.n_a;
    p.n_b = p.n_a;
  }
  p.n_land = (RING_BYTES - p.n_b * p.slot) / p.stage;
  if (p.n_land > MAX_LAND) p.n_land = MAX_LAND;
  return p.n_land >= p.n_a && p.n_b >= p.n_a && p.n_a >= N_GROUPS && p.n_acc >= 2;  // the kernel's parities rely on it
}

// ---- split K (pq_gemm_split.cu) -----------------------------------------------------------------------
constexpr int CH = 128;                    // output channels per CTA
constexpr int SPLIT_BAR_BYTES = 512;       // no less than the kernel's barriers take

// Shapes of the rings. Up to 128 tokens two CTAs share an SM (112 KB and 256 TMEM columns each), so that one loads
// while the other expands or reduces; 256 tokens take a whole SM. K blocks of 256 elements, whose weight rows are 128 bytes (why: pq_gemm_split.cu),
// where the rings hold enough of them: two operand slots, one per expansion group, and as many landing stages as fit beside them. us, rotation and
// GEMM in a graph: 64 x 57344 x 8192 62.9 (128 elements) / 62.5 (256, four weight stages and two of tokens) / 59.5 (three and three);
// 8-bit tokens, 128 x 28672 x 4096 22.6 / 23.0 (two stages) / 20.2 (three). At 96 and 128 packed tokens the landing stages of the tokens leave no room.
constexpr int split_kb(int nt, bool a8, bool whole) { return nt <= (a8 && !whole ? 128 : 64) ? 256 : 128; }

// WHOLE: one CTA to an SM, four expansion groups (above 128 tokens).
template <int NT, bool A8, bool WHOLE = (NT > 128)>
struct SplitCfg {
  static constexpr int KB = split_kb(NT, A8, WHOLE), SUBS = KB / BK;  // elements of a K block
  static constexpr int ROWB = KB / 2;                          // packed bytes of a row in it
  static constexpr int GROUPS = WHOLE ? 4 : 2;
  static constexpr int SLOTS = !WHOLE && (KB == 256 || (NT == 128 && !A8)) ? 2 : 4;
  static constexpr int W_STAGE = CH * ROWB;
  static constexpr int STAGES = WHOLE ? (NT <= 128 ? 8 : 4) : KB == 128 ? 4 : (NT <= 16 ? 6 : (NT <= (A8 ? 96 : 48) ? 4 : 3));  // landing ring, weights
  static constexpr int X_STAGES = !WHOLE && KB == 256 && NT > 48 ? 3 : 4;                                               // landing ring, tokens
  static constexpr bool TOGETHER = KB == 256;  // weights and tokens of a K block are waited for together
  static constexpr bool SLOT_FIRST = STAGES % GROUPS != 0 || (!A8 && X_STAGES % GROUPS != 0);
  static constexpr bool EARLY_W = NT > 128;          // weight stages go back before the (long) token part of the expansion
  static constexpr int X_STAGE = A8 ? 0 : NT * ROWB;
  static constexpr int SUB_SLOT = NT * BK;           // token operand of 128 elements
  static constexpr int SLOT = SUBS * SUB_SLOT;
  static constexpr int A_COLS = SUBS * A_SLOT_COLS;
  static constexpr int A_COL0 = NT < 32 ? 32 : NT;  // accumulator columns, then the A slots
  static constexpr int TMEM_COLS = WHOLE ? 512 : 256;
  static constexpr int CTAS_PER_SM = WHOLE ? 1 : 2;
  static constexpr int RING = SLOTS * SLOT + STAGES * W_STAGE + X_STAGES * X_STAGE;
  static constexpr int PART = NT * CH * 4;  // the int32 partial tile, laid over the rings at the end
  static_assert(A_COL0 + SLOTS * A_COLS <= TMEM_COLS, "tensor memory budget");
  static_assert(SLOTS % GROUPS == 0, "an operand slot is always served by the same group");
  static_assert(SLOTS <= X_STAGES, "what frees an operand slot has landed in both rings");
  static_assert(PART <= RING, "the partial tile fits where the rings were");
  static_assert(SLOTS <= STAGES, "no weight stage is refilled before the first operand slot is");
  static_assert((RING + SPLIT_BAR_BYTES + 1024) * CTAS_PER_SM <= 228 * 1024, "shared memory budget");
};

// At least 80 KB for 256 columns of tensor memory and 160 KB for 512, so that no more CTAs share an SM (228 KB) than its tensor memory
// serves, those of other launches included: a CTA that waited for columns which another cluster's CTA gives back only behind its
// cluster barrier could wait for itself. (8-bit tokens 192 wide need 130 KB, which leave room for a CTA of a narrow form.)
// From 33 to 96 tokens half of an SM's shared memory, also where the rings need less: otherwise CTAs of the next rotation find room beside two of these,
// and let the launch behind them in among the running ones, on whichever SMs have room. us, rotation and GEMM in a graph, rings alone / half: 8-bit
// tokens 56 x 6120 x 3456 13.2 / 10.6, 50 x 9248 x 1280 9.3 / 8.0, 59 x 6320 x 3712 13.3 / 11.5, 62 x 4584 x 2944 11.4 / 10.3; linear sets equal. Up to
// 32 tokens it is a toss-up (4-bit 24 x 2816 x 14720 13.5 / 12.0, 28 x 4440 x 7680 10.3 / 12.6) and at 128 a loss (97 to 128 tokens 1.5 % in the mean of 58 shapes).
// Nor more than the rings of 8-bit tokens 32 wide hold now, 80 KB: with six weight stages, 112 KB, 24 x 4608 x 6912 went 10.6 -> 12.8 us, and no shape gained.
template <int NT, bool A8, bool WHOLE = (NT > 128)>
constexpr size_t split_smem() {
  const size_t need = SplitCfg<NT, A8, WHOLE>::RING + SPLIT_BAR_BYTES, least = WHOLE ? 160 * 1024 : (NT > 32 && NT < 128 ? 113 : 80) * 1024;
  return need < least ? least : need;
}

constexpr int MAX_SPLIT = 8;  // portable cluster size

// As many K splits as leave every CTA resident at once with room for the clusters to be placed (7/8 of the slots: 48 tiles
// x 6 = 288 CTAs ran in two waves, 10.7 us against 7.0 with 96), and at least 640 elements of K per CTA (below that the two
// cluster barriers cost more than the shorter loop saves: 4096 x 4096 at 32 tokens 6.1 us with six splits, 6.6 with eight).
// The splits share whole K blocks, so that their shares can differ by one (16 blocks over five CTAs); the fewest splits with the same longest share
// lose all the same, because fewer CTAs read: 48 x 6144 x 4096, five / four splits, 9.6 / 10.2, per token at 32 8.0 / 9.3, 8B linear set at 32 47.9 / 48.8.
// A cluster's CTAs lie in one GPC: of clusters of seven or eight with a CTA to an SM only fifteen find a place (cudaOccupancyMaxActiveClusters; 22, 26, 33, 45
// of six, five, four, three, so that 7/8 of the SMs is the lower line there). The sixteenth ran behind the others: 345 x 768 x 14336, eighteen tiles, seven splits / six,
// 24.3 / 15.8 us, W4A8 160 x 1152 x 14336 20.3 / 13.4, 200 x 2176 x 8192 24.7 / 15.1. Two CTAs to an SM find 37 of seven and 33 of eight.
inline int split_count(int tiles, int K, int sm_count, int per_sm) {
  int splits = sm_count * per_sm * 7 / 8 / tiles;
  if (splits > MAX_SPLIT) splits = MAX_SPLIT;
  if (per_sm == 1 && splits > 6 && tiles > 15 * sm_count / 148) splits = 6;
  if (splits > K / (5 * BK)) splits = K / (5 * BK);
  return splits < 1 ? 1 : splits;
}

// The forms of which two CTAs share an SM. Above 64 tokens the partial tiles are large, and an SM's two CTAs exchange theirs at the same
// time: one CTA to an SM and fewer splits, of at least 1280 elements of K, win with a short K, and with 8-bit tokens above 88 while that leaves four
// splits. us with the rotation, two to an SM / one (before such launches were kept to one, see split_alone): W4A8 at 96 tokens 6144 x 4096 five splits 11.9 / two 10.0, 4096 x 4096 six 11.2 / three 9.6, 4096 x 14336
// eight 16.6 / four 14.4 (at 80 15.5 / 16.3), but 8192 x 8192 four 15.7 / two 16.3, 8192 x 28672 four 30.6 / two 36.4; 4-bit 4096 x 4096 at 96 11.9 / 10.6,
// at 128 six 13.4 / three 11.9 (four 13.7), 6144 x 4096 at 96 12.9 / 13.3, at 128 15.2 / 13.8, 4096 x 14336 at 80 18.0 / 20.2; at 64 tokens 4096 x 14336
// eight 15.3 / four 17.6.
inline int split_count_pairs(int tiles, int K, int sm_count, int M, bool a8) {
  const int two = split_count(tiles, K, sm_count, 2), one = sm_count * 9 / 10 / tiles, most = K / (10 * BK);
  const bool short_k = K <= 16 * BK * one;
  const bool fewer = M > 64 && two * tiles > sm_count && one >= 2 && (short_k ? a8 || M > 96 || one >= 4 : a8 && M > 88 && one >= 4);
  return fewer && most >= 1 ? (one < most ? one : most) : two;
}

// Is a launch of those forms kept to one CTA to an SM? Above 64 tokens, when the CTAs have an SM each (7/8 of the SMs, clusters of four at most: a
// cluster of eight does not find eight free ones everywhere) and are more than half of the SMs. It then asks for more than half of an SM's shared
// memory. Otherwise its CTAs, placed while the rotation kernel before them still holds a part of the SMs, shared the others by twos. us, rotation and GEMM issued
// into a stream, by twos / alone: 100 x 4096 x 4096 14.3 / 11.9 (before one CTA to an SM was the rule 13.4), 112 x 6144 x 4096 16.5 / 13.9, W4A8 100 x 4096 x 4096
// 12.6 / 11.0, 96 x 4096 x 14336 15.3 / 14.7; linear set in a graph, 4-bit at 112 tokens 78.1 / 73.1, W4A8 at 96 57.1 / 55.0, per token at 128 81.3 / 77.0.
// Without the three conditions: 20 x 2048 x 8192 (clusters of eight) 7.7 / 11.5, 48 x 4096 x 2048 7.1 / 7.6, W4A8 96 x 2048 x 4096 (48 CTAs) 8.6 / 10.0.
constexpr int SPLIT_ALONE_SMEM = 120 * 1024;
inline bool split_alone(int M, int ctas, int splits, int sm_count) {
  return M > 64 && 2 * ctas > sm_count && ctas <= sm_count * 7 / 8 && splits <= 4;
}

// The width of the token tiles up to 128 tokens.
inline int split_width(int M) { return M <= 16 ? 16 : (M <= 32 ? 32 : (M <= 48 ? 48 : (M <= 64 ? 64 : (M <= 96 ? 96 : 128)))); }

// The width above 128 tokens, by the estimate of a launch (one CTA to an SM): K blocks per CTA times what 128 elements of one take at that
// width, and what the partial tiles cost that cross the cluster. Their sums move at some 25 bytes per ns and SM (four splits of 256 tokens: 96 KB per
// CTA, 4 us), so a launch that leaves SMs idle at 256 tokens takes narrower tiles rather than more splits, although the weights are then
// expanded more often. us per 128 elements at 64, 128, 192, 256 tokens: 0.164, 0.275, 0.36, 0.385, with 8-bit tokens 0.13, 0.21, 0.31, 0.33.
// us with the rotation, 192 or 256 tokens wide -> by this rule: 256 x 4096 x 4096 15.2 -> 12.8 (two splits of 128), 192 x 6144 x 4096 14.9 -> 13.1 (64),
// W4A8 256 x 4096 x 4096 14.9 -> 12.1, 256 x 4096 x 14336 23.1 -> 21.7, 512 x 4096 x 4096 15.6 -> 15.2.
inline int split_width_whole(int M, int N, int K, bool a8, int sm_count) {
  const int widths[] = {64, 128, 192, 256};
  const double us4[] = {0.164, 0.275, 0.36, 0.385}, us8[] = {0.13, 0.21, 0.31, 0.33};
  int best = 0;
  double best_us = 0.0;
  for (int i = 0; i < 4; ++i) {
    const int t_tiles = (M + widths[i] - 1) / widths[i], tiles = t_tiles * ((N + CH - 1) / CH), splits = split_count(tiles, K, sm_count, 1);
    const int rounds = (tiles * splits + sm_count - 1) / sm_count, blocks = ((K + BK - 1) / BK + splits - 1) / splits;
    const double tokens = (M + t_tiles - 1) / t_tiles;
    const double us = rounds * blocks * (a8 ? us8 : us4)[i] + tokens * tokens * (splits - 1) / splits * (4.5 / 65536);
    if (best == 0 || us < best_us) best = widths[i], best_us = us;
  }
  return best;
}

}  // namespace pq_plan

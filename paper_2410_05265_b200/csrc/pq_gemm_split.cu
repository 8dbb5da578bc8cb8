// W4A4 / W4A8 GEMM for a few tens to a few hundred tokens (batched decode, short prompts):
//
//   acc[t,n] = sum_k xq[t,k] * wq[n,k]   (exact int32),   out = bf16(acc * s_a * s_w[n])
//
// At these sizes the packed weights are what has to move, and the 256 x 256 tiles of the CTA-pair kernels leave most
// of the chip idle (16 tiles for a 4096 x 4096 layer). Here the MMA is turned round: 128 output channels are its row
// side, NT = 16 .. 256 tokens its column side, so a token tile costs what its tokens cost, and the K blocks of a
// channel tile are split over the CTAs of a cluster (up to 8), whose int32 partial tiles meet in distributed shared
// memory: exact, no workspace, nothing waits on another cluster.
//
// Roles inside a CTA:
//   warp 0      TMA producer, packed weights: a K block of 256 elements [128 x 128 B] (128 at the widest token tiles) into a landing ring.
//               Weights are static: the ring's first copies start before the wait for the previous kernel in the stream.
//   warp 1      MMA issuer and owner of the tensor memory.
//   warp 2      TMA producer, tokens: packed rows [NT x 64 B per 128 elements] into a landing ring of their own, or (A8) the s8 bytes
//               straight into the operand slot (128-byte-swizzled box).
//   warps 4..   expansion, GROUPS groups of four warps (one per TMEM lane quarter): a thread owns one channel row, reads
//               its packed bytes, and writes the s8 bytes (16 * code) to its lane of an A slot in tensor memory; the
//               group's threads also expand the token rows into the B slot in shared memory. Of every 32 codes the even-position ones come
//               first, then the odd-position ones, in both operands (natural order in both with A8).
// Then every warp takes part in the reduction: a lane owns four channels, a warp one or more tokens at a time, the partial
// sums of the cluster's CTAs are added, scaled and stored as 256 contiguous bytes per token.
//
// What bounds it: up to ~64 tokens the weight stream and the fixed chain launch -> tokens -> expand -> MMA -> two cluster
// barriers (about 5 us, most of it overlapped with the neighbours under programmatic dependent launch); at 128 and 256 tokens
// the expansion of the token rows, which every channel tile repeats.
//
// Why a K block has 256 elements: copies of 64 bytes a row do not reach the memory's rate. Copies alone, without any arithmetic (TB/s, the
// same CTAs and bytes in flight): 57344 x 4096 bytes 64-byte rows 4.9, 128-byte rows 5.8-6.3; 28672 x 2048 bytes 4.0 / 4.7. A K block also has a fixed
// price, three waits, three arrivals and a proxy fence, about half of its 1200 clocks, and an mbarrier arrival is the dearest of
// them (it waits for the thread's stores): those that come together are one instruction with a lane each. us, GEMM alone over
// weight copies larger than L2, 64-byte rows / now:
//   4-bit, 33 tokens: 6144 x 4096 8.9 / 8.0, 4096 x 4096 8.4 / 7.5, 28672 x 4096 19.0 / 16.9, 4096 x 14336 13.0 / 11.7, 57344 x 8192 58.9 / 51.2
//   4-bit, 16 tokens: 28672 x 4096 14.8 / 14.2, 57344 x 8192 50.8 / 46.3, 8192 x 28672 24.0 / 22.7, 10240 x 8192 11.5 / 10.4
//   8-bit, 96 tokens: 6144 x 4096 11.1 / 10.1, 4096 x 4096 10.6 / 9.5, 28672 x 4096 20.2 / 17.5, 4096 x 14336 15.8 / 14.5, 57344 x 8192 63.1 / 58.5
//   8-bit, 128 tokens: 28672 x 4096 21.0 / 19.0, 8192 x 28672 34.1 / 32.2
// Tried: the token rows read from L2 into registers instead of a landing ring (gate|up, M = 32: 16.2 us against 14.3); token
// rows expanded by warps of their own (18.1); three or four expansion groups per CTA (14.9-15.2); a weight stage handed back
// right after it was read into registers, which pays only where the token part is long (M = 256, gate|up: 46.5 -> 36.4); with 64-byte rows,
// one vote for the three waits (33 x 28672 x 4096 19.1 -> 21.0: the weights are no longer expanded while the tokens are on their way); tokens
// before weights, or their stage handed back at once (64 x 28672 x 4096 19.2 -> 21.9); the K blocks of several tiles dealt evenly over a cluster
// (five CTAs for four tiles of 28672 x 4096, so that all SMs have the same share: 17.0 -> 20.9; the memory, not the fullest SM, sets the time).
//
// Every mbarrier wait is bounded; when one runs out the CTA raises an abort flag, its roles drain, and PQ_ERR_TIMEOUT
// is reported.
#include "pq_gemm_pair.cuh"

namespace {

using namespace pq_pair;
using namespace pq_plan;

constexpr int EXPAND_WARP0 = 4;

template <int NT, bool A8, bool WHOLE>
struct Cfg : SplitCfg<NT, A8, WHOLE> {
  static constexpr int THREADS = (EXPAND_WARP0 + 4 * Cfg::GROUPS) * 32;
};

struct __align__(8) SplitBarriers {
  uint64_t w_full[8], w_empty[8];             // landing ring of packed weights
  uint64_t xp_full[8], xp_empty[8];             // landing ring of packed tokens
  uint64_t s8_full[4], s8_empty[4], x_full[4];  // operand slots
  uint64_t acc_full;
  uint32_t tmem_base;
  volatile int abort_flag;
};

static_assert(sizeof(SplitBarriers) <= SPLIT_BAR_BYTES, "shared memory budget");

// When the next kernel of the stream may be placed (see pq_launch_pdl). Up to 32 tokens, when it is as small, at once. From 33 to 96 in a captured
// graph, as a decode loop keeps one, when a cluster begins its reduction, and up to 128 with a step per token. us per pass, never / then, 8B linear set:
//   4-bit    33 tokens 52.6 / 50.3, 48 54.2 / 51.9, 64 59.9 / 58.0, 96 72.8 / 70.9, 112 76.5 / 77.7, 128 77.6 / 79.2
//   8-bit    33 50.0 / 48.3, 64 56.2 / 53.3, 80 60.5 / 57.9, 112 64.6 / 66.2, 128 65.5 / 67.7
//   per token 33 57.4 / 55.1, 64 61.9 / 60.1, 112 81.2 / 79.7, 128 82.4 / 81.5;    70B set, 4-bit, 33 111.3 / 109.1, 96 158.2 / 156.5, 128 161.7 / 162.1
// (behind the K loop 51.3 at 33, 62.8 at 64.) A chain of one shape does not always gain: of 163 shapes of 33 to 96 tokens the mean is 0.989, but 4096 x 14336 with steps
// per token, whose quantizer takes a CTA a row, goes 20.5 / 16.8 at 49 tokens, 15.5 / 17.4 at 53 to 64 and 18.3 / 19.6 at 80. Above 96 tokens
// 127 x 2816 x 14720 goes 20.0 / 22.3. Calls issued into a stream lose by it (8B set with steps per token at 33 tokens 54.5 / 56.4, 70B set at 33
// 106.8 / 109.3), as do larger ones (256 x 4096 x 4096 13.0 / 14.5): so they ask whether the stream is being captured.
enum Early { NEVER, AT_ENTRY, AT_REDUCTION };

struct SplitParams {
  const int32_t* zp;
  const int32_t* wsum;
  const float* s_row;  // per-token steps or null
  const float* s_a;
  const float* s_w;
  __nv_bfloat16* out;
  int32_t* acc_dbg;
  int32_t* status;
  int64_t ldo;
  int M, N, K, n_kb;
  int t_tiles, splits, early;
  int vec_out;  // rows of out take 8-byte stores
  long long wait_clocks;
};

// D[tmem] (+)= A[tmem] * B[smem], s8 x s8 -> s32, one thread.
__device__ __forceinline__ void mma_i8_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 32 lanes x 16 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ int4 ld_cluster_int4(uint32_t addr) {
  int4 v;
  asm volatile("ld.shared::cluster.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}

// Adds the partial tiles of the cluster's CTAs (at most PEERS), scales and stores: a warp takes tokens first, first + step,
// ..., U of them at a time so that their shared-memory loads are in flight together; a lane owns four channels.
template <int PEERS, int U, bool ZP>
__device__ __forceinline__ void reduce_tile(const SplitParams& p, const uint8_t* part, int t0, int n0, int tokens, int first, int step,
                                            int lane, const float (&sw)[4], const int (&zw)[4]) {
  const int n = n0 + 4 * lane;
  uint32_t peer[PEERS];
#pragma unroll
  for (int r = 0; r < PEERS; ++r) peer[r] = map_to_cta(part, r < p.splits ? r : 0) + lane * 16;
  for (int tb = first; tb < tokens; tb += U * step) {
    int4 v[U][PEERS];
    float rs[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = tb + u * step < tokens ? tb + u * step : tb;
#pragma unroll
      for (int r = 0; r < PEERS; ++r) {
        if (PEERS == 1) v[u][r] = *reinterpret_cast<const int4*>(part + t * (CH * 4) + lane * 16);
        else v[u][r] = r < p.splits ? ld_cluster_int4(peer[r] + t * (CH * 4)) : make_int4(0, 0, 0, 0);
      }
      rs[u] = p.s_row ? pq::ld_dep(p.s_row + t0 + t) : 1.0f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = tb + u * step;
      if (t >= tokens) break;
      int sum[4] = {0, 0, 0, 0};
#pragma unroll
      for (int r = 0; r < PEERS; ++r) sum[0] += v[u][r].x, sum[1] += v[u][r].y, sum[2] += v[u][r].z, sum[3] += v[u][r].w;
      float f[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (ZP) sum[i] -= zw[i];
        f[i] = static_cast<float>(sum[i]) * sw[i] * rs[u];
      }
      __nv_bfloat16* dst = p.out + static_cast<int64_t>(t0 + t) * p.ldo + n;
      if (p.vec_out && n + 3 < p.N) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(f[0], f[1]), hi = __floats2bfloat162_rn(f[2], f[3]);
        *reinterpret_cast<uint2*>(dst) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (n + i < p.N) dst[i] = __float2bfloat16_rn(f[i]);
      }
      if (p.acc_dbg) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (n + i < p.N) p.acc_dbg[static_cast<int64_t>(t0 + t) * p.N + n + i] = sum[i];
      }
    }
  }
}

template <int NT, bool A8, bool ZP, bool WHOLE>
__global__ void __launch_bounds__(Cfg<NT, A8, WHOLE>::THREADS, Cfg<NT, A8, WHOLE>::CTAS_PER_SM)
    gemm_w4_split_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w, const SplitParams p) {
  using C = Cfg<NT, A8, WHOLE>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw;
  uint8_t* slot_buf = smem;                                // SLOTS token operands [NT x 128 B], 128-byte swizzle
  uint8_t* stage_buf = slot_buf + C::SLOTS * C::SLOT;      // STAGES landing buffers of packed weights
  uint8_t* x_buf = stage_buf + C::STAGES * C::W_STAGE;     // X_STAGES landing buffers of packed tokens
  SplitBarriers* bars = reinterpret_cast<SplitBarriers*>(smem + C::RING);
  volatile int* abort_flag = &bars->abort_flag;
  if (pq::smem_u32(smem_raw) & 1023) {  // the swizzled buffers need it (no slack is kept: two CTAs share the SM to the last kilobyte)
    if (threadIdx.x == 0) pq::report(p.status, PQ_ERR_ALIGN);
    return;
  }
  const int warp = pq::warp_index(), lane = threadIdx.x & 31;
  const int rank = __shfl_sync(0xffffffffu, static_cast<int>(cluster_ctarank()), 0);
  const int tile = static_cast<int>(blockIdx.x) / p.splits;
  const int t0 = (tile % p.t_tiles) * NT;  // the token tiles of a channel tile are neighbours: its weights are in L2
  const int n0 = (tile / p.t_tiles) * CH;
  const int kb0 = static_cast<int>(static_cast<int64_t>(p.n_kb) * rank / p.splits);
  const int total = static_cast<int>(static_cast<int64_t>(p.n_kb) * (rank + 1) / p.splits) - kb0;  // K blocks of this CTA

  if (p.early == AT_ENTRY) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const bool leader = pq::elect_one();  // the lane that issues copies and MMAs (each role's loop is warp-uniform)
  const int first = total < C::STAGES ? total : C::STAGES;
  if (warp == 0) {
    if (leader) {
      pq::tma_prefetch_desc(&tmap_w);
      pq::tma_prefetch_desc(&tmap_x);
      for (int i = 0; i < C::STAGES; ++i) {
        pq::mbar_init(&bars->w_full[i], 1);
        pq::mbar_init(&bars->w_empty[i], 4);
      }
      for (int i = 0; i < C::X_STAGES; ++i) {
        pq::mbar_init(&bars->xp_full[i], 1);
        pq::mbar_init(&bars->xp_empty[i], 4);
      }
      for (int i = 0; i < C::SLOTS; ++i) {
        pq::mbar_init(&bars->s8_full[i], 4);
        pq::mbar_init(&bars->s8_empty[i], 1);
        pq::mbar_init(&bars->x_full[i], 1);
      }
      pq::mbar_init(&bars->acc_full, 1);
      bars->abort_flag = 0;
      pq::mbar_fence_init();
      pq::fence_proxy_async_smem();
    }
    __syncwarp();
    for (int i = 0; i < first; ++i) {  // the first weight copies do not depend on the previous kernel
      if (leader) {
        pq::mbar_arrive_expect_tx(&bars->w_full[i], C::W_STAGE);
        pq::tma_load_2d(stage_buf + i * C::W_STAGE, &tmap_w, (kb0 + i) * C::ROWB, n0, &bars->w_full[i]);
      }
      __syncwarp();
    }
  } else if (warp == 1) {
    // Ahead of the wait for the previous kernel: every kernel of the library that allocates tensor memory takes so much
    // shared memory that two of them share an SM only where both find their columns, so nothing waits here for long.
    pq::tmem_alloc(&bars->tmem_base, C::TMEM_COLS);
    pq::tmem_relinquish();
  }
  pq::tc_fence_before();
  __syncthreads();
  pq::tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  int loads_issued = 0;  // producer warps: copies started
  bool ok = true;
  // The steps and code sums of this lane's channels in the reduction are static, like the weights: they are requested here, not behind
  // the cluster barrier, where their trip to memory would stand in the chain.
  float sw[4];
  int zw[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int n = n0 + 4 * lane + i;
    sw[i] = n < p.N ? __ldg(p.s_w + n) : 0.0f;
    zw[i] = ZP && n < p.N ? __ldg(p.wsum + n) : 0;
  }
  float s_a = 1.0f;  // behind the wait for the previous kernel: the token step and the zero point
  int zp8 = 0;
  auto load_steps = [&]() {
    if (!p.s_row) s_a = pq::ld_dep(p.s_a);
    if (ZP) zp8 = pq::ld_dep(p.zp) - 8;
  };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    asm volatile("griddepcontrol.wait;" ::: "memory");  // room comes back once the tokens are there: the bounded waits start behind them
    load_steps();
    int it = first;
    for (; it < total; ++it) {
      const int s = it % C::STAGES;
      if (!wait_bar_warp(&bars->w_empty[s], ((it / C::STAGES) & 1) ^ 1, abort_flag, p.wait_clocks)) {
        ok = false;
        break;
      }
      if (leader) {
        pq::mbar_arrive_expect_tx(&bars->w_full[s], C::W_STAGE);
        pq::tma_load_2d(stage_buf + s * C::W_STAGE, &tmap_w, (kb0 + it) * C::ROWB, n0, &bars->w_full[s]);
      }
      __syncwarp();
    }
    loads_issued = it;
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    asm volatile("griddepcontrol.wait;" ::: "memory");  // what it waits for needs the tokens
    load_steps();
    constexpr uint32_t idesc = pq::umma_idesc_s8(CH, NT);
    const uint64_t desc0 = pq::umma_desc_sw128(pq::smem_u32(slot_buf));
    auto there = [&](int i) {
      const int s = i % C::SLOTS, ph = (i / C::SLOTS) & 1;
      return mbar_test(&bars->s8_full[s], ph) && (!A8 || mbar_test(&bars->x_full[s], ph));
    };
    auto wait_for = [&](int i) {
      const int s = i % C::SLOTS, ph = (i / C::SLOTS) & 1;
      return wait_bar_warp(&bars->s8_full[s], ph, abort_flag, p.wait_clocks) &&
             (!A8 || wait_bar_warp(&bars->x_full[s], ph, abort_flag, p.wait_clocks));
    };
    auto issue = [&](int i) {
      pq::tc_fence_after();
      if (leader) {
        const int s = i % C::SLOTS;
        const uint64_t b_desc = desc0 + s * (C::SLOT >> 4);
        const uint32_t a_tmem = tmem_base + C::A_COL0 + s * C::A_COLS;
#pragma unroll
        for (int kk = 0; kk < C::KB / 32; ++kk)
          mma_i8_ts(tmem_base, a_tmem + kk * 8, b_desc + (kk >> 2) * (C::SUB_SLOT >> 4) + (kk & 3) * 2, idesc, (i | kk) != 0 ? 1u : 0u);
        pq::mma_commit(&bars->s8_empty[s]);
      }
      __syncwarp();
    };
    for (int it = 0; it < total; it += 2) {  // two K blocks per turn: one vote and one branch for both waits
      const bool second = it + 1 < total;
      const bool r0 = there(it), r1 = second && there(it + 1);
      const bool both = __all_sync(0xffffffffu, r0 && r1);
      if (!both && !wait_for(it)) {
        ok = false;
        break;
      }
      issue(it);
      if (!second) break;
      if (!both && !wait_for(it + 1)) {
        ok = false;
        break;
      }
      issue(it + 1);
    }
    if (leader) pq::mma_commit(&bars->acc_full);
    __syncwarp();
    pq::mbar_wait(&bars->acc_full, 0);  // in every case: tensor memory is released behind the MMAs issued
  } else if (warp == 2) {
    // ------------------------------------------------------------------ TMA producer, tokens (A8: into the operand slots)
    constexpr int RING = A8 ? C::SLOTS : C::X_STAGES, BYTES = A8 ? C::SLOT : C::X_STAGE;
    uint64_t* full = A8 ? bars->x_full : bars->xp_full;
    uint64_t* empty = A8 ? bars->s8_empty : bars->xp_empty;
    uint8_t* buf = A8 ? slot_buf : x_buf;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the tokens may come from the previous kernel
    load_steps();
    int it = 0;
    for (; it < total; ++it) {
      const int s = it % RING;
      if (!wait_bar_warp(&empty[s], ((it / RING) & 1) ^ 1, abort_flag, p.wait_clocks)) {
        ok = false;
        break;
      }
      if (leader) {
        pq::mbar_arrive_expect_tx(&full[s], BYTES);
#pragma unroll
        for (int h = 0; h < C::SUBS; ++h)  // 128 elements of every token row per box
          pq::tma_load_2d(buf + s * BYTES + h * (BYTES / C::SUBS), &tmap_x, (kb0 + it) * (A8 ? C::KB : C::ROWB) + h * (A8 ? BK : PK_ROW), t0, &full[s]);
      }
      __syncwarp();
    }
    loads_issued = it;
  } else if (warp >= EXPAND_WARP0) {
    // ------------------------------------------------------------------ expansion
    const int group = (warp - EXPAND_WARP0) >> 2, q = warp & 3;
    const int gt = q * 32 + lane;  // thread of the group = channel row of the tile = lane of tensor memory
    uint4 w[4];
    auto load_w = [&](int ps, int h) {  // 128 elements of this thread's row; swizzled landing buffer: the row-per-thread reads hit distinct banks
      const uint8_t* src = stage_buf + ps * C::W_STAGE + gt * C::ROWB;
      const int sw = C::ROWB == 64 ? (gt >> 1) & 3 : gt & 7;
#pragma unroll
      for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const uint4*>(src + (((4 * h + j) ^ sw) << 4));
    };
    auto put_w = [&](int ss, int h) {
      uint32_t a[32];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t in[4] = {w[j].x, w[j].y, w[j].z, w[j].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t lo = pq::nib_lo_x16(in[i]), hi = pq::nib_hi_x16(in[i]);
          if (A8) {
            a[8 * j + 2 * i] = __byte_perm(lo, hi, 0x5140), a[8 * j + 2 * i + 1] = __byte_perm(lo, hi, 0x7362);
          } else {
            a[8 * j + i] = lo, a[8 * j + 4 + i] = hi;
          }
        }
      }
      pq::tmem_st_32x32(tmem_base + C::A_COL0 + ss * C::A_COLS + h * A_SLOT_COLS + (static_cast<uint32_t>(q * 32) << 16), a);
    };
    auto rest_w = [&](int ps, int ss) {  // what follows the first 128 elements
#pragma unroll
      for (int h = 1; h < C::SUBS; ++h) load_w(ps, h), put_w(ss, h);
      if (C::EARLY_W) {  // behind the store above, for which what was read has arrived in registers
        __syncwarp();
        if (lane == 0) pq::mbar_arrive(&bars->w_empty[ps]);
      }
    };
    // The weights of the first operand slots, ahead of the tokens (and of the wait for the kernel that writes those).
    for (int it = group; it < C::SLOTS && it < total; it += C::GROUPS) {
      if (!wait_bar_warp(&bars->w_full[it], 0, abort_flag, p.wait_clocks)) {
        ok = false;
        break;
      }
      load_w(it, 0);
      put_w(it, 0);
      rest_w(it, it);
    }
    // Tokens, and refilled stages and slots (SLOTS <= STAGES), come behind the previous kernel only: the bounded waits start there.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    load_steps();
    // Of a K block's three waits and three arrivals, those that come together are one instruction, a lane each: lane 0 has the landing ring
    // of the weights, lane 1 that of the tokens, lane 2 the operand slots.
    const int role = lane == 1 && !A8 ? 1 : (lane == 2 ? 2 : 0);
    uint64_t* const r_full = role == 1 ? bars->xp_full : bars->w_full;
    uint64_t* const r_arrive = role == 1 ? bars->xp_empty : (role == 2 ? bars->s8_full : bars->w_empty);
    const int r_len = role == 1 ? C::X_STAGES : (role == 2 ? C::SLOTS : C::STAGES);
    const bool arrives = lane == 2 || (lane == 0 && !C::EARLY_W) || (lane == 1 && !A8);
    int r_pos = group, r_ph = 0, w_ph = 0;  // group < every ring's length
    int ps = group, xs = group, x_ph = 0, ss = group, s_ph = 1;
    for (int it = group; ok && it < total; it += C::GROUPS) {
      const bool first_slots = it < C::SLOTS;  // the weights are expanded already
      {
        const int pos = role == 1 ? r_pos : ps, ph = role == 1 ? r_ph : w_ph;
        const bool skip = role == 1 ? !C::TOGETHER : first_slots;
        // A landing ring that is no multiple of the groups is served by all of them in turn, and a group has not seen every round of a stage. The
        // operand slot is asked for first there: once it is free, K block it - SLOTS and all before it have landed, so that the parity
        // below cannot be that of two rounds back (SLOTS <= STAGES, X_STAGES).
        const bool r0 = !C::SLOT_FIRST || first_slots || mbar_test(&bars->s8_empty[ss], s_ph);
        const bool r1 = skip || mbar_test(r_full + pos, ph);
        if (!__all_sync(0xffffffffu, r0 && r1)) {
          if ((C::SLOT_FIRST && !first_slots && !wait_bar_warp(&bars->s8_empty[ss], s_ph, abort_flag, p.wait_clocks)) ||
              !__all_sync(0xffffffffu, skip || wait_bar(r_full + pos, ph, abort_flag, p.wait_clocks))) {
            ok = false;
            break;
          }
        }
        __syncwarp();  // what one lane waited for is there for all
      }
      if (!first_slots) {
        load_w(ps, 0);
        if (!C::SLOT_FIRST && !__all_sync(0xffffffffu, mbar_test(&bars->s8_empty[ss], s_ph)) &&
            !wait_bar_warp(&bars->s8_empty[ss], s_ph, abort_flag, p.wait_clocks)) {
          ok = false;
          break;
        }
        put_w(ss, 0);
        rest_w(ps, ss);
      }
      if (!A8 && !C::TOGETHER && !wait_bar_warp(&bars->xp_full[xs], x_ph, abort_flag, p.wait_clocks)) {
        ok = false;
        break;
      }
      if (!A8) {
        const uint8_t* xsrc = x_buf + xs * C::X_STAGE;
        uint8_t* dst = slot_buf + ss * C::SLOT;
        constexpr int UNITS = NT * 4, PER_THREAD = (UNITS + 127) / 128;       // per 128 elements; one unit = one 16-byte packed chunk of a token row
        constexpr int BATCH = PER_THREAD <= 4 ? PER_THREAD : PER_THREAD / 2;  // chunks read together
        static_assert(PER_THREAD % BATCH == 0, "whole batches");
#pragma unroll
        for (int h = 0; h < C::SUBS; ++h) {
#pragma unroll
          for (int i0 = 0; i0 < PER_THREAD; i0 += BATCH) {
            uint4 x[BATCH];
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
              const int unit = (i0 + i) * 128 + gt;
              if (UNITS % 128 == 0 || unit < UNITS) x[i] = *reinterpret_cast<const uint4*>(xsrc + h * (NT * PK_ROW) + unit * 16);
            }
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
              const int unit = (i0 + i) * 128 + gt;
              if (UNITS % 128 != 0 && unit >= UNITS) break;
              const int row = unit >> 2, j = unit & 3, sw = row & 7;
              uint8_t* drow = dst + h * C::SUB_SLOT + row * BK;
              *reinterpret_cast<uint4*>(drow + (((2 * j) ^ sw) << 4)) =
                  make_uint4(pq::nib_lo_x16(x[i].x), pq::nib_lo_x16(x[i].y), pq::nib_lo_x16(x[i].z), pq::nib_lo_x16(x[i].w));
              *reinterpret_cast<uint4*>(drow + (((2 * j + 1) ^ sw) << 4)) =
                  make_uint4(pq::nib_hi_x16(x[i].x), pq::nib_hi_x16(x[i].y), pq::nib_hi_x16(x[i].z), pq::nib_hi_x16(x[i].w));
            }
          }
        }
        pq::fence_proxy_async_smem();  // generic-proxy writes -> visible to the tensor core
      }
      pq::tmem_st_wait();
      pq::tc_fence_before();
      __syncwarp();
      if (arrives) pq::mbar_arrive(r_arrive + (role == 0 ? ps : r_pos));
      r_pos += C::GROUPS;
      if (r_pos >= r_len) r_pos -= r_len, r_ph ^= 1;
      ps += C::GROUPS;
      if (ps >= C::STAGES) ps -= C::STAGES, w_ph ^= 1;
      xs += C::GROUPS;
      if (xs >= C::X_STAGES) xs -= C::X_STAGES, x_ph ^= 1;
      ss += C::GROUPS;
      if (ss >= C::SLOTS) ss -= C::SLOTS, s_ph ^= 1;
    }
    // ------------------------------------------------------------------ accumulator -> the partial tile [token][channel]
    ok = ok && wait_bar_warp(&bars->acc_full, 0, abort_flag, p.wait_clocks);
    if (ok) {
      constexpr int SHIFT = A8 ? 4 : 8;  // the factors 16 the expanded codes carry
      int* part = reinterpret_cast<int*>(smem);
      pq::tc_fence_after();
      for (int c = group; c < NT / 16; c += C::GROUPS) {
        uint32_t r[16];
        tmem_ld_32x16(tmem_base + c * 16 + (static_cast<uint32_t>(q * 32) << 16), r);
        pq::tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) part[(c * 16 + i) * CH + gt] = static_cast<int>(r[i]) >> SHIFT;
      }
      pq::tc_fence_before();
    }
  } else {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    load_steps();
  }
  if (!ok && lane == 0) {
    bars->abort_flag = 1;
    pq::report(p.status, PQ_ERR_TIMEOUT);
  }
  __syncthreads();
  if (bars->abort_flag) {  // copies that nobody consumed must have landed before the CTA goes on (they only wait for memory)
    if (warp == 0)
      for (int j = loads_issued > C::STAGES ? loads_issued - C::STAGES : 0; j < loads_issued; ++j)
        pq::mbar_wait(&bars->w_full[j % C::STAGES], (j / C::STAGES) & 1);
    if (warp == 2) {
      constexpr int RING = A8 ? C::SLOTS : C::X_STAGES;
      for (int j = loads_issued > RING ? loads_issued - RING : 0; j < loads_issued; ++j)
        pq::mbar_wait(A8 ? &bars->x_full[j % RING] : &bars->xp_full[j % RING], (j / RING) & 1);
    }
    __syncthreads();
  }
  if (p.splits > 1) cluster_sync_all();  // every CTA's partial tile is in place (28672 x 4096, one split: 0.5 us)
  if (p.early == AT_REDUCTION) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (warp == 1) {
    pq::tc_fence_after();
    pq::tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
  const int tokens = p.M - t0 < NT ? p.M - t0 : NT;
#pragma unroll
  for (int i = 0; i < 4; ++i) sw[i] *= s_a, zw[i] *= zp8;
  if (p.splits == 1) reduce_tile<1, 4, ZP>(p, smem, t0, n0, tokens, warp, C::THREADS / 32, lane, sw, zw);
  else if (p.splits <= 4) reduce_tile<4, 2, ZP>(p, smem, t0, n0, tokens, rank + p.splits * warp, p.splits * (C::THREADS / 32), lane, sw, zw);
  else reduce_tile<MAX_SPLIT, 1, ZP>(p, smem, t0, n0, tokens, rank + p.splits * warp, p.splits * (C::THREADS / 32), lane, sw, zw);
  // no CTA leaves while a peer may still read its partial tile; relaxed: the reads are done, and the output stores need not
  // have reached memory
  if (p.splits > 1) {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  }
}

template <int NT, bool A8, bool ZP, bool WHOLE>
pq_status launch_split(pq_ctx* ctx, const CUtensorMap& tx, const CUtensorMap& tw, SplitParams& p, cudaStream_t st) {
  using C = Cfg<NT, A8, WHOLE>;
  constexpr size_t smem = split_smem<NT, A8, WHOLE>();
  static_assert(WHOLE || smem <= SPLIT_ALONE_SMEM, "half of an SM at most");
  static bool attr_set[64] = {};  // the attribute belongs to the device's copy of the kernel: once per device
  if (ctx->device < 0 || ctx->device >= 64) return PQ_ERR_UNSUPPORTED;
  if (!attr_set[ctx->device]) {
    if (cudaFuncSetAttribute(gemm_w4_split_kernel<NT, A8, ZP, WHOLE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(WHOLE ? smem : SPLIT_ALONE_SMEM)) != cudaSuccess)
      return PQ_ERR_CUDA;
    attr_set[ctx->device] = true;
  }
  p.t_tiles = (p.M + NT - 1) / NT;
  p.n_kb = (p.K + C::KB - 1) / C::KB;
  const int tiles = p.t_tiles * ((p.N + CH - 1) / CH);
  p.splits = WHOLE ? split_count(tiles, p.K, ctx->sm_count, 1) : split_count_pairs(tiles, p.K, ctx->sm_count, p.M, A8);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(tiles) * p.splits);
  cfg.blockDim = dim3(C::THREADS);
  cfg.dynamicSmemBytes = !WHOLE && split_alone(p.M, tiles * p.splits, p.splits, ctx->sm_count) ? SPLIT_ALONE_SMEM : smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.splits;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, gemm_w4_split_kernel<NT, A8, ZP, WHOLE>, tx, tw, p) != cudaSuccess) return PQ_ERR_CUDA;
  return pq_launch_status();
}

template <bool A8, bool ZP>
pq_status launch_tokens(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, SplitParams& p, int64_t K, cudaStream_t st) {
  const bool whole = p.M > 128;
  const int nt = whole ? split_width_whole(p.M, p.N, p.K, A8, ctx->sm_count) : split_width(p.M), kb = split_kb(nt, A8, whole);
  CUtensorMap tx, tw;
  if (!(A8 ? make_s8_map(ctx, &tx, xq, p.M, K, nt) : make_packed_map(ctx, &tx, xq, p.M, K / 2, nt)) ||
      !make_packed_map(ctx, &tw, wq, p.N, K / 2, CH, kb == BK ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, kb / 2))
    return PQ_ERR_CUDA;
  if (whole) {
    switch (nt) {
      case 64: return launch_split<64, A8, ZP, true>(ctx, tx, tw, p, st);
      case 128: return launch_split<128, A8, ZP, true>(ctx, tx, tw, p, st);
      case 192: return launch_split<192, A8, ZP, true>(ctx, tx, tw, p, st);
      default: return launch_split<256, A8, ZP, true>(ctx, tx, tw, p, st);
    }
  }
  switch (nt) {
    case 16: return launch_split<16, A8, ZP, false>(ctx, tx, tw, p, st);
    case 32: return launch_split<32, A8, ZP, false>(ctx, tx, tw, p, st);
    case 48: return launch_split<48, A8, ZP, false>(ctx, tx, tw, p, st);
    case 64: return launch_split<64, A8, ZP, false>(ctx, tx, tw, p, st);
    case 96: return launch_split<96, A8, ZP, false>(ctx, tx, tw, p, st);
    default: return launch_split<128, A8, ZP, false>(ctx, tx, tw, p, st);
  }
}

}  // namespace

// Rows [0, M) of xq/out (the caller has already applied row_begin). s_row: per-token steps (then s_a is ignored), or
// null. zp, wsum: the zero point of Eq. 1 and the weight code sums, or null.
pq_status pq_gemm_split_launch(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, const float* s_a, const float* s_w, void* out,
                               int64_t ldo, int64_t M, int64_t N, int64_t K, int32_t* acc_dbg, cudaStream_t st, bool a8,
                               const float* s_row, const int32_t* zp, const int32_t* wsum) {
  if (zp && !wsum) return PQ_ERR_INVALID_ARG;
  SplitParams p;
  p.zp = zp;
  p.wsum = wsum;
  p.s_row = s_row;
  p.s_a = s_a;
  p.s_w = s_w;
  p.out = static_cast<__nv_bfloat16*>(out);
  p.acc_dbg = acc_dbg;
  p.status = ctx->d_status;
  p.ldo = ldo;
  p.M = static_cast<int>(M);
  p.N = static_cast<int>(N);
  p.K = static_cast<int>(K);
  p.early = M <= 32 ? AT_ENTRY : NEVER;
  if (M > 32 && M <= (s_row ? 128 : 96)) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &capture) != cudaSuccess) cudaGetLastError();  // (the launch says what is wrong with the stream)
    if (capture == cudaStreamCaptureStatusActive) p.early = AT_REDUCTION;
  }
  p.vec_out = ldo % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 7) == 0;
  p.wait_clocks = ctx->wait_clocks;
  if (a8) return launch_tokens<true, false>(ctx, xq, wq, p, K, st);
  return zp ? launch_tokens<false, true>(ctx, xq, wq, p, K, st) : launch_tokens<false, false>(ctx, xq, wq, p, K, st);
}

// W4A4 / W4A8 GEMM for prefill-shaped problems: CTA pairs on the 5th-generation tensor cores, weights fed from tensor memory.
//
//   acc[t,n] = sum_k xq[t,k] * wq[n,k]   (exact int32),   out = bf16(acc * s_a * s_w[n])
//
// sm_100a has no 4-bit integer MMA, so packed nibbles are expanded to 16*code as s8 on the way to the MMA. Two CTAs of a cluster
// share a tile of 256 output channels x up to 256 tokens (cta_group::2). The channels are the MMA's row side: each CTA expands its
// own 128 weight rows in registers (one thread per row, 64-byte-swizzled landing buffer) and writes them to its lanes of tensor
// memory; the tokens are the column side: each CTA expands half of them into the 128-byte-swizzled shared-memory operand, and the
// tensor cores of the pair exchange the halves.
//
// The width of a tile is a multiple of 32 tokens, chosen per launch (tile_rule in pq_gemm_plan.cuh): a token tile costs what its tokens cost, and a
// launch fills whole rounds of the chip's CTA pairs. A tile is accumulated in two halves of at most 128 columns, each with an MMA
// issuer, epilogue warps and one or two slots of tensor memory of its own; the rest of it is six to eight A slots of
// 32 columns (128 K bytes per lane). The half that is ahead is read out while the other still runs.
//
// What bounds it: on one round of 256-token tiles the MMAs (four of 64 clocks per half and K block, 512 clocks; 578 measured), on narrow
// tiles the issue and the expansion (450-500 clocks); on many rounds the chip's power limit. Found on the way (clock stamps of each
// role, then variants; one round of 256-token tiles, K = 4096, weights from HBM, us):
//   - the former kernels waited for their copies: four landing stages came back (latency, expansion, two barrier hops: 1750 clocks,
//     2350 from HBM) later than four K blocks of MMAs take. Six to eight stages: 24.6 -> 19.5; K = 16384 55 -> 45;
//   - then the issuer: a wait that succeeds at once, four MMAs, a commit and the loop took 500 clocks whatever the width. Two K blocks
//     per turn (one vote for both waits): 128-token tiles 19.3 -> 16.3; an issuer per half costs the same and needs no ordering of the
//     halves. mbarrier.try_wait may suspend the warp although another K block could be issued: polls use test_wait;
//   - then the epilogue: a warp per lane quarter took 2.6 us at the end of a launch and 0.7-1.7 us between tiles. Eight warps, integers
//     made floats by two additions instead of the conversion unit, fragments transposed by stmatrix: 18.7 -> 18.2, 2044 x 28672 x 4096
//     158 -> 151.
// GEMM alone, us, before -> now: 512 x 9472 x 4096 22.3 -> 17.7, 2048 x 9472 x 4096 55.1 -> 49.7, 512 x 9472 x 14336 49.9 -> 41.3.
//
// Roles inside each CTA (28 warps):
//   warp 0        TMA producer: packed weight rows [128 x 64 B] and packed token rows per 128-wide K block into the landing stages,
//                 all behind the wait for the previous kernel in the stream. First weights requested ahead of it would ask of every
//                 writer of weights what the header asks for small calls only, and the tokens of the first K block would queue behind
//                 them (us, ahead of the wait / behind it: 8B block at 515 tokens 173.2 / 169.5, 300 x 6144 x 4096 with the rotation 17.8 / 16.2,
//                 515 x 8192 x 28672 125.3 / 120.9, 2044 x 28672 x 4096 153.3 / 152.5).
//   warps 1, 3    (leader CTA only) MMA issuers of the two halves; warp 1 of each CTA owns its TMEM allocation.
//   warp 2        A8: producer of the s8 token boxes, straight into operand slots (128-byte-swizzled).
//   warps 4..7    epilogue of the first half, 24..27 of the second: one warp per TMEM lane quarter (32 channels), 32 tokens at a time:
//                 fragments of 16 lanes x 256 bit, shift, scale, bf16, transposed into token rows by stmatrix, TMA store of
//                 [32 tokens x 64 B].
//   warps 8..23   expansion, four groups of four warps (one per TMEM lane quarter), group g serving K blocks g, g + 4, ...
//                 A 16-byte packed chunk (32 codes) becomes 32 s8 bytes: even-position codes, then odd-position
//                 codes, the same order in both operands, so the dot product is unchanged (natural order with A8).
//
// Every mbarrier wait is bounded; when one runs out the CTA raises an abort flag, every role of
// the CTA drains, the peer's waits run out in turn, and PQ_ERR_TIMEOUT is reported.
#include "pq_gemm_pair.cuh"

namespace {

using namespace pq_pair;
using namespace pq_plan;

constexpr int GROUP_THREADS = 128;
constexpr int EPI_WARP0 = 4, EXPAND_WARP0 = 8, EPI_WARP1 = EXPAND_WARP0 + 4 * N_GROUPS;
constexpr int N_THREADS = (EPI_WARP1 + 4) * 32;
constexpr int ST_BOX = UNIT * 64;           // one store: 32 tokens x 32 channels of bf16
constexpr int ST_BUFS = 2;                  // staging buffers of an epilogue warp

struct __align__(8) Barriers {
  uint64_t land_full[MAX_LAND], land_empty[MAX_LAND];
  uint64_t s8_full[MAX_A];    // waited on in the leader CTA only: the four warps of a group of each CTA
  uint64_t s8_empty[MAX_A];   // both issuers' multicast tcgen05.commit
  uint64_t x_full[MAX_B], x_empty[MAX_B];  // A8 only: token boxes in the operand slots
  uint64_t acc_full[MAX_ACC];   // multicast tcgen05.commit
  uint64_t acc_empty[MAX_ACC];  // leader CTA only: 4 epilogue warps of each CTA
  uint64_t drain;
  uint32_t tmem_base;
  volatile int abort_flag;
};

constexpr size_t PAIR_SMEM = 1024 /*alignment slack*/ + RING_BYTES + 8 * ST_BUFS * ST_BOX + sizeof(Barriers);
static_assert(PAIR_SMEM <= 227 * 1024, "shared memory budget");

struct PairParams : PairPlan {
  const int32_t* zp;    // ZP: the activation zero point z (device scalar) ...
  const int32_t* wsum;  // ... and the sum of every output channel's weight codes [N]
  const float* s_row;   // ROWS: per-token steps [M]; else the scalar s_a applies
  const float* s_a;
  const float* s_w;
  __nv_bfloat16* out;
  int32_t* acc_dbg;
  int32_t* status;
  int64_t ldo;
  int M, N, n_kb;
  int tma_store;           // out can be written with TMA stores (tma_store_fits)
  long long wait_clocks;   // bound of every device-side wait, in SM clocks
};

// D[tmem of both CTAs] (+)= A[tmem of both CTAs] * B[smem halves of both CTAs], issued by one thread of the leader CTA.
__device__ __forceinline__ void mma2_i8_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                           uint32_t accumulate) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::i8 [%0], [%1], %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 16 lanes x 32 columns as 8 x 8 fragments: register 4j + 2h + e holds lane i/4 + 8h, column 8j + 2(i%4) + e (thread i of the warp).
__device__ __forceinline__ void tmem_ld_16x32(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// Four 8 x 8 matrices of 16-bit elements, each stored transposed: thread i gives the address of stored row i % 8 of matrix i / 8.
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
               : "memory");
}

template <bool A8, bool ZP, bool ROWS, bool SMALL>
__global__ void __launch_bounds__(N_THREADS, 1)
    gemm_w4a4_pair_ts_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
                             const __grid_constant__ CUtensorMap tmap_out, const PairParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* b_buf = smem;                          // n_b token operands, 1024-aligned
  uint8_t* land_buf = b_buf + p.n_b * p.slot;     // n_land stages: packed weight rows, then packed token rows
  uint8_t* st_buf = smem + RING_BYTES;            // 8 warps x ST_BUFS buffers
  Barriers* bars = reinterpret_cast<Barriers*>(st_buf + 8 * ST_BUFS * ST_BOX);
  volatile int* abort_flag = &bars->abort_flag;

  const int warp = pq::warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = __shfl_sync(0xffffffffu, cluster_ctarank(), 0);
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int n_tiles = p.c_tiles * p.t_tiles;
  const int my_tiles = pair < n_tiles ? (n_tiles - pair + n_pairs - 1) / n_pairs : 0;
  const uint32_t total = static_cast<uint32_t>(my_tiles) * p.n_kb;  // K blocks of this pair

  if (threadIdx.x == 0) {
    for (int i = 0; i < MAX_LAND; ++i) {
      pq::mbar_init(&bars->land_full[i], 1);
      pq::mbar_init(&bars->land_empty[i], 4);
    }
    for (int i = 0; i < MAX_A; ++i) {
      pq::mbar_init(&bars->s8_full[i], 8);
      pq::mbar_init(&bars->s8_empty[i], 2);
    }
    for (int i = 0; i < MAX_B; ++i) {
      pq::mbar_init(&bars->x_full[i], 1);
      pq::mbar_init(&bars->x_empty[i], 2);
    }
    for (int i = 0; i < MAX_ACC; ++i) {
      pq::mbar_init(&bars->acc_full[i], 1);
      pq::mbar_init(&bars->acc_empty[i], 8);
    }
    pq::mbar_init(&bars->drain, 2);
    bars->abort_flag = 0;
    pq::mbar_fence_init();
    pq::fence_proxy_async_smem();
    pq::tma_prefetch_desc(&tmap_x);
    pq::tma_prefetch_desc(&tmap_w);
    pq::tma_prefetch_desc(&tmap_out);
  }
  if (warp == 1) {
    tmem_alloc2(&bars->tmem_base, PAIR_TMEM_COLS);
    tmem_relinquish2();
  }
  pq::tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the peer's barriers exist before anything arrives on them
  pq::tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  const uint32_t a_ring = tmem_base + p.n_acc * p.acc_cols;  // A slots behind the accumulator halves
  uint32_t loads_issued = 0;  // producer warps: stages whose copies were started
  bool ok = true;

  // no early launch of the next kernel: its CTAs would crowd on the SMs whose pair has no tile left (see pq_launch_pdl)
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    const bool leader = pq::elect_one();
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the operands may come from the previous kernel
    uint32_t it = 0;
    Pos ls;
    for (int tile = pair; tile < n_tiles && ok; tile += n_pairs) {
      const Tile t = tile_at(p, tile);
      for (int kb = 0; kb < p.n_kb; ++kb, ++it, ls.advance(1, p.n_land)) {
        if (!wait_bar_warp(&bars->land_empty[ls.i], ls.ph ^ 1, abort_flag, p.wait_clocks)) {
          ok = false;
          break;
        }
        if (leader) {
          const int boxes = A8 ? 0 : (t.u1 > 0 ? 2 : 1);
          uint8_t* dst = land_buf + ls.i * p.stage;
          pq::mbar_arrive_expect_tx(&bars->land_full[ls.i], W_STAGE + boxes * p.box * PK_ROW);
          pq::tma_load_2d(dst, &tmap_w, kb * PK_ROW, t.n0 + rank * CH_CTA, &bars->land_full[ls.i]);
          if (boxes > 0) pq::tma_load_2d(dst + W_STAGE, &tmap_x, kb * PK_ROW, t.t0 + rank * t.u0 * (UNIT / 2), &bars->land_full[ls.i]);
          if (boxes > 1)
            pq::tma_load_2d(dst + W_STAGE + p.box * PK_ROW, &tmap_x, kb * PK_ROW, t.t0 + t.u0 * UNIT + rank * t.u1 * (UNIT / 2), &bars->land_full[ls.i]);
        }
        __syncwarp();
      }
    }
    loads_issued = it;
  } else if (A8 && warp == 2) {
    // ------------------------------------------------------------------ token producer (A8)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const bool leader = pq::elect_one();
    uint32_t it = 0;
    Pos xs;
    for (int tile = pair; tile < n_tiles && ok; tile += n_pairs) {
      const Tile t = tile_at(p, tile);
      for (int kb = 0; kb < p.n_kb; ++kb, ++it, xs.advance(1, p.n_b)) {
        if (!wait_bar_warp(&bars->x_empty[xs.i], xs.ph ^ 1, abort_flag, p.wait_clocks)) {
          ok = false;
          break;
        }
        if (leader) {
          uint8_t* dst = b_buf + xs.i * p.slot;
          pq::mbar_arrive_expect_tx(&bars->x_full[xs.i], (t.u1 > 0 ? 2 : 1) * p.box * BK);
          pq::tma_load_2d(dst, &tmap_x, kb * BK, t.t0 + rank * t.u0 * (UNIT / 2), &bars->x_full[xs.i]);
          if (t.u1 > 0)
            pq::tma_load_2d(dst + p.box * BK, &tmap_x, kb * BK, t.t0 + t.u0 * UNIT + rank * t.u1 * (UNIT / 2), &bars->x_full[xs.i]);
        }
        __syncwarp();
      }
    }
    loads_issued = it;
  } else if (warp == 1 || warp == 3) {
    // ------------------------------------------------------------------ MMA issuers (leader CTA): one per accumulator half
    if (rank == 0) {
      asm volatile("griddepcontrol.wait;" ::: "memory");  // what they wait for needs the tokens
      const bool leader = pq::elect_one();
      const int h = warp >> 1;
      const uint64_t desc0 = pq::umma_desc_sw128(pq::smem_u32(b_buf) + h * p.box * BK);
      const uint32_t slot_desc = p.slot >> 4;
      Pos as, bs;  // operand slots (8-bit tokens: of their own)
      AccRing u;
      for (int tile = pair; tile < n_tiles && ok; tile += n_pairs) {
        const Tile t = tile_at(p, tile);
        const int units = h ? t.u1 : t.u0;  // none: only the slots are handed on
        const Pos mine = u.slot(h, p);
        const uint32_t d_tmem = tmem_base + mine.i * p.acc_cols, idesc = pq::umma_idesc_s8(2 * CH_CTA, units * UNIT);
        if (units > 0 && !wait_bar_warp(&bars->acc_empty[mine.i], mine.ph ^ 1, abort_flag, p.wait_clocks)) {
          ok = false;
          break;
        }
        pq::tc_fence_after();
        auto k_block = [&](bool first) {  // with the operands in slots as, bs; both CTAs may refill them once both halves' MMAs have read them
          if (leader) {
            if (units > 0) {
              const uint32_t a_tmem = a_ring + as.i * A_SLOT_COLS;
              const uint64_t b_desc = desc0 + bs.i * slot_desc;
              mma2_i8_ts(d_tmem, a_tmem, b_desc, idesc, first ? 0u : 1u);
#pragma unroll
              for (int kk = 1; kk < BK / 32; ++kk) mma2_i8_ts(d_tmem, a_tmem + kk * 8, b_desc + kk * 2, idesc, 1u);  // 32 bytes of K further
            }
            mma2_commit_both(&bars->s8_empty[as.i]);
            if (A8) mma2_commit_both(&bars->x_empty[bs.i]);
          }
          __syncwarp();
          as.advance(1, p.n_a), bs.advance(1, p.n_b);
        };
        int kb = 0;
        for (; kb + 1 < p.n_kb; kb += 2) {  // two K blocks per turn: one vote and one branch for both waits
          Pos next = as;
          next.advance(1, p.n_a);
          const bool r0 = mbar_test(&bars->s8_full[as.i], as.ph), r1 = mbar_test(&bars->s8_full[next.i], next.ph);
          const bool both = __all_sync(0xffffffffu, r0 && r1);
          if (!both && !wait_bar_warp(&bars->s8_full[as.i], as.ph, abort_flag, p.wait_clocks)) {
            ok = false;
            break;
          }
          pq::tc_fence_after();
          k_block(kb == 0);
          if (!both && !wait_bar_warp(&bars->s8_full[as.i], as.ph, abort_flag, p.wait_clocks)) {
            ok = false;
            break;
          }
          pq::tc_fence_after();
          k_block(false);
        }
        if (ok && kb < p.n_kb) {
          ok = wait_bar_warp(&bars->s8_full[as.i], as.ph, abort_flag, p.wait_clocks);
          pq::tc_fence_after();
          if (ok) k_block(kb == 0);
        }
        if (!ok) break;
        if (leader && units > 0) mma2_commit_both(&bars->acc_full[mine.i]);
        __syncwarp();
        u.advance(h, t, p);
      }
      if (leader) mma2_commit_both(&bars->drain);  // whatever was issued has finished before either CTA releases its tensor memory
      __syncwarp();
    }
    pq::mbar_wait(&bars->drain, 0);
  } else if (warp >= EXPAND_WARP0 && warp < EPI_WARP1) {
    // ------------------------------------------------------------------ expansion
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the landing stages' tokens come behind it
    const int group = (warp - EXPAND_WARP0) >> 2, q = warp & 3;
    const int gt = q * 32 + lane;  // thread of the group = channel row of the CTA = lane of tensor memory
    int tile = pair, kb = group;
    Tile t = tile_at(p, tile);
    Pos ls, as, xs;
    ls.advance(group, p.n_land), as.advance(group, p.n_a), xs.advance(group, p.n_b);
    for (uint32_t it = group; it < total;
         it += N_GROUPS, kb += N_GROUPS, ls.advance(N_GROUPS, p.n_land), as.advance(N_GROUPS, p.n_a), xs.advance(N_GROUPS, p.n_b)) {
      if (kb >= p.n_kb) {
        do kb -= p.n_kb, tile += n_pairs;
        while (kb >= p.n_kb);
        t = tile_at(p, tile);
      }
      // The operand slot first: once it is free, the MMAs of K block it - n_a and of all before it have run, so the copies of those K
      // blocks have landed, and with n_land >= n_a (and n_b >= n_a) the parities below cannot be mistaken for those of two rounds back.
      if (!wait_bar_warp(&bars->s8_empty[as.i], as.ph ^ 1, abort_flag, p.wait_clocks) ||
          !wait_bar_warp(&bars->land_full[ls.i], ls.ph, abort_flag, p.wait_clocks)) {
        ok = false;
        break;
      }
      const uint8_t* src = land_buf + ls.i * p.stage;
      const int chunks = (t.u0 + t.u1) * (UNIT / 2) * 4;  // 16-byte chunks of this CTA's token rows (the second box's follow the first's)
      uint4 w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)  // 64-byte swizzle of the landing buffer: the row-per-thread reads hit distinct banks
        w[j] = *reinterpret_cast<const uint4*>(src + gt * PK_ROW + ((j ^ ((gt >> 1) & 3)) << 4));
      uint4 x[4];
      if (!A8) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i * GROUP_THREADS + gt < chunks) x[i] = *reinterpret_cast<const uint4*>(src + W_STAGE + (i * GROUP_THREADS + gt) * 16);
      }
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
      pq::tmem_st_32x32(a_ring + as.i * A_SLOT_COLS + (static_cast<uint32_t>(q * 32) << 16), a);
      if (!A8) {
        const int row = gt >> 2, j = gt & 3, sw = row & 7;  // the thread's rows are 32 apart: one swizzle
        uint8_t* lo = b_buf + as.i * p.slot + row * BK + (((2 * j) ^ sw) << 4);
        uint8_t* hi = b_buf + as.i * p.slot + row * BK + (((2 * j + 1) ^ sw) << 4);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (i * GROUP_THREADS + gt < chunks) {
            *reinterpret_cast<uint4*>(lo + i * 32 * BK) =
                make_uint4(pq::nib_lo_x16(x[i].x), pq::nib_lo_x16(x[i].y), pq::nib_lo_x16(x[i].z), pq::nib_lo_x16(x[i].w));
            *reinterpret_cast<uint4*>(hi + i * 32 * BK) =
                make_uint4(pq::nib_hi_x16(x[i].x), pq::nib_hi_x16(x[i].y), pq::nib_hi_x16(x[i].z), pq::nib_hi_x16(x[i].w));
          }
        }
      }
      if (A8) {  // the slot is complete only with this CTA's token boxes in place
        if (!wait_bar_warp(&bars->x_full[xs.i], xs.ph, abort_flag, p.wait_clocks)) {
          ok = false;
          break;
        }
      }
      pq::tmem_st_wait();     // the TMEM lane is written ...
      pq::tc_fence_before();  // ... and ordered before the arrival below
      if (!A8) pq::fence_proxy_async_smem();  // generic-proxy writes -> visible to the tensor core's async proxy
      __syncwarp();
      if (lane == 0) {
        mbar_arrive_cluster(map_to_cta(&bars->s8_full[as.i], 0));
        pq::mbar_arrive(&bars->land_empty[ls.i]);  // behind the stores, for which what was read has arrived in registers
      }
    }
  } else if (warp >= EPI_WARP0) {
    // ------------------------------------------------------------------ epilogue
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the scales and the output may belong to the previous kernel
    constexpr int SHIFT = A8 ? 4 : 8;  // the factors 16 the expanded codes carry
    const int q = warp & 3;            // TMEM lane quarter this warp may access
    const float s_a = ROWS ? 1.0f : pq::ld_dep(p.s_a);
    const int zp8 = ZP ? pq::ld_dep(p.zp) - 8 : 0;
    const int h = warp >= EPI_WARP1 ? 1 : 0;  // the accumulator half this warp reads
    uint8_t* my_buf = st_buf + (4 * h + q) * ST_BUFS * ST_BOX;
    const uint32_t st_row = pq::smem_u32(my_buf) + (lane & 7) * 64;  // stmatrix: this lane addresses token row lane % 8 of a group of eight ...
    const int st_chunk = lane >> 3;                                  // ... and the 16-byte chunk (eight channels) of matrix lane / 8
    uint32_t n_store = 0;
    AccRing u;
    for (int tile = pair; tile < n_tiles && ok; tile += n_pairs) {
      const Tile t = tile_at(p, tile);
      const int n0 = t.n0 + static_cast<int>(rank) * CH_CTA + q * 32;  // the warp's channels
      float sw[4];
      int zw[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {  // this lane's channels: lane / 4 of each group of eight
        const int n = n0 + i * 8 + (lane >> 2);
        sw[i] = n < p.N ? s_a * __ldg(p.s_w + n) : 0.0f;
        zw[i] = ZP && n < p.N ? zp8 * __ldg(p.wsum + n) : 0;
      }
      const Pos mine = u.slot(h, p);
      u.advance(h, t, p);
      const int units = h ? t.u1 : t.u0, th = t.t0 + (h ? t.u0 * UNIT : 0);
      if (units > 0) {
        if (!wait_bar_warp(&bars->acc_full[mine.i], mine.ph, abort_flag, p.wait_clocks)) {
          ok = false;
          break;
        }
        pq::tc_fence_after();
        const uint32_t taddr = tmem_base + mine.i * p.acc_cols + (static_cast<uint32_t>(q * 32) << 16);
#pragma unroll 1
        for (int c = 0; c < units; ++c) {
          const int t0 = th + c * UNIT;
          [[maybe_unused]] float rs[8];  // the steps of this lane's tokens, requested ahead of the accumulators (behind: 2044 x 28672 x 4096 168 us, now 164)
          if constexpr (ROWS) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int tok = t0 + (i >> 1) * 8 + (lane & 3) * 2 + (i & 1);
              rs[i] = tok < p.M ? pq::ld_dep(p.s_row + tok) : 1.0f;
            }
          }
          uint32_t r[2][16];  // lanes (channels) 0..15 and 16..31 of the quarter
          tmem_ld_16x32(taddr + c * UNIT, r[0]);
          tmem_ld_16x32(taddr + c * UNIT + (16u << 16), r[1]);
          pq::tmem_ld_wait();
          if (c == units - 1) {  // the half is read: its MMA warp may overwrite it
            pq::tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_to_cta(&bars->acc_empty[mine.i], 0));
          }
          auto sum = [&](int g, int j, int e) { return (static_cast<int32_t>(r[g >> 1][4 * j + 2 * (g & 1) + e]) >> SHIFT) - (ZP ? zw[g] : 0); };
          auto val = [&](int g, int j, int e) {
            const int v = sum(g, j, e);
            // SMALL: |v| <= 2^22, so v + 1.5 * 2^23 is exact and its bits are those of the integer sum; the conversion instruction runs
            // at an eighth of the rate of the two additions.
            const float f = (SMALL ? __int_as_float(0x4B400000 + v) - 12582912.0f : static_cast<float>(v)) * sw[g];
            if constexpr (ROWS) return f * rs[2 * j + e];
            else return f;
          };
          const uint32_t buf = (n_store % ST_BUFS) * ST_BOX;
          if (lane == 0) bulk_wait_read<ST_BUFS - 1>();  // the store that last read this buffer is ST_BUFS stores back
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 4; ++j) {  // eight tokens: four matrices of eight channels
            uint32_t v[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              const __nv_bfloat162 b = __floats2bfloat162_rn(val(g, j, 0), val(g, j, 1));
              v[g] = *reinterpret_cast<const uint32_t*>(&b);
            }
            // 64-byte rows under the 64-byte swizzle: chunk XOR (row / 2) % 4
            stmatrix_x4_trans(st_row + buf + j * 512 + ((st_chunk ^ ((lane >> 1) & 3)) << 4), v[0], v[1], v[2], v[3]);
          }
          if (p.acc_dbg) {
            int32_t* d = p.acc_dbg + static_cast<int64_t>(t0 + (lane & 3) * 2) * p.N + n0 + (lane >> 2);
#pragma unroll
            for (int i = 0; i < 8; ++i, d += i & 1 ? p.N : 7 * static_cast<int64_t>(p.N))
#pragma unroll
              for (int g = 0; g < 4; ++g)
                if (t0 + (i >> 1) * 8 + (lane & 3) * 2 + (i & 1) < p.M && n0 + g * 8 + (lane >> 2) < p.N) d[g * 8] = sum(g, i >> 1, i & 1);
          }
          if (p.tma_store) {
            pq::fence_proxy_async_smem();
            __syncwarp();
            if (n0 < p.N) {  // counted only when stored: the wait above is in stores
              if (lane == 0) {
                tma_store_2d(&tmap_out, my_buf + buf, n0, t0);
                bulk_commit();
              }
              ++n_store;
            }
          } else {
            __syncwarp();
            for (int row = 0; row < UNIT && t0 + row < p.M; ++row)
              if (n0 + lane < p.N)
                p.out[static_cast<int64_t>(t0 + row) * p.ldo + n0 + lane] =
                    *reinterpret_cast<const __nv_bfloat16*>(my_buf + buf + row * 64 + (((lane >> 3) ^ ((row >> 1) & 3)) << 4) + (lane & 7) * 2);
            __syncwarp();
          }
        }
      }
    }
    if (lane == 0) bulk_wait_read<0>();  // the staging buffers have been read: the CTA may end
  }

  if (!ok && lane == 0) {
    bars->abort_flag = 1;
    pq::report(p.status, PQ_ERR_TIMEOUT);
  }
  pq::tc_fence_before();
  __syncthreads();
  if (bars->abort_flag) {
    // a role gave up: copies that nobody consumed must still have landed before the CTA may exit (they only wait for memory,
    // hence the generous bound)
    if (warp == 0 && lane == 0)
      for (uint32_t j = loads_issued > static_cast<uint32_t>(p.n_land) ? loads_issued - p.n_land : 0; j < loads_issued; ++j)
        pq::mbar_wait(&bars->land_full[j % p.n_land], (j / p.n_land) & 1);
    if (A8 && warp == 2 && lane == 0)
      for (uint32_t j = loads_issued > static_cast<uint32_t>(p.n_b) ? loads_issued - p.n_b : 0; j < loads_issued; ++j)
        pq::mbar_wait(&bars->x_full[j % p.n_b], (j / p.n_b) & 1);
    __syncthreads();
  }
  cluster_sync_all();  // neither CTA frees tensor memory or exits while the pair may still touch it
  if (warp == 1) {
    pq::tc_fence_after();
    tmem_dealloc2(tmem_base, PAIR_TMEM_COLS);
  }
}

template <bool A8, bool ZP, bool ROWS, bool SMALL>
pq_status launch_pair(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, void* out, int64_t K, PairParams& p, cudaStream_t st) {
  static bool attr_set[64] = {};  // the attribute belongs to the device's copy of the kernel: once per device
  if (ctx->device < 0 || ctx->device >= 64) return PQ_ERR_UNSUPPORTED;
  if (!attr_set[ctx->device]) {
    if (cudaFuncSetAttribute(gemm_w4a4_pair_ts_kernel<A8, ZP, ROWS, SMALL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(PAIR_SMEM)) != cudaSuccess)
      return PQ_ERR_CUDA;
    attr_set[ctx->device] = true;
  }
  if (!pair_plan(p, p.M, p.N, p.n_kb, A8, ctx->sm_count)) return PQ_ERR_UNSUPPORTED;
  CUtensorMap tx, tw, to;
  if (!(A8 ? make_s8_map(ctx, &tx, xq, p.M, K, p.box) : make_packed_map(ctx, &tx, xq, p.M, K / 2, p.box)) ||
      !make_packed_map(ctx, &tw, wq, p.N, K / 2, CH_CTA, CU_TENSOR_MAP_SWIZZLE_64B))
    return PQ_ERR_CUDA;
  p.tma_store = tma_store_fits(out, p.N, p.ldo);
  if (p.tma_store) {
    if (!make_out_map(ctx, &to, out, p.M, p.N, p.ldo, 32)) return PQ_ERR_CUDA;
  } else {
    to = tx;  // never dereferenced
  }
  const int n_tiles = p.c_tiles * p.t_tiles, max_pairs = ctx->sm_count / 2;
  const int pairs = n_tiles < max_pairs ? n_tiles : max_pairs;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(N_THREADS);
  cfg.dynamicSmemBytes = PAIR_SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  // the kernel may be launched while its predecessor drains; it waits for it on the device before it reads or writes anything,
  // which hides the launch itself
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, gemm_w4a4_pair_ts_kernel<A8, ZP, ROWS, SMALL>, tx, tw, to, p) != cudaSuccess) return PQ_ERR_CUDA;
  return pq_launch_status();
}

}  // namespace

// Rows [0, M) of xq/out (the caller has already applied row_begin). a8: xq holds one s8 code per element. s_row: per-token steps
// (then s_a is ignored), or null. zp, wsum: the zero point of Eq. 1 and the weight code sums, or null.
pq_status pq_gemm_pair_ts_launch(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, const float* s_a, const float* s_w,
                                 void* out, int64_t ldo, int64_t M, int64_t N, int64_t K, int32_t* acc_dbg,
                                 cudaStream_t st, bool a8, const float* s_row, const int32_t* zp, const int32_t* wsum) {
  if (zp && (a8 || !wsum || s_row)) return PQ_ERR_INVALID_ARG;
  if (a8 && s_row) return PQ_ERR_INVALID_ARG;
  PairParams p;
  p.s_a = s_a;
  p.s_w = s_w;
  p.s_row = s_row;
  p.zp = zp;
  p.wsum = wsum;
  p.out = static_cast<__nv_bfloat16*>(out);
  p.acc_dbg = acc_dbg;
  p.status = ctx->d_status;
  p.wait_clocks = ctx->wait_clocks;
  p.ldo = ldo;
  p.M = static_cast<int>(M);
  p.N = static_cast<int>(N);
  p.n_kb = static_cast<int>((K + BK - 1) / BK);
  const bool small = K <= 4096;  // 8-bit tokens: |sum| <= 128 * 8 * K <= 2^22; 4-bit tokens: 8 * 8 * K for every K
  if (a8) return small ? launch_pair<true, false, false, true>(ctx, xq, wq, out, K, p, st) : launch_pair<true, false, false, false>(ctx, xq, wq, out, K, p, st);
  if (zp) return launch_pair<false, true, false, false>(ctx, xq, wq, out, K, p, st);
  return s_row ? launch_pair<false, false, true, true>(ctx, xq, wq, out, K, p, st) : launch_pair<false, false, false, true>(ctx, xq, wq, out, K, p, st);
}

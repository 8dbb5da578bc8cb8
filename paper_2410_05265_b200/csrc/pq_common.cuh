// Shared internals of the pq library: context, status plumbing, and thin wrappers over the
// sm_100a PTX this library issues (mbarrier, TMA, tcgen05). Device-side waits are all bounded.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/pq.h"

struct pq_ctx {
  int device;
  int sm_count;
  int32_t* d_status;    // device status word (PQ_OK or the first error a kernel reported)
  uint32_t* d_tickets;  // zero-initialised, self-resetting "last block done" counters
  int n_tickets;
  void* encode_tiled;   // cuTensorMapEncodeTiled resolved through the runtime
  long long wait_clocks;  // bound of every device-side wait, in SM clocks (pq_set_wait_limit)
};

#define PQ_DEFAULT_WAIT_CLOCKS (1ll << 31)  // about a second

#define PQ_N_TICKETS 65536

#define PQ_CUDA_OK(expr)                      \
  do {                                        \
    cudaError_t e__ = (expr);                 \
    if (e__ != cudaSuccess) return PQ_ERR_CUDA; \
  } while (0)

static inline pq_status pq_launch_status() { return cudaGetLastError() == cudaSuccess ? PQ_OK : PQ_ERR_CUDA; }

// Launch under programmatic dependent launch: the kernel may be placed once every CTA of the one before it in the stream has
// let it (pdl_trigger) or has ended, and executes pq::pdl_wait() before it touches anything that kernel may write or still read.
//
// Who lets its successor be placed EARLY is decided by the successor's size. CTAs placed while the predecessor still runs land on
// the SMs that happen to have room, four to an SM, instead of being spread over the chip; that costs more than the hidden
// launch. So the rotation kernels (the GEMM behind them takes whole SMs, or prefetches its weights), the decode kernels and the
// small kernels of small grids trigger early; the CTA-pair GEMMs, the split-K GEMM above 32 tokens (in a captured graph above 96) and the
// kernels of larger grids do not, and their successor starts when they end without a launch gap. Measured on whole passes (us, before the rule,
// when the GEMMs always triggered and the element-wise kernels were launched plainly / with it): 8B linear set at 2044 tokens
// 395 / 376, per-token set at 1000 253 / 243, W4A8 set at 300 137 / 129; 8B block at 515 tokens 243 / 228, at 1500 418 / 398,
// at 128 tokens (graph) 115 / 105; decode layer, one sequence at 4000 tokens, 62.2 / 60.0. With every kernel triggering early
// the 515-token block took 238 us in a graph against 224.
//
// Kernels that write KV-cache rows, lengths or steps (the appends and the one-launch decode step), packed weights or code sums
// never trigger. Some kernels read these ahead of their own wait (the one-launch decode step its first cache rows and lengths,
// the streaming and split-K GEMMs their weights), and several pass an early start on ahead of their wait (the rotation kernels,
// those GEMMs): a writer that triggers could then still be running any number of launches further down the stream. One that
// does not has ended before anything behind it in the stream starts.
#define PQ_PDL_MAX_CTAS 64
template <typename... P, typename... A>
static inline pq_status pq_launch_pdl(void (*kern)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...) != cudaSuccess) return PQ_ERR_CUDA;
  return pq_launch_status();
}

namespace pq {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel be placed, from a small grid (see pq_launch_pdl). Issued behind pdl_wait(): whoever starts early then finds
// everything before this kernel complete. Not in kernels whose output a later kernel may read ahead of its wait.
__device__ __forceinline__ void pdl_trigger() {
  if (gridDim.x * gridDim.y <= PQ_PDL_MAX_CTAS) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Loads of what an earlier kernel in the stream may have written, behind pdl_wait(). Not __ldg, nor a plain load through a const
// __restrict__ pointer: the compiler takes such data for unchanging and may move the load ahead of the wait (the per-token step of the
// streaming GEMM was read there: in a graph the GEMM behind the two-launch dynamic quantizer saw the zeros the step array starts
// from, and its outputs were zero). Volatile assembly keeps its order.
__device__ __forceinline__ uint32_t ld_dep(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float ld_dep(const float* p) { return __uint_as_float(ld_dep(reinterpret_cast<const uint32_t*>(p))); }
__device__ __forceinline__ int32_t ld_dep(const int32_t* p) { return static_cast<int32_t>(ld_dep(reinterpret_cast<const uint32_t*>(p))); }
__device__ __forceinline__ uint2 ld_dep(const uint2* p) {
  uint2 v;
  asm volatile("ld.global.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ uint4 ld_dep(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

__device__ __forceinline__ void report(int32_t* status, int32_t code) { atomicCAS(status, 0, code); }

// SiLU(g) * u = g / (1 + 2^(-g log2 e)) * u in fp32 with the hardware's 2^x and reciprocal (about 2 ulp of fp32, far below the bf16
// rounding that follows). The form for two elements does the same operations on packed pairs: the stand-alone kernel and the one fused
// into the rotation agree bit for bit.
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float silu_mul_f32(float g, float u) {
  return __fmul_rn(__fmul_rn(g, rcp_approx(__fadd_rn(1.0f, ex2_approx(__fmul_rn(g, -1.4426950408889634f))))), u);
}
__device__ __forceinline__ float2 silu_mul_f32(float2 g, float2 u) {
  const float2 t = __fmul2_rn(g, make_float2(-1.4426950408889634f, -1.4426950408889634f));
  const float2 d = __fadd2_rn(make_float2(1.0f, 1.0f), make_float2(ex2_approx(t.x), ex2_approx(t.y)));
  return __fmul2_rn(__fmul2_rn(g, make_float2(rcp_approx(d.x), rcp_approx(d.y))), u);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// ---- mbarrier -----------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait: gives up after `limit` SM clocks and returns false (a single try_wait may itself suspend the
// thread for a short, implementation-defined time, so the bound is checked after every one of them).
__device__ __forceinline__ bool mbar_wait_for(uint64_t* bar, uint32_t parity, long long limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (clock64() - t0 > limit) return false;
  }
}
// The same with the default bound of about a second (used where only memory latency is waited for).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  return mbar_wait_for(bar, parity, PQ_DEFAULT_WAIT_CLOCKS);
}

// One lane of the (converged) warp. A role that issues TMA copies or MMAs keeps its whole warp in the loop and lets the
// elected lane issue: addresses and descriptors are then warp-uniform values and stay in uniform registers, which those
// instructions read; in a branch that one lane takes alone every operand is moved there again for every instruction
// (four MMAs and their commit: 300 clocks, against 70-100 with the loop kept uniform).
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "elect.sync _|p, 0xffffffff;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(pred));
  return pred != 0;
}
// The warp's index as a value the compiler knows to be the same in all lanes.
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0); }

__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---- TMA ----------------------------------------------------------------------------------
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// 2-D tiled load global -> shared, completion counted in bytes on an mbarrier (no multicast).
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* m, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

// ---- tcgen05 ------------------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem], s8 x s8 -> s32, issued by one thread.
__device__ __forceinline__ void mma_i8_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The mbarrier receives one arrival once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp receives lane (base+i).
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// The same wait, with the loaded registers as operands: when other work is placed between a load and its wait, this
// keeps every use of r behind the wait.
__device__ __forceinline__ void tmem_ld_wait_for(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                 "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]),
                 "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),
                 "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}

// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp writes lane (base+i).
__device__ __forceinline__ void tmem_st_32x32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor for a K-major operand stored in the 128-byte-swizzled canonical
// layout: rows of 128 bytes, 8-row groups 1024 bytes apart, 16-byte chunks XOR-ed with (row & 7).
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr >> 4) & 0x3FFF);  // start address
  d |= static_cast<uint64_t>(1) << 16;                    // leading byte offset (unused for swizzled K-major)
  d |= static_cast<uint64_t>(1024 >> 4) << 32;            // stride byte offset between 8-row groups
  d |= static_cast<uint64_t>(1) << 46;                    // descriptor version for sm_100
  d |= static_cast<uint64_t>(2) << 61;                    // SWIZZLE_128B
  return d;
}

// Instruction descriptor of kind::i8: s8 x s8 -> s32, both operands K-major, dense.
__host__ __device__ constexpr uint32_t umma_idesc_s8(int M, int N) {
  return (2u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(M >> 4) << 24);
}

// ---- small numeric helpers ----------------------------------------------------------------
// Packed two's-complement nibbles -> s8 values scaled by 16: the high nibble of a byte already is
// 16*hi as an s8; the low nibble shifted up by four is 16*lo.
__device__ __forceinline__ uint32_t nib_hi_x16(uint32_t w) { return w & 0xF0F0F0F0u; }
__device__ __forceinline__ uint32_t nib_lo_x16(uint32_t w) { return (w << 4) & 0xF0F0F0F0u; }

}  // namespace pq

// Offline RTN weight quantization, one symmetric INT4 scale per output channel
// (Table 1 "per-channel"; Table 6 "RTN"; Eq. 1). One CTA per weight row: rows of up to 32768 weights with 16-byte alignment are
// read once and kept in registers, the others take two passes over the row.
#include "pq_common.cuh"

namespace {

constexpr int QW_THREADS = 256;

__global__ void __launch_bounds__(QW_THREADS) quant_weights_kernel(const __nv_bfloat16* __restrict__ W, int64_t N,
                                                                    int64_t K, int64_t ldw, uint8_t* __restrict__ wq,
                                                                    float* __restrict__ s_w) {
  __shared__ float red[QW_THREADS / 32];
  __shared__ float s_scale;
  for (int64_t n = blockIdx.x; n < N; n += gridDim.x) {
    const __nv_bfloat16* row = W + n * ldw;
    float mx = 0.0f;
    for (int64_t k = threadIdx.x; k < K; k += QW_THREADS) mx = fmaxf(mx, fabsf(__bfloat162float(row[k])));
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
      float m = red[0];
      for (int i = 1; i < QW_THREADS / 32; ++i) m = fmaxf(m, red[i]);
      float s = (m == 0.0f) ? 1.0f : __fdiv_rn(m, 7.0f);
      s_scale = s;
      s_w[n] = s;
    }
    __syncthreads();
    const float s = s_scale;
    uint8_t* orow = wq + n * (K / 2);
    for (int64_t j = threadIdx.x; j < K / 2; j += QW_THREADS) {
      float a = __fdiv_rn(__bfloat162float(row[2 * j]), s);      // IEEE fp32 division
      float b = __fdiv_rn(__bfloat162float(row[2 * j + 1]), s);
      int ca = max(-8, min(7, __float2int_rn(a)));                // round-half-even, clamp
      int cb = max(-8, min(7, __float2int_rn(b)));
      orow[j] = static_cast<uint8_t>((ca & 0xF) | ((cb & 0xF) << 4));
    }
    __syncthreads();
  }
}

// The same for rows that are read once: VPT 16-byte vectors per thread stay in registers between the maximum and the codes.
// Bound by HBM (2.5 bytes per weight) once a code costs few instructions. A code is rint(w / s) with an IEEE division; here it is
// rint(w * r), r ~ 1 / s, from one fused multiply-add into the rounding constant 1.5 * 2^23, checked per row: both are monotone in w
// and can differ only next to a half-integer, which for bf16 weights means at one of the few bf16 values around (k + 1/2) s,
// k = 0 .. 6 (bf16 values are 2^-8 apart, the two quotients less than 2^-21). A lane each compares the two forms there, for r = 1 / s and
// its two neighbours; a row where none agrees (about one maximum in nine: a multiple of 7), that holds an infinity or a NaN, or
// whose step is far from 1 divides element by element.
// Eight codes are packed by multiply-adds (a digit each), and each lane checks one of the 28 values, for all of its four vectors: with
// masks and shifts, and four checked values per lane, instruction issue (82 %) was the bound.
// Measured (us, two passes with a division each / masks, four values a lane / now): 28672 x 4096 129 / 58.7 / 48.9 (6.0 TB/s),
// 4096 x 14336 64 / 31.5 / 29.0, 8192 x 28672 256 / 118 / 106, 4096 x 4096 20.6 / 12.2 / 10.6. Half the threads with twice the
// vectors: 47.7, 32.6 (512 threads), 106, 12.0.
__device__ __forceinline__ int code_div(float w, float s) { return max(-8, min(7, __float2int_rn(__fdiv_rn(w, s)))); }
// code + 8 in the low bits; what stands above them is constant
__device__ __forceinline__ uint32_t code_mul(float w, float r) { return __float_as_uint(fmaf(w, r, 12582920.0f)); }

template <int THREADS, int VPT>
__global__ void __launch_bounds__(THREADS) quant_weights_once_kernel(const __nv_bfloat16* __restrict__ W, int K, int64_t ldw,
                                                                     uint8_t* __restrict__ wq, float* __restrict__ s_w) {
  __shared__ uint32_t red[THREADS / 32];
  const int64_t n = blockIdx.x;
  const uint4* row = reinterpret_cast<const uint4*>(W + n * ldw);
  const int n_vec = K / 8;
  pq::pdl_wait();  // placed while the kernel before it drains; it never lets its own successor start early (see pq_launch_pdl)
  uint4 v[VPT];
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int j = threadIdx.x + i * THREADS;
    v[i] = make_uint4(0, 0, 0, 0);
    if (j < n_vec)
      asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[i].x), "=r"(v[i].y), "=r"(v[i].z), "=r"(v[i].w) : "l"(row + j));
  }
  uint32_t m2 = 0;  // packed maxima of the patterns without sign
#pragma unroll
  for (int i = 0; i < VPT; ++i)
    m2 = __vmaxu2(__vmaxu2(m2, __vmaxu2(v[i].x & 0x7FFF7FFFu, v[i].y & 0x7FFF7FFFu)), __vmaxu2(v[i].z & 0x7FFF7FFFu, v[i].w & 0x7FFF7FFFu));
  uint32_t m = max(m2 & 0xFFFFu, m2 >> 16);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < THREADS / 32; ++i) m = max(m, red[i]);
  const bool special = m >= 0x7F80u;
  if (special) {  // an infinity or a NaN in the row: the maximum that ignores NaN, then the same two steps
    float mx = 0.0f;
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
      const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) mx = fmaxf(mx, fmaxf(fabsf(__uint_as_float(w[e] << 16)), fabsf(__uint_as_float(w[e] & 0xFFFF0000u))));
    }
    const uint32_t mb = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mb;
    __syncthreads();
    m = 0;
#pragma unroll
    for (int i = 0; i < THREADS / 32; ++i) m = max(m, red[i]);
    m >>= 16;
  }
  const float mx = __uint_as_float(m << 16);
  const float s = mx == 0.0f ? 1.0f : __fdiv_rn(mx, 7.0f);
  if (threadIdx.x == 0) s_w[n] = s;
  // 1 / s or one of its neighbours: half the maximum is a tie in every row, and which way it falls depends on that last bit
  float r = __fdiv_rn(1.0f, s);
  bool same = s > 1e-30f && s < 1e30f && !special;
  {
    const int k = min(static_cast<int>(threadIdx.x & 7), 6), d = static_cast<int>((threadIdx.x & 31) >> 3) - 1;
    const uint32_t h = __float_as_uint((k + 0.5f) * s) >> 16;  // the bf16 value at or below the half-integer; its neighbours: one a lane
    const uint32_t rb = __float_as_uint(r);
    uint32_t ok = 7;  // bit c: candidate c agrees
    const float b = __uint_as_float((h + d) << 16);
    const uint32_t want = static_cast<uint32_t>(code_div(b, s) + 8);
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if ((code_mul(b, __uint_as_float(rb + (c == 2 ? -1 : c))) & 0xFu) != want) ok &= ~(1u << c);
    ok = __reduce_and_sync(0xffffffffu, ok);
    same = same && ok != 0;
    r = __uint_as_float(rb + ((ok & 1) ? 0 : (ok & 2) ? 1 : -1));
  }
  uint32_t* orow = reinterpret_cast<uint32_t*>(wq + n * (K / 2));
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int j = threadIdx.x + i * THREADS;
    if (j >= n_vec) break;
    const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
    uint32_t o = 0;
    if (same) {
      // the sum of (constant + code + 8) * 16^i: no digit carries into the next, the constants' part is subtracted, and flipping
      // every digit's top bit turns code + 8 into the two's-complement code
#pragma unroll
      for (int e = 3; e >= 0; --e)
        o = (o * 16u + code_mul(__uint_as_float(w[e] & 0xFFFF0000u), r)) * 16u + code_mul(__uint_as_float(w[e] << 16), r);
      o = (o - 0x4B400000u * 0x11111111u) ^ 0x88888888u;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        o |= static_cast<uint32_t>((code_div(__uint_as_float(w[e] << 16), s) & 0xF) | ((code_div(__uint_as_float(w[e] & 0xFFFF0000u), s) & 0xF) << 4)) << (8 * e);
    }
    orow[j] = o;
  }
}

}  // namespace

extern "C" pq_status pq_quant_weights(pq_ctx* ctx, const void* W, int64_t N, int64_t K, int64_t ldw, uint8_t* wq,
                                      float* s_w, void* stream) {
  if (!ctx || !W || !wq || !s_w) return PQ_ERR_INVALID_ARG;
  if (N < 0 || K < 0 || ldw < K) return PQ_ERR_INVALID_ARG;
  if (K % 2 != 0) return PQ_ERR_SHAPE;
  if (N == 0 || K == 0) return PQ_OK;
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  // Rows that start on 16 bytes and hold whole vectors are read once; threads and vectors per thread so that four to eight rows'
  // loads are in flight on an SM.
  if (K % 8 == 0 && ldw % 8 == 0 && K <= 32768 && N <= 0x7FFFFFFF && (reinterpret_cast<uintptr_t>(W) & 15) == 0 &&
      (reinterpret_cast<uintptr_t>(wq) & 3) == 0) {
    const __nv_bfloat16* w = static_cast<const __nv_bfloat16*>(W);
    const int k = static_cast<int>(K);
    const unsigned rows = static_cast<unsigned>(N);
    if (K <= 4096) return pq_launch_pdl(quant_weights_once_kernel<128, 4>, dim3(rows), 128, 0, st, w, k, ldw, wq, s_w);
    if (K <= 8192) return pq_launch_pdl(quant_weights_once_kernel<256, 4>, dim3(rows), 256, 0, st, w, k, ldw, wq, s_w);
    if (K <= 16384) return pq_launch_pdl(quant_weights_once_kernel<256, 8>, dim3(rows), 256, 0, st, w, k, ldw, wq, s_w);
    return pq_launch_pdl(quant_weights_once_kernel<512, 8>, dim3(rows), 512, 0, st, w, k, ldw, wq, s_w);
  }
  int grid = static_cast<int>(N < 65535 * 4 ? N : 65535 * 4);
  quant_weights_kernel<<<grid, QW_THREADS, 0, st>>>(
      static_cast<const __nv_bfloat16*>(W), N, K, ldw, wq, s_w);
  return pq_launch_status();
}

// Sum of the signed 4-bit codes of every weight row (the zero-point correction of the asymmetric activation
// quantizer needs it): a warp per row; `(w << 4) & 0xF0F0F0F0` and `w & 0xF0F0F0F0` are the codes times 16
// as signed bytes, summed four at a time with dp4a.
namespace {
__global__ void __launch_bounds__(256) weight_code_sums_kernel(const uint8_t* wq, int64_t N, int64_t kwords, int32_t* wsum) {
  const int lane = threadIdx.x & 31;
  const int64_t row = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= N) return;
  const uint32_t* src = reinterpret_cast<const uint32_t*>(wq) + row * kwords;
  int acc = 0;
  for (int64_t i = lane; i < kwords; i += 32) {
    const uint32_t w = __ldg(src + i);
    acc = __dp4a(static_cast<int>((w << 4) & 0xF0F0F0F0u), 0x01010101, acc);
    acc = __dp4a(static_cast<int>(w & 0xF0F0F0F0u), 0x01010101, acc);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) wsum[row] = acc >> 4;  // exact: every term carries the factor 16
}
}  // namespace

extern "C" pq_status pq_weight_code_sums(pq_ctx* ctx, const uint8_t* wq, int64_t N, int64_t K, int32_t* wsum, void* stream) {
  if (!ctx || !wq || !wsum || N < 0 || K <= 0) return PQ_ERR_INVALID_ARG;
  if (K % 8 != 0) return PQ_ERR_SHAPE;
  if (reinterpret_cast<uintptr_t>(wq) & 3) return PQ_ERR_ALIGN;
  if (N == 0) return PQ_OK;
  weight_code_sums_kernel<<<static_cast<unsigned>((N + 7) / 8), 256, 0, static_cast<cudaStream_t>(stream)>>>(wq, N, K / 8, wsum);
  return pq_launch_status();
}

// Group-wise dynamic KV4 (Table 1, O1: the "group-wise dynamic" KV cache of the paper's comparison setting; with a
// group size of 128 and a head dimension of 128 a group is one (token, head) vector): the step of a vector is
// computed when the token is written and stored beside the codes; attention scales every key's score and every
// value row by the key's own step (the DYN instantiations in pq_kv4.cu and pq_prefill_attn.cu). Here: the append.
#include "pq_common.cuh"

namespace {

constexpr int DY_THREADS = 256;

// ---------------------------------------------------------------------------------------------- append
// Four consecutive threads share one 128-wide vector (32 elements each): maximum over the four, step = max / 7 in
// fp32 (1 for an all-zero vector), fp32 division + round-half-even per element, like the static append.
__global__ void __launch_bounds__(DY_THREADS)
    kv4_append_dyn_kernel(const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v, uint8_t* __restrict__ kq,
                          uint8_t* __restrict__ vq, float* __restrict__ sk_tok, float* __restrict__ sv_tok, int32_t* __restrict__ len,
                          int B, int T_new, int Hkv, int Tmax, int64_t ld_tok, int32_t* status, uint32_t* ticket) {
  __shared__ int bad;
  __shared__ int last;
  if (threadIdx.x == 0) bad = 0, last = 0;
  __syncthreads();
  for (int b = threadIdx.x; b < B; b += DY_THREADS)
    if (len[b] < 0 || len[b] + T_new > Tmax) bad = 1;
  __syncthreads();
  if (bad) {  // every CTA reaches the same verdict: nothing is written, len stays
    if (blockIdx.x == 0 && threadIdx.x == 0) pq::report(status, PQ_ERR_SHAPE);
    return;
  }
  const int64_t n_units = static_cast<int64_t>(B) * T_new * Hkv * 4;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * DY_THREADS;
  for (int64_t base = static_cast<int64_t>(blockIdx.x) * DY_THREADS; base < n_units; base += stride) {  // the same trip count for a warp
    const int64_t unit = base + threadIdx.x;
    const bool ok = unit < n_units;  // whole groups of four: n_units is a multiple of 4
    const int part = static_cast<int>(unit & 3);
    const int64_t bth = ok ? unit >> 2 : 0;
    const int h = static_cast<int>(bth % Hkv);
    const int64_t bt = bth / Hkv;
    const int t = static_cast<int>(bt % T_new), b = static_cast<int>(bt / T_new);
    const int64_t pos = len[b] + t;
    const int64_t src = bt * ld_tok + h * 128 + part * 32;
    const int64_t vec = (static_cast<int64_t>(b) * Hkv + h) * Tmax + pos;
#pragma unroll
    for (int which = 0; which < 2; ++which) {
      const uint4* in = reinterpret_cast<const uint4*>((which ? v : k) + src);
      uint4 w[4];
      float mx = 0.0f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        w[i] = ok ? __ldg(in + i) : make_uint4(0, 0, 0, 0);
        const uint32_t ww[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) mx = fmaxf(mx, fmaxf(fabsf(__uint_as_float(ww[j] << 16)), fabsf(__uint_as_float(ww[j] & 0xFFFF0000u))));
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float s = mx == 0.0f ? 1.0f : __fdiv_rn(mx, 7.0f);
      uint32_t o[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t ww[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
        uint32_t acc = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int ca = max(-8, min(7, __float2int_rn(__fdiv_rn(__uint_as_float(ww[j] << 16), s))));
          const int cc = max(-8, min(7, __float2int_rn(__fdiv_rn(__uint_as_float(ww[j] & 0xFFFF0000u), s))));
          acc |= static_cast<uint32_t>((ca & 0xF) | ((cc & 0xF) << 4)) << (8 * j);
        }
        o[i] = acc;
      }
      if (ok) {
        *reinterpret_cast<uint4*>((which ? vq : kq) + vec * 64 + part * 16) = make_uint4(o[0], o[1], o[2], o[3]);
        if (part == 0) (which ? sv_tok : sk_tok)[vec] = s;
      }
    }
  }
  if (gridDim.x > 1) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
  } else if (threadIdx.x == 0) {
    last = 1;
  }
  __syncthreads();
  if (last) {
    for (int b = threadIdx.x; b < B; b += DY_THREADS) len[b] += T_new;
    if (threadIdx.x == 0 && gridDim.x > 1) *ticket = 0;
  }
}

}  // namespace

pq_status pq_kv4_append_dyn_launch(pq_ctx* ctx, const pq_kv4_cache* c, const void* k, const void* v, int32_t T_new, int64_t ld_tok,
                                   cudaStream_t st) {
  const int64_t n_units = static_cast<int64_t>(c->B) * T_new * c->Hkv * 4;
  int64_t grid = (n_units + DY_THREADS - 1) / DY_THREADS;
  if (grid > 8LL * ctx->sm_count) grid = 8LL * ctx->sm_count;
  kv4_append_dyn_kernel<<<static_cast<int>(grid), DY_THREADS, 0, st>>>(
      static_cast<const __nv_bfloat16*>(k), static_cast<const __nv_bfloat16*>(v), c->kq, c->vq, c->sk_tok, c->sv_tok, c->len, c->B, T_new,
      c->Hkv, c->Tmax, ld_tok, ctx->d_status, ctx->d_tickets);
  return pq_launch_status();
}

// Entry point of the W4A4 linear layer: argument checks and the choice between the tensor-core
// kernels (prefill-shaped) and the weight-streaming kernel (decode-shaped).
#include "pq_common.cuh"

pq_status pq_gemm_pair_launch(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, const float* s_a, const float* s_w,
                              void* out, int64_t ldo, int64_t M, int64_t N, int64_t K, int32_t* acc_dbg, cudaStream_t st);
pq_status pq_gemm_pair_ts_launch(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, const float* s_a, const float* s_w,
                                 void* out, int64_t ldo, int64_t M, int64_t N, int64_t K, int32_t* acc_dbg, cudaStream_t st,
                                 bool a8, const float* s_row, const int32_t* zp, const int32_t* wsum);
pq_status pq_gemm_stream_launch(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, const float* s_a,
                                const float* s_w, void* out, int64_t ldo, int64_t M, int64_t N, int64_t K,
                                int32_t* acc_dbg, cudaStream_t st, bool per_token, bool a8, const int32_t* zp,
                                const int32_t* wsum);

pq_status pq_gemm_split_launch(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, const float* s_a, const float* s_w, void* out,
                               int64_t ldo, int64_t M, int64_t N, int64_t K, int32_t* acc_dbg, cudaStream_t st, bool a8,
                               const float* s_row, const int32_t* zp, const int32_t* wsum);

// Chooses the kernel for m rows (row_begin already applied). s_row: per-token steps instead of s_a; zp, wsum: Eq. 1's
// zero point and the weight code sums; a8: one s8 code per activation.
static pq_status run_gemm(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, const float* s_a, const float* s_w, void* out, int64_t ldo,
                          int64_t m, int64_t N, int64_t K, int32_t* dbg, void* stream, bool a8, const float* s_row, const int32_t* zp,
                          const int32_t* wsum) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // Weight-streaming kernel or split-K tensor-core kernel (figures: rotate+quantize and GEMM in a graph, us, streaming against
  // split). The streaming kernel has the shorter chain, but expands the tokens again for every 16 channels and has no K split:
  //   up to 8 tokens   always streaming. Alone behind its rotation kernel the other is faster on 8192 x 28672 (1 token: 29.2 / 24.4)
  //                    and 8192 x 8192 (11.4 / 10.4), but inside a decode layer the streaming kernel's shorter chain and earlier
  //                    weight requests win: whole 70B layer 124 / 132 us
  //   9 to 16 tokens   only layers below 20 M weights (16 tokens, 4096 x 4096: 5.6 / 7.1; 6144 x 4096: 8.1 / 7.8,
  //                    28672 x 4096: 21.3 / 15.7, 8192 x 28672: 33.9 / 26.0)
  //   up to 96         always split (CTA pairs: 40 tokens, 28672 x 4096: 23.0 / 19.8; 8192 x 28672: 59.5 / 31.6)
  //   97 to 128        while every channel tile has its CTAs at once (128 tokens, pairs against split, 57344 x 8192: 74.6 / 85.7,
  //                    28672 x 4096: 25.1 / 27.0; but 10240 x 8192: 25.3 / 23.5)
  //   above            while the 256-token tiles leave room for two K splits (pairs against split at 256 tokens: 8192 x 8192 26.0 / 23.5,
  //                    4096 x 14336 35.7 / 24.2, 6144 x 4096 17.4 / 17.2; at 400, 4096 x 14336 37.8 / 31.9, 4096 x 4096 17.7 / 17.3). With a single
  //                    split the pairs win: 57344 x 8192 at 200 tokens 91 / 129, 28672 x 4096 30.1 / 39.3, 10240 x 8192 31.5 / 35.8, 6144 x 4096
  //                    at 300 17.9 / 21.7, 4096 x 14336 at 515 39.2 / 49.4.
  const int64_t ctiles = (N + 127) / 128, weights = N * K;
  const bool split = m <= 8     ? false
                     : m <= 16  ? weights >= (int64_t{20} << 20)
                     : m <= 96  ? true
                     : m <= 128 ? ctiles <= ctx->sm_count
                                : 2 * ((m + 255) / 256) * ctiles <= ctx->sm_count * 7 / 8;
  if (split) return pq_gemm_split_launch(ctx, xq, wq, s_a, s_w, out, ldo, m, N, K, dbg, st, a8, s_row, zp, wsum);
  if (m <= 16)
    return pq_gemm_stream_launch(ctx, xq, wq, s_row ? s_row : s_a, s_w, out, ldo, m, N, K, dbg, st, s_row != nullptr, a8, zp, wsum);
  // CTA pairs. Few rounds of 8-bit tiles, and 4-bit tokens always: weights in tensor memory, tiles as wide as fit the chip
  // (pq_gemm_tc3.cu). More than three rounds of 8-bit tiles at K <= 8192: both operands in shared memory, two whole accumulators
  // (pq_gemm_tc2.cu, with the figures).
  const int64_t tiles = ((m + 255) / 256) * ((N + 255) / 256);
  if (a8 && K <= 8192 && tiles > 3 * (ctx->sm_count / 2)) return pq_gemm_pair_launch(ctx, xq, wq, s_a, s_w, out, ldo, m, N, K, dbg, st);
  return pq_gemm_pair_ts_launch(ctx, xq, wq, s_a, s_w, out, ldo, m, N, K, dbg, st, a8, s_row, zp, wsum);
}

extern "C" size_t pq_w4a4_gemm_workspace_bytes(int64_t, int64_t, int64_t) { return 0; }

extern "C" pq_status pq_w4a4_gemm(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, const float* s_a,
                                  const float* s_w, void* out, int64_t ldo, int64_t M, int64_t N, int64_t K,
                                  int64_t row_begin, int32_t* acc_dbg, void* ws, size_t ws_bytes, void* stream) {
  (void)ws;
  (void)ws_bytes;
  if (!ctx || !xq || !wq || !s_a || !s_w || !out) return PQ_ERR_INVALID_ARG;
  if (M < 0 || N < 0 || K < 0 || row_begin < 0 || ldo < N) return PQ_ERR_INVALID_ARG;
  if (K % 32 != 0 || K > 65536 || M > (1 << 30) || N > (1 << 30)) return PQ_ERR_SHAPE;
  if ((reinterpret_cast<uintptr_t>(xq) & 15) || (reinterpret_cast<uintptr_t>(wq) & 15) ||
      (reinterpret_cast<uintptr_t>(out) & 1))
    return PQ_ERR_ALIGN;
  if (row_begin >= M || N == 0) return PQ_OK;
  const int64_t m = M - row_begin;
  const uint8_t* xq0 = xq + row_begin * (K / 2);
  void* out0 = static_cast<__nv_bfloat16*>(out) + row_begin * ldo;
  int32_t* dbg0 = acc_dbg ? acc_dbg + row_begin * N : nullptr;
  if (K == 0) return PQ_ERR_SHAPE;
  return run_gemm(ctx, xq0, wq, s_a, s_w, out0, ldo, m, N, K, dbg0, stream, false, nullptr, nullptr, nullptr);
}

// W4A8 (Sec. 5.1): the token operand is one s8 code per element. The kernels and the rule are those of the 4-bit calls
// but for the largest launches (see run_gemm).
extern "C" pq_status pq_w4a8_gemm(pq_ctx* ctx, const int8_t* xq8, const uint8_t* wq, const float* s_a,
                                  const float* s_w, void* out, int64_t ldo, int64_t M, int64_t N, int64_t K,
                                  int64_t row_begin, int32_t* acc_dbg, void* stream) {
  if (!ctx || !xq8 || !wq || !s_a || !s_w || !out) return PQ_ERR_INVALID_ARG;
  if (M < 0 || N < 0 || K < 0 || row_begin < 0 || ldo < N) return PQ_ERR_INVALID_ARG;
  // |code_a * 16 code_w| <= 128 * 128 per term: K <= 65536 keeps the int32 accumulator exact
  if (K % 32 != 0 || K == 0 || K > 65536 || M > (1 << 30) || N > (1 << 30)) return PQ_ERR_SHAPE;
  if ((reinterpret_cast<uintptr_t>(xq8) & 15) || (reinterpret_cast<uintptr_t>(wq) & 15) ||
      (reinterpret_cast<uintptr_t>(out) & 1))
    return PQ_ERR_ALIGN;
  if (row_begin >= M || N == 0) return PQ_OK;
  const int64_t m = M - row_begin;
  const uint8_t* xq0 = reinterpret_cast<const uint8_t*>(xq8) + row_begin * K;
  void* out0 = static_cast<__nv_bfloat16*>(out) + row_begin * ldo;
  int32_t* dbg0 = acc_dbg ? acc_dbg + row_begin * N : nullptr;
  return run_gemm(ctx, xq0, wq, s_a, s_w, out0, ldo, m, N, K, dbg0, stream, true, nullptr, nullptr, nullptr);
}

// W4A4 with per-token dynamic activation steps (Table 1, O1): out[t,n] = bf16(acc * s_tok[t] * s_w[n]).
extern "C" pq_status pq_w4a4_gemm_rows(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, const float* s_tok,
                                       const float* s_w, void* out, int64_t ldo, int64_t M, int64_t N, int64_t K,
                                       int64_t row_begin, int32_t* acc_dbg, void* stream) {
  if (!ctx || !xq || !wq || !s_tok || !s_w || !out) return PQ_ERR_INVALID_ARG;
  if (M < 0 || N < 0 || K < 0 || row_begin < 0 || ldo < N) return PQ_ERR_INVALID_ARG;
  if (K % 32 != 0 || K == 0 || K > 65536 || M > (1 << 30) || N > (1 << 30)) return PQ_ERR_SHAPE;
  if ((reinterpret_cast<uintptr_t>(xq) & 15) || (reinterpret_cast<uintptr_t>(wq) & 15) ||
      (reinterpret_cast<uintptr_t>(out) & 1))
    return PQ_ERR_ALIGN;
  if (row_begin >= M || N == 0) return PQ_OK;
  const int64_t m = M - row_begin;
  const uint8_t* xq0 = xq + row_begin * (K / 2);
  const float* s0 = s_tok + row_begin;
  void* out0 = static_cast<__nv_bfloat16*>(out) + row_begin * ldo;
  int32_t* dbg0 = acc_dbg ? acc_dbg + row_begin * N : nullptr;
  return run_gemm(ctx, xq0, wq, nullptr, s_w, out0, ldo, m, N, K, dbg0, stream, false, s0, nullptr, nullptr);
}

// W4A4 with the activation quantizer of Eq. 1 as printed (zero point z): the stored token codes are u - 8,
// out[t,n] = bf16(s_a * s_w[n] * sum_k (u[t,k] - z) * w[n,k]); wsum[n] = sum_k w[n,k] comes from pq_weight_code_sums.
extern "C" pq_status pq_w4a4_gemm_asym(pq_ctx* ctx, const uint8_t* xq, const uint8_t* wq, const float* s_a,
                                       const int32_t* z_a, const float* s_w, const int32_t* wsum, void* out, int64_t ldo,
                                       int64_t M, int64_t N, int64_t K, int64_t row_begin, int32_t* acc_dbg,
                                       void* stream) {
  if (!ctx || !xq || !wq || !s_a || !z_a || !s_w || !wsum || !out) return PQ_ERR_INVALID_ARG;
  if (M < 0 || N < 0 || K < 0 || row_begin < 0 || ldo < N) return PQ_ERR_INVALID_ARG;
  if (K % 32 != 0 || K == 0 || K > 65536 || M > (1 << 30) || N > (1 << 30)) return PQ_ERR_SHAPE;
  if ((reinterpret_cast<uintptr_t>(xq) & 15) || (reinterpret_cast<uintptr_t>(wq) & 15) ||
      (reinterpret_cast<uintptr_t>(out) & 1))
    return PQ_ERR_ALIGN;
  if (row_begin >= M || N == 0) return PQ_OK;
  const int64_t m = M - row_begin;
  const uint8_t* xq0 = xq + row_begin * (K / 2);
  void* out0 = static_cast<__nv_bfloat16*>(out) + row_begin * ldo;
  int32_t* dbg0 = acc_dbg ? acc_dbg + row_begin * N : nullptr;
  return run_gemm(ctx, xq0, wq, s_a, s_w, out0, ldo, m, N, K, dbg0, stream, false, nullptr, z_a, wsum);
}

// bf16 linear layer out = a w^T + bias on the tcgen05 GEMM mainloop (the QKV and output
// projections of the attention block, Sec. 3.1).  The output leaves the SM through TMA stores of
// 32-row x 64-column blocks, so `out` needs a 16-byte aligned base and a row pitch (n) that is a
// multiple of 8 elements.
#include "gemm_tc.cuh"
#include "runtime.h"

namespace lv {

// out [m, n] = epi(a [m, k] w [n, k]^T)
template <class Epi>
static cudaError_t launch_gemm_out(litevggt_ctx* ctx, const __nv_bfloat16* a, long long m, long long k,
                                   const __nv_bfloat16* w, long long n, __nv_bfloat16* out, const Epi& epi,
                                   bool heads, const ZeroWords& zero, cudaStream_t s, int* launches) {
  const int columns = gemm_tile_columns(m, n, k, heads, ctx->num_sms), bn = columns != 0 ? columns : 256;
  CUtensorMap tmap_a, tmap_b, tmap_out;
  if (!make_tmap_bf16_2d(ctx->encode_tiled, &tmap_a, a, (uint64_t)k, (uint64_t)m, (uint64_t)k, kGemmBK, kGemmBM) ||
      !make_tmap_bf16_2d(ctx->encode_tiled, &tmap_b, w, (uint64_t)k, (uint64_t)n, (uint64_t)k, kGemmBK, columns != 0 ? bn / 2 : bn) ||
      !make_tmap_bf16_2d(ctx->encode_tiled, &tmap_out, out, (uint64_t)n, (uint64_t)m, (uint64_t)n, kGemmOutChunkCols,
                         32))
    return cudaErrorInvalidValue;
  const long long rows = columns != 0 ? 2 * kGemmBM : kGemmBM, tiles = ((m + rows - 1) / rows) * ((n + bn - 1) / bn);
  ++*launches;
  auto run = [&](auto launch) { return launch(tmap_a, tmap_b, tmap_out, m, n, k, epi, tiles, ctx->num_sms, ctx->ws.status, zero, next_stamp(ctx), s); };
  switch (columns) {
    case 0: return run(gemm_launch<Epi, 256, 1>);
    case 64: return run(gemm_launch<Epi, 64, 2>);
    case 128: return run(gemm_launch<Epi, 128, 2>);
    case 160: return run(gemm_launch<Epi, 160, 2>);
    case 192: return run(gemm_launch<Epi, 192, 2>);
    case 224: return run(gemm_launch<Epi, 224, 2>);
    default: return run(gemm_launch<Epi, 256, 2>);
  }
}

cudaError_t launch_linear(litevggt_ctx* ctx, const __nv_bfloat16* a, long long m, long long k, const __nv_bfloat16* w,
                          long long n, const __nv_bfloat16* bias, const ZeroWords& zero, __nv_bfloat16* out, cudaStream_t s,
                          int* launches) {
  if (m == 0) return cudaSuccess;
  LinearEpilogue epi = {};
  epi.bias = bias;
  epi.m_rows = (int)m;
  epi.n_cols = (int)n;
  epi.scale = 1.0f;
  epi.out = out;
  return launch_gemm_out(ctx, a, m, k, w, n, out, epi, false, zero, s, launches);
}

cudaError_t launch_linear_scaled(litevggt_ctx* ctx, const __nv_bfloat16* a, long long m, long long k,
                                 const __nv_bfloat16* w, long long n, const __nv_bfloat16* bias, int scale_begin,
                                 int scale_end, float scale, const LinearStat& stat, __nv_bfloat16* out, cudaStream_t s,
                                 int* launches) {
  if (m == 0) return cudaSuccess;
  if (scale_begin % 64 != 0 || scale_end % 64 != 0) return cudaErrorInvalidValue;
  if (stat.key_norm != nullptr && stat.seq_len <= 0) return cudaErrorInvalidValue;
  if (stat.amax != nullptr) {
    cudaError_t e = cudaMemsetAsync(stat.amax, 0, (size_t)(n / 64) * sizeof(float), s);
    if (e != cudaSuccess) return e;
  }
  LinearEpilogue epi;
  epi.bias = bias;
  epi.m_rows = (int)m;
  epi.n_cols = (int)n;
  epi.scale_begin = scale_begin;
  epi.scale_end = scale_end;
  epi.scale = scale;
  epi.stat_kind = stat.key_norm != nullptr ? (stat.values_only ? kStatValues : kStatKeyNorm) : stat.amax != nullptr ? kStatAmax : kStatNone;
  epi.seq_len = (int)stat.seq_len;
  epi.stat = stat.key_norm != nullptr ? stat.key_norm : stat.amax;
  // (a context without counters runs attention launches that need none)
  const ZeroWords taken{reinterpret_cast<uint32_t*>(ctx->ws.attn_taken), ctx->ws.attn_taken != nullptr ? kAttnCounters : 0};
  epi.out = out;
  return launch_gemm_out(ctx, a, m, k, w, n, out, epi, true, taken, s, launches);
}

// out = act(a w^T + bias) + residual, the two layers of the transformer MLP (fc1: GELU, no residual;
// fc2: identity, residual = the block's input).
cudaError_t launch_linear_mlp(litevggt_ctx* ctx, const __nv_bfloat16* a, long long m, long long k,
                              const __nv_bfloat16* w, long long n, const __nv_bfloat16* bias, int gelu,
                              const __nv_bfloat16* residual, const ZeroWords& zero, __nv_bfloat16* out, cudaStream_t s,
                              int* launches) {
  if (m == 0) return cudaSuccess;
  MlpEpilogue epi;
  epi.bias = bias;
  epi.residual = residual;
  epi.m_rows = (int)m;
  epi.n_cols = (int)n;
  epi.ld_res = n;
  epi.gelu = gelu;
  epi.out = out;
  return launch_gemm_out(ctx, a, m, k, w, n, out, epi, false, zero, s, launches);
}

}  // namespace lv

// Size-weighted merge and gather-unmerge (Sec. 3.4: merge equation and "Token Unmerging").
// Both are pure HBM streaming: one warp per 2 KB row, 16-byte vector accesses, 512
// contiguous bytes per warp instruction.
//
// Merge: row j of the merged sequence is the mean of its own token and the src tokens
// listed for it in the CSR, summed in fp32 in ascending token order (deterministic) and
// rounded once; rows that absorb nothing are copied bit-exactly.
// Unmerge: out_i = y'[dst_of[i]] (+ residual_i, added in fp32).
#include "common.cuh"
#include "runtime.h"

namespace lv {

constexpr int kRowThreads = 256;
constexpr int kRowsPerCta = kRowThreads / 32;

__device__ __forceinline__ void add_row(float (&acc)[32], const uint4 (&v)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint32_t w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      acc[q * 8 + 2 * i] += bf16_lo(w[i]);
      acc[q * 8 + 2 * i + 1] += bf16_hi(w[i]);
    }
  }
}

__device__ __forceinline__ void load_row(uint4 (&v)[4], const __nv_bfloat16* row, int lane) {
  const uint4* p = reinterpret_cast<const uint4*>(row);
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = p[q * 32 + lane];
}

// kRows: absorbed rows in flight.  Few blocks last as long as their longest row, a chain of loads, and four shorten it; many
// are bound by HBM and want warps, of which 96 registers leave 16 an SM where two rows' 64 leave 32 (us, two / four: 543
// merged rows 4.7 / 3.9, 2,520 5.6 / 4.7, 5,205 6.3 / 7.2, 83,280 107 / 145; the line is two and a half blocks an SM, 2,960 rows).
template <int kRows>
__global__ void __launch_bounds__(kRowThreads)
merge_kernel(const __nv_bfloat16* __restrict__ x, const int* __restrict__ kept_idx, const int* __restrict__ seg_off,
             const int* __restrict__ seg_src, __nv_bfloat16* __restrict__ xm, long long n_merged,
             long long n_tokens, long long n_remove, uint32_t* status, Stamp stamp) {
  const Span span(stamp);
  const int lane = threadIdx.x & 31;
  const long long j = (long long)blockIdx.x * kRowsPerCta + (threadIdx.x >> 5);
  if (j >= n_merged) return;
  long long own = kept_idx[j];
  int s0 = seg_off[j], s1 = seg_off[j + 1];
  if (own < 0 || own >= n_tokens || s0 < 0 || s1 < s0 || s1 > n_remove) {
    if (lane == 0) atomicOr(status, kStatusBounds);
    own = own < 0 || own >= n_tokens ? 0 : own;
    s1 = s0;
  }
  uint4 v[4];
  load_row(v, x + own * 1024, lane);
  uint4* out = reinterpret_cast<uint4*>(xm + j * 1024);
  if (s1 == s0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) out[q * 32 + lane] = v[q];
    return;
  }
  float acc[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i] = 0.0f;
  add_row(acc, v);
  int s = s0;
  for (; s + kRows <= s1; s += kRows) {  // kRows rows in flight
    long long t[kRows];
    bool inside = true;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      t[i] = seg_src[s + i];
      inside = inside && t[i] >= 0 && t[i] < n_tokens;
    }
    if (!inside) {
      if (lane == 0) atomicOr(status, kStatusBounds);
      continue;
    }
    uint4 a[kRows][4];
#pragma unroll
    for (int i = 0; i < kRows; ++i) load_row(a[i], x + t[i] * 1024, lane);
#pragma unroll
    for (int i = 0; i < kRows; ++i) add_row(acc, a[i]);
  }
  if (s < s1) {  // the rest together too
    uint4 a[kRows - 1][4];
#pragma unroll
    for (int i = 0; i < kRows - 1; ++i) {
      const long long t = s + i < s1 ? seg_src[s + i] : -1;
      if (s + i < s1 && t >= 0 && t < n_tokens) {
        load_row(a[i], x + t * 1024, lane);
      } else {
        if (s + i < s1 && lane == 0) atomicOr(status, kStatusBounds);
#pragma unroll
        for (int q = 0; q < 4; ++q) a[i][q] = make_uint4(0u, 0u, 0u, 0u);
      }
    }
#pragma unroll
    for (int i = 0; i < kRows - 1; ++i)
      if (s + i < s1) add_row(acc, a[i]);
  }
  const float denom = (float)(1 + s1 - s0);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint4 o;
    o.x = pack_bf16(acc[q * 8 + 0] / denom, acc[q * 8 + 1] / denom);
    o.y = pack_bf16(acc[q * 8 + 2] / denom, acc[q * 8 + 3] / denom);
    o.z = pack_bf16(acc[q * 8 + 4] / denom, acc[q * 8 + 5] / denom);
    o.w = pack_bf16(acc[q * 8 + 6] / denom, acc[q * 8 + 7] / denom);
    out[q * 32 + lane] = o;
  }
}

template <bool kSmall>  // a grid of at most kOverlapBlocks blocks (common.cuh: SpanOf)
__global__ void __launch_bounds__(kRowThreads)
unmerge_kernel(const __nv_bfloat16* __restrict__ ym, const int* __restrict__ dst_of,
               const __nv_bfloat16* __restrict__ residual, __nv_bfloat16* __restrict__ out, long long n_tokens,
               long long n_merged, uint32_t* status, Stamp stamp) {
  const SpanOf<kSmall> span(stamp);
  const int lane = threadIdx.x & 31;
  const long long i = (long long)blockIdx.x * kRowsPerCta + (threadIdx.x >> 5);
  if (i >= n_tokens) return;
  long long row = dst_of[i];
  if (row < 0 || row >= n_merged) {
    if (lane == 0) atomicOr(status, kStatusBounds);
    row = 0;
  }
  uint4 v[4];
  load_row(v, ym + row * 1024, lane);
  uint4* o = reinterpret_cast<uint4*>(out + i * 1024);
  if (residual == nullptr) {
#pragma unroll
    for (int q = 0; q < 4; ++q) o[q * 32 + lane] = v[q];
    return;
  }
  uint4 r[4];
  load_row(r, residual + i * 1024, lane);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint32_t a[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
    const uint32_t b[4] = {r[q].x, r[q].y, r[q].z, r[q].w};
    uint32_t c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k] = pack_bf16(bf16_lo(a[k]) + bf16_lo(b[k]), bf16_hi(a[k]) + bf16_hi(b[k]));
    o[q * 32 + lane] = make_uint4(c[0], c[1], c[2], c[3]);
  }
}

// The unmerge of merged rows [row0, row1) only: to their own tokens and to the src tokens of their segments, into memory that
// may be the host's.  PCIe bounds it (2 KB a token at 45 GB/s by these stores), so few warps do; what matters is that they are all
// busy to the end (a token each, not a row: some anchors stand for hundreds) and how they get on with the attention
// beside them.  Its CTA leaves 1024 registers of every scheduler free: one block of four warps on 32 registers, a warp
// half a token at a time.  Where stores queue up for PCIe the attention's warps on that SM wait behind them, so
// the blocks are no more than it takes (pass of 32 frames of 37 x 37: 12 blocks 2.73 ms, 16: 2.71, 20: 2.69, 24: 2.66,
// 32: 2.80, 48: 2.81; a slab's attention 355 us beside 16 of them, 380 beside 24, 480 beside 48).
constexpr int kOutThreads = 128;
constexpr int kOutBlocks = 24;
__global__ void __launch_bounds__(kOutThreads, 16)
unmerge_rows_kernel(const __nv_bfloat16* __restrict__ ym, const int* __restrict__ dst_of, const int* __restrict__ kept_idx,
                    const int* __restrict__ seg_off, const int* __restrict__ seg_src, const __nv_bfloat16* __restrict__ residual,
                    __nv_bfloat16* __restrict__ out, int row0, int row1, int n_tokens, int n_merged, int n_remove, uint32_t* status,
                    Stamp stamp) {
  const Span span(stamp);
  const int lane = threadIdx.x & 31, step = gridDim.x * (kOutThreads / 32);
  int first = seg_off[row0], last = seg_off[row1];
  if (first < 0 || last < first || last > n_remove) {
    if (threadIdx.x == 0) atomicOr(status, kStatusBounds);
    first = last = 0;
  }
  const int rows = row1 - row0, count = rows + (last - first);
  auto token_at = [&](int i) { return i >= count ? 0 : i < rows ? kept_idx[row0 + i] : seg_src[first + i - rows]; };
  int i = blockIdx.x * (kOutThreads / 32) + (int)(threadIdx.x >> 5);
  int ahead = token_at(i);
  for (; i < count; i += step) {
    const int token = ahead;
    ahead = token_at(i + step);
    const int row = token >= 0 && token < n_tokens ? dst_of[token] : -1;
    if (row < 0 || row >= n_merged) {
      if (lane == 0) atomicOr(status, kStatusBounds);
      continue;
    }
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      const int at = half * 64 + lane;  // in 16-byte units
      const uint4* rp = reinterpret_cast<const uint4*>(residual + (long long)token * 1024) + at;
      const uint4* yp = reinterpret_cast<const uint4*>(ym + (long long)row * 1024) + at;
      const uint4 r0 = rp[0], r1 = rp[32], y0 = yp[0], y1 = yp[32];
      uint4* o = reinterpret_cast<uint4*>(out + (long long)token * 1024) + at;
      auto sum = [](uint32_t a, uint32_t b) { return pack_bf16(bf16_lo(a) + bf16_lo(b), bf16_hi(a) + bf16_hi(b)); };
      o[0] = make_uint4(sum(y0.x, r0.x), sum(y0.y, r0.y), sum(y0.z, r0.z), sum(y0.w, r0.w));
      o[32] = make_uint4(sum(y1.x, r1.x), sum(y1.y, r1.y), sum(y1.z, r1.z), sum(y1.w, r1.w));
    }
  }
}

cudaError_t launch_unmerge_rows(const litevggt_ctx* ctx, const int* dst_of, const int* kept_idx, const int* seg_off,
                                const int* seg_src, const __nv_bfloat16* ym, const __nv_bfloat16* residual, __nv_bfloat16* out,
                                long long row0, long long row1, cudaStream_t s, int* launches) {
  const Sizes& z = ctx->sz;
  // Shared memory for whoever comes beside it: an SM that this kernel reaches first would be set up with little, and keep
  // the attention's CTA away until it is done.
  static std::atomic<unsigned long long> carveout_set{0};
  const cudaError_t e = set_attribute_once(reinterpret_cast<const void*>(unmerge_rows_kernel), cudaFuncAttributePreferredSharedMemoryCarveout,
                                           cudaSharedmemCarveoutMaxShared, carveout_set);
  if (e != cudaSuccess) return e;
  ++*launches;
  return launch_clusters(1, false, unmerge_rows_kernel, dim3(kOutBlocks), kOutThreads, 0, s, ym, dst_of, kept_idx, seg_off, seg_src,
                         residual, out, (int)row0, (int)row1, (int)z.n_tokens, (int)z.n_merged, (int)z.n_remove, ctx->ws.status,
                         next_stamp(ctx));
}

// LayerNorm over the 1024 channels of every row (the pre-norm of the transformer blocks, Sec. 3.1):
// y = (x - mean) / sqrt(var + eps) * gamma + beta, population variance, two passes over the row held
// in registers, fp32, one rounding.  One warp per row like the kernels above.
__global__ void __launch_bounds__(kRowThreads)
layernorm_kernel(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ gamma,
                 const __nv_bfloat16* __restrict__ beta, __nv_bfloat16* __restrict__ out, long long rows, float eps,
                 Stamp stamp) {
  const Span span(stamp);
  const int lane = threadIdx.x & 31;
  const long long i = (long long)blockIdx.x * kRowsPerCta + (threadIdx.x >> 5);
  if (i >= rows) return;
  uint4 v[4];
  load_row(v, x + i * 1024, lane);
  float f[32];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint32_t w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      f[q * 8 + 2 * k] = bf16_lo(w[k]);
      f[q * 8 + 2 * k + 1] = bf16_hi(w[k]);
    }
  }
  float sum = 0.0f;
#pragma unroll
  for (int k = 0; k < 32; ++k) sum += f[k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const float mean = sum * (1.0f / 1024.0f);
  float ss = 0.0f;
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    f[k] -= mean;
    ss = fmaf(f[k], f[k], ss);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  const float rstd = rsqrtf(ss * (1.0f / 1024.0f) + eps);
  uint4* op = reinterpret_cast<uint4*>(out + i * 1024);
  const uint4* gp = reinterpret_cast<const uint4*>(gamma);
  const uint4* bp = reinterpret_cast<const uint4*>(beta);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint4 g = gp[q * 32 + lane], b = bp[q * 32 + lane];
    const uint32_t gw[4] = {g.x, g.y, g.z, g.w}, bw[4] = {b.x, b.y, b.z, b.w};
    uint32_t c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      c[k] = pack_bf16(fmaf(f[q * 8 + 2 * k] * rstd, bf16_lo(gw[k]), bf16_lo(bw[k])),
                       fmaf(f[q * 8 + 2 * k + 1] * rstd, bf16_hi(gw[k]), bf16_hi(bw[k])));
    op[q * 32 + lane] = make_uint4(c[0], c[1], c[2], c[3]);
  }
}

cudaError_t launch_layernorm(const __nv_bfloat16* x, const __nv_bfloat16* gamma, const __nv_bfloat16* beta,
                             __nv_bfloat16* out, long long rows, float eps, const Stamp& stamp, cudaStream_t s,
                             int* launches) {
  if (rows == 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((rows + kRowsPerCta - 1) / kRowsPerCta);
  ++*launches;
  return launch(layernorm_kernel, dim3(blocks), kRowThreads, 0, s, x, gamma, beta, out, rows, eps, stamp);
}

cudaError_t launch_merge(const litevggt_ctx* ctx, const litevggt_plan* plan, const __nv_bfloat16* x,
                         __nv_bfloat16* xm, cudaStream_t s, int* launches) {
  const Sizes& z = ctx->sz;
  const unsigned blocks = (unsigned)((z.n_merged + kRowsPerCta - 1) / kRowsPerCta);
  ++*launches;
  const bool few = 2 * (long long)blocks <= 5 * ctx->num_sms;
  return launch(few ? merge_kernel<4> : merge_kernel<2>, dim3(blocks), kRowThreads, 0, s, x, plan->kept_idx, plan->seg_off,
                plan->seg_src, xm, z.n_merged, z.n_tokens, z.n_remove, ctx->ws.status, next_stamp(ctx));
}

cudaError_t launch_unmerge(const litevggt_ctx* ctx, const litevggt_plan* plan, const __nv_bfloat16* ym,
                           const __nv_bfloat16* residual, __nv_bfloat16* out, cudaStream_t s, int* launches) {
  const Sizes& z = ctx->sz;
  const unsigned blocks = (unsigned)((z.n_tokens + kRowsPerCta - 1) / kRowsPerCta);
  ++*launches;
  return launch(blocks <= kOverlapBlocks ? unmerge_kernel<true> : unmerge_kernel<false>, dim3(blocks), kRowThreads, 0, s, ym, plan->dst_of, residual, out, z.n_tokens, z.n_merged,
                ctx->ws.status, next_stamp(ctx));
}

}  // namespace lv

// What the files behind the C ABI share on the host side: argument checks, stopwatch slots, the workspace that
// is allocated on first use, the state of the key norms.
#pragma once

#include "runtime.h"

namespace lv {

struct DeviceGuard {
  int prev = -1;
  bool ok = false;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) return;
    ok = cudaSetDevice(dev) == cudaSuccess;
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline bool ctx_ok(const litevggt_ctx* c) { return c != nullptr && c->magic == kCtxMagic; }
inline bool plan_ok(const litevggt_plan* p) { return p != nullptr && p->magic == kPlanMagic; }

inline void bump(litevggt_ctx* ctx, int n) { ctx->launches += n; }

// Hands the launches of one step the stopwatch slot that their kernels write; `launches` and `e` are what
// the step counts its launches in and ends with.
struct StepTimer {
  litevggt_ctx* ctx;
  int which, slot;
  const int& launches;
  const int before;
  const cudaError_t& e;
  StepTimer(litevggt_ctx* c, int w, const int& n, const cudaError_t& err)
      : ctx(c), which(w), slot(c->timers.used[w] % kTimerSlots), launches(n), before(n), e(err) {
    unsigned long long* stamps = c->timers.stamps + 2 * (w * kTimerSlots + slot);
    c->step.start = stamps;
    c->step.stop = stamps + 1;
  }
  ~StepTimer() {
    ctx->step = Stamp{};
    ctx->timers.empty[which][slot] = launches == before || e != cudaSuccess;
    ctx->timers.in_pieces[which][slot] = 0;
    ++ctx->timers.used[which];
  }
};

// The same for a step that is launched in pieces, with other steps between them.  One record; empty unless all went well.
struct PieceTimer {
  litevggt_ctx* ctx;
  const int which, slot;
  int pieces = 0;
  const cudaError_t& e;
  PieceTimer(litevggt_ctx* c, int w, const cudaError_t& err) : ctx(c), which(w), slot(c->timers.used[w] % kTimerSlots), e(err) {}
  template <class Launch>
  cudaError_t piece(const Launch& launch) {
    unsigned long long* stamps = ctx->timers.pieces + 2 * (((which - kFirstInPieces) * kTimerSlots + slot) * kAttnCounters + pieces++);
    ctx->step.start = stamps;
    ctx->step.stop = stamps + 1;
    const cudaError_t result = launch();
    ctx->step = Stamp{};
    return result;
  }
  ~PieceTimer() {
    if (pieces == 0) return;  // as a step that was not come to
    ctx->timers.empty[which][slot] = e != cudaSuccess;
    ctx->timers.in_pieces[which][slot] = pieces;
    ++ctx->timers.used[which];
  }
};

inline litevggt_status cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return LITEVGGT_OK;
  (void)cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? LITEVGGT_ERR_ALLOC : LITEVGGT_ERR_CUDA;
}

// Two buffers of `rows` token rows in one allocation, whose address is the first one's; once per context.
inline litevggt_status ensure_row_pair(litevggt_ctx* ctx, long long rows, __nv_bfloat16** first, __nv_bfloat16** second) {
  if (*first != nullptr) return LITEVGGT_OK;
  DeviceGuard g(ctx->device);
  if (!g.ok) return LITEVGGT_ERR_CUDA;
  const size_t each = (size_t)round_up(rows * ctx->sz.dim * 2, 256);
  uint8_t* base = nullptr;
  if (cudaMalloc(&base, 2 * each) != cudaSuccess) {
    (void)cudaGetLastError();
    return LITEVGGT_ERR_ALLOC;
  }
  *first = reinterpret_cast<__nv_bfloat16*>(base);
  *second = reinterpret_cast<__nv_bfloat16*>(base + each);
  ctx->ws.bytes += 2 * each;
  return LITEVGGT_OK;
}
// The layer's input and output in merged rows, which both host entries use in the order of the caller's stream.
inline litevggt_status ensure_merged_staging(litevggt_ctx* ctx) {
  return ensure_row_pair(ctx, ctx->sz.n_merged, &ctx->ws.stage_xm, &ctx->ws.stage_ym);
}

// The key norms and value magnitudes of `sequences` sequences, which an output projection leaves zero for the next layer.
inline ZeroWords kmax_words(const litevggt_ctx* ctx, long long sequences) {
  return ZeroWords{reinterpret_cast<uint32_t*>(ctx->ws.attn_kmax), sequences * 2 * ctx->sz.heads};
}

// Before a call raises the key norms: they are zero unless an earlier call failed half-way.
inline cudaError_t begin_norms(litevggt_ctx* ctx, cudaStream_t s) {
  if (ctx->norms_left) {
    const cudaError_t e = cudaMemsetAsync(ctx->ws.attn_kmax, 0, sizeof(float) * (size_t)ctx->sz.frames * 2 * ctx->sz.heads, s);
    if (e != cudaSuccess) return e;
  }
  ctx->norms_left = true;  // until the output projection is enqueued
  return cudaSuccess;
}

// What the global layer's attention core needs to know about Q, K and V before it starts.
inline LinearStat core_stat(const litevggt_ctx* ctx, long long m) {
  LinearStat st;
  if (ctx->cfg.qkv_dtype == 1) {
    st.amax = ctx->ws.qkv_amax;
  } else {
    st.key_norm = ctx->ws.attn_kmax;
    st.seq_len = m;
  }
  return st;
}

}  // namespace lv

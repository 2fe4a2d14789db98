// The whole layer from and to host memory, call after call (litevggt_global_layer_host_pipelined): copies on the
// context's own streams, double-buffered staging, and an output that leaves while the layer still computes.
//
// Device to host is what such a pass waits for longest: 90 MB at 32 frames of 37 x 37 take 1.65 ms of PCIe behind 1.9
// ms of kernels.  A token's output needs one merged row, its own or its anchor's, so the attention runs in
// slabs of query rows, and when a slab has been projected a kernel on the copy stream adds its rows to their
// tokens' residuals and writes the tokens straight into the pinned buffer, under the next slab's
// attention: 3.72 -> 2.66 to 2.83 ms a pass.  What bounds it now is PCIe, both ways at once (the next call's input comes in
// meanwhile), at 45 GB/s out.  The first slab is one round of the attention's CTAs, so that PCIe starts early, the
// others two, which lose 3 % of a round at their end.  Output buffers that the device cannot write (pageable memory, odd
// addresses), E4M3 contexts, sequences of up to 4096 rows and some little longer ones (attn_slabs.h) and those of several key
// chunks, whose copies are 6 % of a pass or less, take the copy behind the layer.  So does a call with no drain since the one before: in a stream
// of calls a copy engine moves an output at 55 GB/s under the next call's kernels and takes nothing from them, while the
// writers do (40 calls in a row and a drain, ms a call: 16 frames of 37 x 37 1.00 by copies, 1.20 in slabs, 32 frames 2.14
// and 2.55, 44 frames 3.9 and 4.4; a call and its drain 2.22 and 1.98, 5.2 and 4.1, 7.9 and 6.3).  What a call does
// thus follows from the calls before it and not from how far the device has come: results repeat.
#include "host_common.h"

using namespace lv;

namespace {

// Copy streams, events and both pairs of [N, D] staging buffers of the pipelined host entry.  None of them is the ordered
// entry's: that one overwrites its own on the caller's stream, where nothing waits for what a pipelined call has left to
// the copy streams - and a wait for their events would not go into a graph that captures the ordered entry.
litevggt_status ensure_host_pipe(litevggt_ctx* ctx) {
  litevggt_status st = ensure_merged_staging(ctx);
  if (st != LITEVGGT_OK) return st;
  HostPipe& hp = ctx->pipe;
  if (hp.created) return LITEVGGT_OK;
  DeviceGuard g(ctx->device);
  if (!g.ok) return LITEVGGT_ERR_CUDA;
  const Sizes& z = ctx->sz;
  const size_t big = (size_t)round_up(z.n_tokens * z.dim * 2, 256);
  const size_t index = (size_t)(round_up(4 * z.n_tokens, 256) + 2 * round_up(4 * z.n_merged, 256) +
                                round_up(4 * (z.n_merged + 1), 256) + round_up(4 * (z.n_remove + 1), 256));
  const size_t stamps = sizeof(unsigned long long) * 2 * kStepsInPieces * kTimerSlots * kAttnCounters;
  if (cudaMalloc(&hp.base, 2 * (2 * big + index) + stamps) != cudaSuccess) {
    (void)cudaGetLastError();
    hp.base = nullptr;
    return LITEVGGT_ERR_ALLOC;
  }
  cudaError_t e = cudaStreamCreateWithFlags(&hp.copy_in, cudaStreamNonBlocking);
  // ahead of the next kernels on the caller's stream, which wait for an SM of their own while these fit beside what runs
  int least = 0, greatest = 0;
  if (e == cudaSuccess) e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
  if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&hp.copy_out, cudaStreamNonBlocking, greatest);
  cudaEvent_t* sets[4] = {hp.in_ready, hp.x_free, hp.out_ready, hp.out_free};
  for (int k = 0; k < 4 && e == cudaSuccess; ++k)
    for (int i = 0; i < 2 && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&sets[k][i], cudaEventDisableTiming);
  unsigned long long* pieces = reinterpret_cast<unsigned long long*>(hp.base + 2 * (2 * big + index));
  if (e == cudaSuccess) e = cudaMemsetAsync(pieces, 0, stamps, hp.copy_in);  // ahead of the input that all else waits for
  if (e != cudaSuccess) {
    // partial set-up is released at destroy time only if `created`; release it here instead
    if (hp.copy_in) cudaStreamDestroy(hp.copy_in);
    if (hp.copy_out) cudaStreamDestroy(hp.copy_out);
    for (int k = 0; k < 4; ++k)
      for (int i = 0; i < 2; ++i)
        if (sets[k][i]) cudaEventDestroy(sets[k][i]);
    cudaFree(hp.base);
    hp = HostPipe();
    return cuda_status(e);
  }
  for (int i = 0; i < 2; ++i) {
    uint8_t* slot = hp.base + i * (2 * big + index);
    hp.x[i] = reinterpret_cast<__nv_bfloat16*>(slot);
    hp.out[i] = reinterpret_cast<__nv_bfloat16*>(slot + big);
    hp.index[i] = reinterpret_cast<int*>(slot + 2 * big);
  }
  ctx->timers.pieces = pieces;
  ctx->ws.bytes += 2 * (2 * big + index) + stamps;
  hp.created = true;
  return LITEVGGT_OK;
}

// Where the device writes `bytes` of page-locked host memory, or nothing: one allocation or registration must hold them
// all (two that hold the ends may have pages between them that the device cannot reach), and 16-byte units must fit.
void* device_view(void* host, size_t bytes) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, host) != cudaSuccess) {
    (void)cudaGetLastError();
    return nullptr;
  }
  if (at.type != cudaMemoryTypeHost || at.devicePointer == nullptr || !aligned16(at.devicePointer)) return nullptr;
  const uint8_t *first = static_cast<const uint8_t*>(at.devicePointer), *begin = nullptr;
  size_t size = 0;
  if (!allocation_of(first, &begin, &size) || begin > first || (size_t)(first - begin) > size || size - (size_t)(first - begin) < bytes)
    return nullptr;
  return at.devicePointer;
}

// The attention layer and the unmerge in slabs of query rows, the finished tokens written to `out`.
cudaError_t layer_in_slabs(litevggt_ctx* ctx, const litevggt_plan* plan, int slot, const void* w_qkv, const void* b_qkv, const void* w_o, const void* b_o, __nv_bfloat16* out, cudaStream_t s,
                           bool* started) {
  const Sizes& z = ctx->sz;
  Workspace& ws = ctx->ws;
  HostPipe& hp = ctx->pipe;
  const long long m = z.n_merged;
  const int d = z.dim;
  int n = 0;
  cudaError_t e = begin_norms(ctx, s);
  if (e == cudaSuccess) {
    StepTimer t(ctx, 6, n, e);
    e = launch_linear_scaled(ctx, ws.stage_xm, m, d, static_cast<const __nv_bfloat16*>(w_qkv), 3 * d,
                             static_cast<const __nv_bfloat16*>(b_qkv), d, 2 * d, kKeyScaleLog2e, core_stat(ctx, m), ws.qkv, s, &n);
  }
  // this slot's rows and indices may still be on their way out, two calls ago
  if (e == cudaSuccess && hp.used[slot]) e = cudaStreamWaitEvent(s, hp.out_free[slot], 0);
  // the writers' own copy of the indices: the plan may be rebuilt as soon as this call has returned
  // (a plan's arrays lie in one allocation, in this order)
  const size_t index_bytes = reinterpret_cast<uint8_t*>(plan->seg_src + z.n_remove) - reinterpret_cast<uint8_t*>(plan->dst_of);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hp.index[slot], plan->dst_of, index_bytes, cudaMemcpyDeviceToDevice, s);
  auto copied = [&](const int* array) { return hp.index[slot] + (array - plan->dst_of); };
  __nv_bfloat16* ym = hp.out[slot];  // (the staged output is not needed: M <= N rows of it hold the merged ones)
  PieceTimer attention(ctx, 7, e), projection(ctx, 8, e), unmerge(ctx, 9, e);
  for (long long row0 = 0, row1; row0 < m && e == cudaSuccess; row0 = row1) {
    row1 = attention_slab_end(m, row0, ctx->num_sms, z.heads);
    e = attention.piece([&] { return launch_flash_attention_rows(ctx, ws.qkv, m, row0, row1, ws.attn_o, s, &n); });
    if (e == cudaSuccess)
      e = projection.piece([&] {
        return launch_linear(ctx, ws.attn_o + row0 * d, row1 - row0, d, static_cast<const __nv_bfloat16*>(w_o), d,
                             static_cast<const __nv_bfloat16*>(b_o), row1 == m ? kmax_words(ctx, 1) : ZeroWords{}, ym + row0 * d, s, &n);
      });
    if (e == cudaSuccess) e = cudaEventRecord(hp.out_ready[slot], s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(hp.copy_out, hp.out_ready[slot], 0);
    if (e == cudaSuccess) {
      e = unmerge.piece([&] {
        return launch_unmerge_rows(ctx, copied(plan->dst_of), copied(plan->kept_idx), copied(plan->seg_off), copied(plan->seg_src), ym,
                                   hp.x[slot], out, row0, row1, hp.copy_out, &n);
      });
      *started = true;
    }
  }
  if (e == cudaSuccess) ctx->norms_left = false;
  bump(ctx, n);
  return e;
}

}  // namespace

extern "C" {

litevggt_status litevggt_global_layer_host_pipelined(litevggt_ctx* ctx, litevggt_plan** plan_inout, const float* grad,
                                                     const void* x_host, const void* w_qkv, const void* b_qkv,
                                                     const void* w_o, const void* b_o, void* out_host, void* stream) {
  if (!ctx_ok(ctx) || plan_inout == nullptr || x_host == nullptr || out_host == nullptr) return LITEVGGT_ERR_NULL;
  if (grad == nullptr) {
    const litevggt_plan* plan = *plan_inout;
    if (!plan_ok(plan) || plan->owner != ctx || !plan->built) return LITEVGGT_ERR_STALE_PLAN;
  }
  litevggt_status st = ensure_host_pipe(ctx);
  if (st != LITEVGGT_OK) return st;
  DeviceGuard g(ctx->device);
  if (!g.ok) return LITEVGGT_ERR_CUDA;
  const Sizes& z = ctx->sz;
  Workspace& ws = ctx->ws;
  HostPipe& hp = ctx->pipe;
  cudaStream_t s = (cudaStream_t)stream;
  const size_t bytes = (size_t)z.n_tokens * z.dim * 2;
  const int slot = (int)(hp.calls & 1ull);
  // copy-in stream: the buffer is free once the unmerge two calls ago has read its residual from it
  cudaError_t e = cudaSuccess;
  if (hp.used[slot]) e = cudaStreamWaitEvent(hp.copy_in, hp.x_free[slot], 0);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hp.x[slot], x_host, bytes, cudaMemcpyHostToDevice, hp.copy_in);
  if (e == cudaSuccess) e = cudaEventRecord(hp.in_ready[slot], hp.copy_in);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(s, hp.in_ready[slot], 0);
  if (e != cudaSuccess) return cuda_status(e);
  if (grad != nullptr) {
    st = litevggt_merge_plan(ctx, hp.x[slot], grad, plan_inout, stream);
    if (st != LITEVGGT_OK) return st;
  }
  const litevggt_plan* plan = *plan_inout;
  st = litevggt_merge(ctx, plan, hp.x[slot], ws.stage_xm, stream);
  // In a stream of calls the copy of one hides behind the kernels of the next.
  const bool apart = hp.drained && ctx->cfg.qkv_dtype == 0 && attention_slabs_pay(z.n_merged, z.n_tokens, ctx->num_sms, z.heads);
  hp.drained = false;
  void* direct = st == LITEVGGT_OK && apart ? device_view(out_host, bytes) : nullptr;
  if (direct != nullptr) {
    bool started = false;
    // what a call's kernels check of their pointers; an argument they refuse stays refused
    if (w_qkv == nullptr || w_o == nullptr) return LITEVGGT_ERR_NULL;
    if (!aligned16(w_qkv) || !aligned16(w_o) || (b_qkv != nullptr && !aligned16(b_qkv)) || (b_o != nullptr && !aligned16(b_o)))
      return LITEVGGT_ERR_ALIGN;
    e = layer_in_slabs(ctx, plan, slot, w_qkv, b_qkv, w_o, b_o, static_cast<__nv_bfloat16*>(direct), s, &started);
    if (started) {  // also where a later launch failed: what has begun still uses the slot
      cudaError_t done = cudaEventRecord(hp.x_free[slot], hp.copy_out);
      if (done == cudaSuccess) done = cudaEventRecord(hp.out_free[slot], hp.copy_out);
      if (done == cudaSuccess) {
        hp.used[slot] = hp.in_slabs[slot] = true;
        ++hp.calls;
      }
      if (e == cudaSuccess) e = done;
    }
    return cuda_status(e);
  }
  if (st == LITEVGGT_OK)
    st = litevggt_global_attn(ctx, ws.stage_xm, z.n_merged, w_qkv, b_qkv, w_o, b_o, ws.stage_ym, stream);
  if (st != LITEVGGT_OK) return st;
  // the output buffer is free once the copy-out two calls ago has drained it
  if (hp.used[slot]) e = cudaStreamWaitEvent(s, hp.out_free[slot], 0);
  if (e != cudaSuccess) return cuda_status(e);
  st = litevggt_unmerge(ctx, plan, ws.stage_ym, hp.x[slot], hp.out[slot], stream);
  if (st != LITEVGGT_OK) return st;
  e = cudaEventRecord(hp.out_ready[slot], s);
  if (e == cudaSuccess) e = cudaEventRecord(hp.x_free[slot], s);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(hp.copy_out, hp.out_ready[slot], 0);
  if (e == cudaSuccess) e = cudaMemcpyAsync(out_host, hp.out[slot], bytes, cudaMemcpyDeviceToHost, hp.copy_out);
  if (e == cudaSuccess) e = cudaEventRecord(hp.out_free[slot], hp.copy_out);
  if (e == cudaSuccess) {
    hp.used[slot] = true;
    hp.in_slabs[slot] = false;
    ++hp.calls;
  }
  return cuda_status(e);
}

litevggt_status litevggt_host_drain(litevggt_ctx* ctx, void* stream) {
  if (!ctx_ok(ctx)) return LITEVGGT_ERR_NULL;
  HostPipe& hp = ctx->pipe;
  if (!hp.created) return LITEVGGT_OK;
  DeviceGuard g(ctx->device);
  if (!g.ok) return LITEVGGT_ERR_CUDA;
  cudaError_t e = cudaSuccess;
  for (int slot = 0; slot < 2 && e == cudaSuccess; ++slot)
    if (hp.used[slot]) e = cudaStreamWaitEvent((cudaStream_t)stream, hp.out_free[slot], 0);
  if (e == cudaSuccess) hp.drained = true;
  return cuda_status(e);
}

}  // extern "C"

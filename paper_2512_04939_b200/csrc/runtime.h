// Host-side runtime objects behind the C ABI: context (workspace, device status word,
// launch counter), plan (cached merge indices) and the launchers of each kernel group.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

#include "../../include/litevggt.h"
#include "attn_slabs.h"

namespace lv {

struct Sizes {
  int frames, grid_h, grid_w, n_special, dim, heads;
  int patches;        // P
  int tokens_frame;   // T
  long long n_tokens; // N
  int n_dst_frame, n_ga_frame, n_src_frame;
  long long n_src, n_dst;
  long long n_remove; // R
  long long n_merged; // M
};

inline long long round_up(long long v, long long a) { return (v + a - 1) / a * a; }

// Sets an attribute of a kernel once per device (`done` holds one bit per device, one object per kernel), so that
// a launcher's later calls only enqueue work.
inline cudaError_t set_attribute_once(const void* kernel, cudaFuncAttribute attribute, int value, std::atomic<unsigned long long>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, attribute, value);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}
inline cudaError_t set_max_dynamic_smem_once(const void* kernel, int bytes, std::atomic<unsigned long long>& done) {
  return set_attribute_once(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes, done);
}

// The attention kernels take the exponentials in base 2 of scores that already carry the softmax
// scale: 1/sqrt(64) log2(e) is folded into K where K is last rounded to bf16 (the QKV projection's
// epilogue, or the Q/K normalisation pass), so that no arithmetic stands between the tensor core's
// scores and the exponential, at no extra rounding.
constexpr float kKeyScaleLog2e = 0.125f * 1.4426950408889634f;

constexpr long long kMlpChunkRows = 131072;  // rows of the 4D-wide hidden activations held at a time (1 GiB)

// One device allocation carved into named regions.
struct Workspace {
  uint8_t* base = nullptr;
  size_t bytes = 0;
  // scoring
  float* var_map = nullptr;     // [F*P]
  float* ga_score = nullptr;    // [F*P]
  uint8_t* cls = nullptr;       // [N]
  int* src_list = nullptr;      // [|Src|] token index, ascending
  int* dst_list = nullptr;      // [|Dst|] token index, ascending
  // matching
  __nv_bfloat16* panel_src = nullptr;  // [|Src|, D] packed rows
  __nv_bfloat16* panel_dst = nullptr;  // [|Dst|, D]
  float* inv_norm_src = nullptr;       // [|Src|]
  float* inv_norm_dst = nullptr;       // [round_up(|Dst|,256)]
  unsigned long long* match_keys = nullptr;  // [|Src|] best (cosine, anchor) so far, as one ordered word
  // index build
  int* src_pos = nullptr;        // [N] a token's index in src_list, -1 for tokens of the other classes
  int* index_scratch = nullptr;  // keys, counts and the merged tokens on their way (index_build.cu)
  // attention
  __nv_bfloat16* qkv = nullptr;    // [M, 3D]
  __nv_bfloat16* attn_o = nullptr; // [M, D]
  float* attn_o_state = nullptr;   // [M, D] running output between key chunks (long sequences), or split parts
  float* attn_ml_state = nullptr;  // [M, heads, 4] references and partial row sums, or those of the parts
  int* attn_taken = nullptr;       // [kAttnCounters] jobs taken by an attention launch's CTAs; every Q/K/V projection zeroes them
  float* attn_kmax = nullptr;      // [max(frames, 1), 2, heads] largest |k|^2 and largest |v| per sequence and head
  // E4M3 variant of the attention operands (qkv_dtype = 1)
  uint8_t* q8 = nullptr;           // [M, D] bytes
  uint8_t* k8 = nullptr;           // [M, D] bytes
  uint8_t* v8t = nullptr;          // [D, round_up(M, 128)] bytes: V transposed, head-major rows
  float* qkv_amax = nullptr;       // [3, heads] largest magnitude of Q, K, V per head
  // whole-layer-from-host staging
  __nv_bfloat16* stage_x = nullptr;   // [N, D], the ordered entry's
  __nv_bfloat16* stage_out = nullptr; // [N, D], behind it
  __nv_bfloat16* stage_xm = nullptr;  // [M, D]
  __nv_bfloat16* stage_ym = nullptr;  // [M, D], behind it
  // block workspace of the frame-local attention and the MLP (allocated on first use)
  __nv_bfloat16* blk_qkv = nullptr;   // [N, 3D]
  __nv_bfloat16* blk_o = nullptr;     // [N, D]
  __nv_bfloat16* blk_hidden = nullptr; // [kMlpChunkRows, 4D]
  uint32_t* status = nullptr;         // device status word
};

}  // namespace lv

namespace lv {
// Where a kernel notes when it was on the device (common.cuh: Span).
struct Stamp {
  unsigned long long* start = nullptr;  // only the step's first kernel
  unsigned long long* stop = nullptr;   // every kernel of the step; the latest time stays
};
// Device-time stopwatches, one per step of the path: the times at which the step's kernels came
// and went, by the device's own clock, kept in a small ring per step.
constexpr int kNumTimers = 15;
constexpr int kTimerSlots = 64;
constexpr int kFirstInPieces = 7, kStepsInPieces = 3;  // attention core, output projection, unmerge
struct Timers {
  unsigned long long* stamps = nullptr;  // device [kNumTimers][kTimerSlots]{start, stop}, in the workspace
  int used[kNumTimers] = {};             // launches recorded since the last reset
  bool empty[kNumTimers][kTimerSlots] = {};  // the record's step launched nothing (or failed): its stamps are an older one's
  // A layer that leaves in slabs takes the steps from kFirstInPieces on in turns: stamps of every piece, of which a record
  // is the sum.
  unsigned long long* pieces = nullptr;  // device [kStepsInPieces][kTimerSlots][kAttnCounters]{start, stop}, with the host pipeline
  int in_pieces[kNumTimers][kTimerSlots] = {};  // pieces of a record, 0: it has stamps of its own
};
}  // namespace lv

// Streams, events and staging buffers behind litevggt_global_layer_host_pipelined.
struct HostPipe {
  bool created = false;
  cudaStream_t copy_in = nullptr, copy_out = nullptr;
  cudaEvent_t in_ready[2] = {}, x_free[2] = {}, out_ready[2] = {}, out_free[2] = {};
  bool used[2] = {false, false};
  bool in_slabs[2] = {false, false};            // the slot's last output was written by kernels on copy_out, until x_free
  bool drained = true;                          // nothing has been called since the last drain
  unsigned long long calls = 0;
  __nv_bfloat16* x[2] = {nullptr, nullptr};    // [N, D] each
  __nv_bfloat16* out[2] = {nullptr, nullptr};  // [N, D] each
  int* index[2] = {nullptr, nullptr};          // a plan's arrays, as a call found them
  uint8_t* base = nullptr;                      // allocation that holds them all
};

struct litevggt_ctx {
  uint32_t magic;
  litevggt_config cfg;
  lv::Sizes sz;
  int device;
  int num_sms;
  lv::Workspace ws;
  long long launches;
  void* encode_tiled;  // cuTensorMapEncodeTiled, resolved at run time
  lv::Timers timers;
  mutable lv::Stamp step;  // of the step whose kernels are being launched
  bool norms_left = false;  // a call that raised the key norms did not get as far as zeroing them
  HostPipe pipe;
};

struct litevggt_plan {
  uint32_t magic;
  const litevggt_ctx* owner;
  int built;
  int last_refresh_layer;
  bool has_maps;       // var/ga/best_* valid (plan built by the library's own scoring)
  uint8_t* base;       // one device allocation
  int* dst_of;         // [N]
  int* size;           // [M]
  int* kept_idx;       // [M]
  int* seg_off;        // [M+1]
  int* seg_src;        // [R]
  int* best_dst;       // [|Src|] anchor token index
  float* best_sim;     // [|Src|]
};

namespace lv {

// Enqueues a kernel of this library on `s`, `cluster` CTAs to a cluster.  With `overlap` and a grid of at most
// kOverlapBlocks blocks it may start before the kernel in front of it has ended - each calls
// wait_for_previous_kernel (common.cuh) before it touches memory, so what overlaps is launch latency and
// set-up: 288 -> 255 us for a block over seven frames, 116 -> 94 us for the first layer of four small
// ones.  Larger grids gain nothing by it, and asking costs their short blocks time (LayerNorm of 208 K
// rows: 145 -> 181 us).  The line, eight blocks on each of 148 SMs, is known to both sides of a launch.
constexpr long long kOverlapBlocks = 148 * 8;
template <class... P, class... A>
inline cudaError_t launch_clusters(int cluster, bool overlap, void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem,
                                   cudaStream_t s, A&&... args) {
  cudaLaunchAttribute attrs[2];
  unsigned n = 0;
  if (overlap && (long long)grid.x * grid.y * grid.z <= kOverlapBlocks) {
    attrs[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attrs[n].id = cudaLaunchAttributeClusterDimension;
    attrs[n].val.clusterDim.x = (unsigned)cluster;
    attrs[n].val.clusterDim.y = 1;
    attrs[n++].val.clusterDim.z = 1;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attrs;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<A&&>(args)...);
}
template <class... P, class... A>
inline cudaError_t launch(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s, A&&... args) {
  return launch_clusters(1, true, kernel, grid, threads, smem, s, static_cast<A&&>(args)...);
}

// The stamp of the step's next kernel.
inline Stamp next_stamp(const litevggt_ctx* ctx) {
  const Stamp s = ctx->step;
  ctx->step.start = nullptr;
  return s;
}

// bits of the device status word
constexpr uint32_t kStatusTimeout = 1u;
constexpr uint32_t kStatusBounds = 2u;

constexpr uint32_t kCtxMagic = 0x4c564358u;
constexpr uint32_t kPlanMagic = 0x4c56504cu;

// Words that a launch sets to zero for whoever comes after it.
struct ZeroWords {
  uint32_t* words = nullptr;
  long long count = 0;
};

// tensor_map.cu
bool resolve_encode_tiled(void** fn);
// The allocation or registration that an address which the device can use lies in.
bool allocation_of(const void* device_ptr, const uint8_t** begin, size_t* bytes);
// 2-D bf16 tensor [outer, inner] row-major with row pitch `pitch_elems`; box [box_outer, box_inner],
// 128-byte swizzle, zero fill outside the tensor.  A load brings 256 bytes of a row into L2, or, where what lies beside the box is
// not wanted before L2 has lost it (`box_alone`), 128.
bool make_tmap_bf16_2d(void* encode_fn, CUtensorMap* out, const void* base, uint64_t inner, uint64_t outer,
                       uint64_t pitch_elems, uint32_t box_inner, uint32_t box_outer, bool box_alone = false);
bool make_tmap_u8_2d(void* encode_fn, CUtensorMap* out, const void* base, uint64_t inner, uint64_t outer,
                     uint64_t pitch_bytes, uint32_t box_inner, uint32_t box_outer);

// scoring.cu
cudaError_t launch_grad_map(const litevggt_ctx* ctx, const float* images, float* grad, cudaStream_t s, int* launches);
cudaError_t launch_var_map(const litevggt_ctx* ctx, const __nv_bfloat16* x, float* var,
                           cudaStream_t s, int* launches);
cudaError_t launch_partition(const litevggt_ctx* ctx, const float* grad, const float* var, float* ga, uint8_t* cls,
                             cudaStream_t s, int* launches);
// (the partition leaves the token lists behind as well; this is for classes that come from the caller)
cudaError_t launch_build_lists(const litevggt_ctx* ctx, const uint8_t* cls, cudaStream_t s, int* launches);

// similarity.cu: leaves every src row's best anchor in ctx->ws.match_keys
cudaError_t launch_match(litevggt_ctx* ctx, const __nv_bfloat16* x, cudaStream_t s, int* launches);

// index_build.cu
cudaError_t launch_index_build(litevggt_ctx* ctx, litevggt_plan* plan, cudaStream_t s, int* launches);
long long index_scratch_words(const Sizes& z);
// the part of the scratch array that has to be zero before launch_index_build; the matching sees to it
ZeroWords index_zero_words(const litevggt_ctx* ctx);

// merge_unmerge.cu
cudaError_t launch_merge(const litevggt_ctx* ctx, const litevggt_plan* plan, const __nv_bfloat16* x,
                         __nv_bfloat16* xm, cudaStream_t s, int* launches);
cudaError_t launch_unmerge(const litevggt_ctx* ctx, const litevggt_plan* plan, const __nv_bfloat16* ym,
                           const __nv_bfloat16* residual, __nv_bfloat16* out, cudaStream_t s, int* launches);
// merged rows [row0, row1) to all tokens that they stand for, residual added: out may be host memory.  The index arrays are
// a plan's; the blocks fit beside the attention kernel's.
cudaError_t launch_unmerge_rows(const litevggt_ctx* ctx, const int* dst_of, const int* kept_idx, const int* seg_off,
                                const int* seg_src, const __nv_bfloat16* ym, const __nv_bfloat16* residual, __nv_bfloat16* out,
                                long long row0, long long row1, cudaStream_t s, int* launches);

// linear.cu
cudaError_t launch_linear(litevggt_ctx* ctx, const __nv_bfloat16* a, long long m, long long k, const __nv_bfloat16* w,
                          long long n, const __nv_bfloat16* bias, const ZeroWords& zero, __nv_bfloat16* out, cudaStream_t s,
                          int* launches);
// The same with output columns [scale_begin, scale_end) (multiples of 64) multiplied by `scale` in
// fp32 before the one rounding to bf16: the QKV projection of an attention layer scales its K columns.
// It also leaves behind one of two statistics
// of the rounded output.  Zeroing the key norms takes no launch: they are zero between calls, because
// the output projection, which runs after their last reader, leaves them so.
struct LinearStat {
  float* key_norm = nullptr;  // [sequences, 2, heads] largest |k|^2 over the columns [scale_begin, scale_end) and largest |v| ...
  long long seq_len = 0;      // ... of sequences of this many rows
  float* amax = nullptr;      // [n / 64] largest magnitude of every 64 columns, zeroed here first
  bool values_only = false;   // of key_norm only |v|: a later pass rounds K
};
cudaError_t launch_linear_scaled(litevggt_ctx* ctx, const __nv_bfloat16* a, long long m, long long k,
                                 const __nv_bfloat16* w, long long n, const __nv_bfloat16* bias, int scale_begin,
                                 int scale_end, float scale, const LinearStat& stat, __nv_bfloat16* out, cudaStream_t s,
                                 int* launches);

cudaError_t launch_linear_mlp(litevggt_ctx* ctx, const __nv_bfloat16* a, long long m, long long k,
                              const __nv_bfloat16* w, long long n, const __nv_bfloat16* bias, int gelu,
                              const __nv_bfloat16* residual, const ZeroWords& zero, __nv_bfloat16* out, cudaStream_t s,
                              int* launches);
cudaError_t launch_layernorm(const __nv_bfloat16* x, const __nv_bfloat16* gamma, const __nv_bfloat16* beta,
                             __nv_bfloat16* out, long long rows, float eps, const Stamp& stamp, cudaStream_t s,
                             int* launches);

// selftest.cu: one CTA waits on a barrier that nobody arrives on, with the given cycle limit
cudaError_t launch_bounded_wait_selftest(litevggt_ctx* ctx, long long limit_cycles, uint32_t* outcome, cudaStream_t s,
                                         int* launches);

// attention.cu
// n_seq independent sequences of seq_len rows each, laid back to back in qkv / o
// qk_embed.cu: optional per-head LayerNorm and 2-D rotary embedding of Q and K, in place on [m, 3D]
cudaError_t launch_qk_embed(const litevggt_ctx* ctx, __nv_bfloat16* qkv, const int* kept_idx, long long m,
                            const __nv_bfloat16* q_gamma, const __nv_bfloat16* q_beta, const __nv_bfloat16* k_gamma,
                            const __nv_bfloat16* k_beta, float eps, int rope, float rope_base, float* key_norm,
                            cudaStream_t s, int* launches);
// ctx->ws.attn_kmax holds the largest |k|^2 per sequence and head (left there by whichever pass rounded
// K last: the projection or qk_embed) and the largest |v| (by the projection)
cudaError_t launch_flash_attention(litevggt_ctx* ctx, const __nv_bfloat16* qkv, long long seq_len, int n_seq,
                                   __nv_bfloat16* o, cudaStream_t s, int* launches);
// The same for a slab of the one sequence's m query rows: rows [row0, row1) with row1 = attention_slab_end(row0).
cudaError_t launch_flash_attention_rows(litevggt_ctx* ctx, const __nv_bfloat16* qkv, long long m, long long row0, long long row1,
                                        __nv_bfloat16* o, cudaStream_t s, int* launches);
size_t attention_state_bytes(long long m, int dim, int heads, int num_sms, size_t* ml_offset);
// E4M3 variant: quantised copies of Q, K, V by the per-head magnitudes in ctx->ws.qkv_amax - taken from
// qkv here first unless the projection has left them there - (fp8_quant.cu), then the attention core on
// those (attention.cu); one sequence of m rows
cudaError_t launch_qkv_quantize(litevggt_ctx* ctx, const __nv_bfloat16* qkv, long long m, bool have_amax, cudaStream_t s,
                                int* launches);
cudaError_t launch_flash_attention_fp8(litevggt_ctx* ctx, long long m, __nv_bfloat16* o, cudaStream_t s, int* launches);

}  // namespace lv

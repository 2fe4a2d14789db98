// Stand-ins for the CUDA runtime and for the kernel launchers, so that the host side of the library (api.cu,
// attn_static.cu) can be linked and driven without a GPU.  "Device" memory is host memory; launchers only
// do what the host code can see: count, note, and fail where the test asks for it.
#include <stdlib.h>
#include <string.h>

#include <functional>
#include <vector>

#include "../paper_2512_04939_b200/csrc/runtime.h"

using namespace lv;

static int g_fail_linear = 0;         // this many of the next output projections are refused
static float g_norm_seen = 0.0f;      // key norm of the first head before the latest projection raised it
static float g_norm_last_seen = 0.0f; // and of the last sequence
extern "C" void fake_fail_linear(int n) { g_fail_linear = n; }
extern "C" float fake_norm_seen() { return g_norm_seen; }
extern "C" float fake_norm_last_seen() { return g_norm_last_seen; }
// cudaMemset goes to the default stream and returns before it has run; nothing but a synchronisation orders it
// before work on a non-blocking stream.
static std::vector<std::function<void()>> g_default_stream;
static void finish_default_stream() {
  for (auto& f : g_default_stream) f();
  g_default_stream.clear();
}
extern "C" int fake_default_stream_pending() { return (int)g_default_stream.size(); }

// ---- CUDA runtime
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  memset(p, 0, sizeof(*p));
  p->major = 10;
  p->multiProcessorCount = 148;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : 148;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { return (*p = calloc(n, 1)) != nullptr ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { g_default_stream.push_back([=] { memset(p, v, n); }); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  finish_default_stream();
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { finish_default_stream(); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  if (s == nullptr) finish_default_stream();
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = reinterpret_cast<cudaStream_t>(64); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) { *p = const_cast<void*>(symbol); return cudaSuccess; }
}

// ---- launchers
namespace lv {
static unsigned long long g_clock = 1000;
static cudaError_t ran(const litevggt_ctx* ctx, int* launches) {  // one kernel of 500 ns
  const Stamp s = next_stamp(ctx);
  if (s.start != nullptr) *s.start = g_clock;
  g_clock += 500;
  if (s.stop != nullptr && *s.stop < g_clock) *s.stop = g_clock;
  ++*launches;
  return cudaSuccess;
}
static void zero_words(const ZeroWords& z) { if (z.count > 0) memset(z.words, 0, (size_t)z.count * 4); }

bool resolve_encode_tiled(void** fn) { *fn = reinterpret_cast<void*>(1); return true; }
long long index_scratch_words(const Sizes&) { return 1; }
size_t attention_state_bytes(long long, int, int, int, size_t* ml) { *ml = 0; return 0; }
cudaError_t launch_grad_map(const litevggt_ctx* c, const float*, float*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_var_map(const litevggt_ctx* c, const __nv_bfloat16*, float*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_partition(const litevggt_ctx* c, const float*, const float*, float*, uint8_t*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_build_lists(const litevggt_ctx* c, const uint8_t*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_match(litevggt_ctx* c, const __nv_bfloat16*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_index_build(litevggt_ctx* c, litevggt_plan*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_merge(const litevggt_ctx* c, const litevggt_plan*, const __nv_bfloat16*, __nv_bfloat16*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_unmerge(const litevggt_ctx* c, const litevggt_plan*, const __nv_bfloat16*, const __nv_bfloat16*, __nv_bfloat16*,
                           cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_linear_scaled(litevggt_ctx* c, const __nv_bfloat16*, long long m, long long, const __nv_bfloat16*, long long,
                                 const __nv_bfloat16*, int, int, float, const LinearStat& st, __nv_bfloat16*, cudaStream_t, int* n) {
  if (st.key_norm != nullptr) {  // raises every norm to 4, as an atomic maximum would
    const long long words = m / st.seq_len * 16;
    g_norm_seen = st.key_norm[0];
    g_norm_last_seen = st.key_norm[words - 1];
    for (long long i = 0; i < words; ++i) st.key_norm[i] = st.key_norm[i] > 4.0f ? st.key_norm[i] : 4.0f;
  }
  return ran(c, n);
}
static cudaError_t output_projection(litevggt_ctx* c, const ZeroWords& z, int* n) {
  if (g_fail_linear > 0) {
    --g_fail_linear;
    return cudaErrorInvalidValue;
  }
  zero_words(z);
  return ran(c, n);
}
cudaError_t launch_linear(litevggt_ctx* c, const __nv_bfloat16*, long long, long long, const __nv_bfloat16*, long long,
                          const __nv_bfloat16*, const ZeroWords& z, __nv_bfloat16*, cudaStream_t, int* n) {
  return output_projection(c, z, n);
}
cudaError_t launch_linear_mlp(litevggt_ctx* c, const __nv_bfloat16*, long long, long long, const __nv_bfloat16*, long long,
                              const __nv_bfloat16*, int, const __nv_bfloat16*, const ZeroWords& z, __nv_bfloat16*, cudaStream_t,
                              int* n) {
  return output_projection(c, z, n);
}
cudaError_t launch_layernorm(const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*, __nv_bfloat16*, long long rows, float,
                             const Stamp& s, cudaStream_t, int* n) {
  if (rows == 0) return cudaSuccess;
  *s.start = g_clock;
  *s.stop = g_clock += 500;
  ++*n;
  return cudaSuccess;
}
cudaError_t launch_bounded_wait_selftest(litevggt_ctx* c, long long, uint32_t*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_qk_embed(const litevggt_ctx* c, __nv_bfloat16*, const int*, long long, const __nv_bfloat16* g, const __nv_bfloat16*,
                            const __nv_bfloat16*, const __nv_bfloat16*, float, int rope, float, float*, cudaStream_t, int* n) {
  return g == nullptr && !rope ? cudaSuccess : ran(c, n);
}
cudaError_t launch_flash_attention(litevggt_ctx* c, const __nv_bfloat16*, long long, int, __nv_bfloat16*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_qkv_quantize(litevggt_ctx* c, const __nv_bfloat16*, long long, bool, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_flash_attention_fp8(litevggt_ctx* c, long long, __nv_bfloat16*, cudaStream_t, int* n) { return ran(c, n); }
}  // namespace lv

// Stand-ins for the CUDA runtime and for the kernel launchers, so that the host side of the library (api.cu,
// attn_static.cu, host_pipeline.cu) can be linked and driven without a GPU.  "Device" memory is host memory; launchers only
// do what the host code can see: count, note, and fail where the test asks for it.
#include <stdlib.h>
#include <string.h>

#include <functional>
#include <map>
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

// Which memory the work on a stream touches, and what of it nothing orders: a vector clock per stream, joined
// where a stream waits for an event and where the host has waited for a stream.
using Clock = std::map<const void*, long>;
struct Access {
  const char *begin, *end;
  bool writes;
  const void* stream;
  long time;
};
static std::map<const void*, Clock> g_stream_clocks;
static std::map<const void*, Clock> g_events;
static Clock g_host_clock;
static std::vector<Access> g_accesses;
static int g_races = 0;
static void join(Clock& to, const Clock& from) {
  for (const auto& c : from)
    if (to[c.first] < c.second) to[c.first] = c.second;
}
static Clock& clock_of(cudaStream_t s) {
  Clock& c = g_stream_clocks[s];
  join(c, g_host_clock);
  return c;
}
struct Range {
  const void* p;
  long long bytes;
};
static void touch(cudaStream_t s, std::vector<Range> reads, std::vector<Range> writes) {
  Clock& now = clock_of(s);
  const long time = ++now[s];
  for (int w = 0; w < 2; ++w)
    for (const Range& r : w ? writes : reads) {
      if (r.p == nullptr || r.bytes <= 0) continue;
      const Access a{static_cast<const char*>(r.p), static_cast<const char*>(r.p) + r.bytes, w == 1, s, time};
      for (const Access& b : g_accesses)
        if (b.begin < a.end && a.begin < b.end && (a.writes || b.writes) && now[b.stream] < b.time) ++g_races;
      g_accesses.push_back(a);
    }
}
// Page-locked host memory: all of it, unless a test says which.
static const Range kAll{nullptr, 1ll << 62};
static std::vector<Range> g_locked;
static const Range* page_locked(const void* p) {
  for (const Range& r : g_locked)
    if (p >= r.p && p < static_cast<const char*>(r.p) + r.bytes) return &r;
  return g_locked.empty() ? &kAll : nullptr;
}
static int g_rows_written = 0;  // launches that write rows to their tokens in host memory
extern "C" void fake_page_lock(const void* p, long long bytes) { g_locked.push_back({p, bytes}); }
extern "C" void fake_page_lock_all() { g_locked.clear(); }
extern "C" long long fake_slab_end(long long m, long long row0, int sms) { return attention_slab_end(m, row0, sms, 16); }
extern "C" int fake_slab_index(long long row0, int sms) { return attention_slab_index(row0, sms, 16); }
static int g_sms = 148;
extern "C" void fake_sms(int n) { g_sms = n; }
extern "C" int fake_rows_written() { return g_rows_written; }
extern "C" int fake_races() { return g_races; }
extern "C" void fake_forget_accesses() {
  g_stream_clocks.clear();
  g_events.clear();
  g_host_clock.clear();
  g_accesses.clear();
  g_races = 0;
}

// ---- CUDA runtime
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  memset(p, 0, sizeof(*p));
  p->major = 10;
  p->multiProcessorCount = g_sms;
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
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t stream) {
  touch(stream, {{s, (long long)n}}, {{d, (long long)n}});
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  finish_default_stream();
  for (const auto& c : g_stream_clocks) join(g_host_clock, c.second);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  if (s == nullptr) finish_default_stream();
  join(g_host_clock, clock_of(s));
  return cudaSuccess;
}
static long long g_handles = 64;  // streams and events
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = reinterpret_cast<cudaStream_t>(g_handles++); return cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { return cudaStreamCreateWithFlags(s, 0); }
cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest) { *least = 0; *greatest = -5; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  join(clock_of(s), g_events[e]);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(g_handles++); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  g_events[e] = clock_of(s);
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof(*a));
  a->hostPointer = const_cast<void*>(p);
  if (page_locked(p) == nullptr) return cudaSuccess;
  a->type = cudaMemoryTypeHost;
  a->devicePointer = a->hostPointer;
  return cudaSuccess;
}
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
bool allocation_of(const void* p, const uint8_t** begin, size_t* bytes) {
  const Range* r = page_locked(p);
  if (r == nullptr) return false;
  *begin = static_cast<const uint8_t*>(r->p);
  *bytes = (size_t)r->bytes;
  return true;
}
long long index_scratch_words(const Sizes&) { return 1; }
size_t attention_state_bytes(long long, int, int, int, size_t* ml) { *ml = 0; return 0; }
cudaError_t launch_grad_map(const litevggt_ctx* c, const float*, float*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_var_map(const litevggt_ctx* c, const __nv_bfloat16*, float*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_partition(const litevggt_ctx* c, const float*, const float*, float*, uint8_t*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_build_lists(const litevggt_ctx* c, const uint8_t*, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_match(litevggt_ctx* c, const __nv_bfloat16*, cudaStream_t, int* n) { return ran(c, n); }
static Range rows(const void* p, long long n) { return {p, n * 1024 * 2}; }
cudaError_t launch_index_build(litevggt_ctx* c, litevggt_plan* p, cudaStream_t s, int* n) {
  const Sizes& z = c->sz;
  touch(s, {}, {{p->dst_of, 4 * z.n_tokens}, {p->kept_idx, 4 * z.n_merged}, {p->seg_off, 4 * (z.n_merged + 1)}, {p->seg_src, 4 * z.n_remove}});
  return ran(c, n);
}
cudaError_t launch_merge(const litevggt_ctx* c, const litevggt_plan* p, const __nv_bfloat16* x, __nv_bfloat16* xm, cudaStream_t s, int* n) {
  touch(s, {rows(x, c->sz.n_tokens), {p->kept_idx, 4 * c->sz.n_merged}}, {rows(xm, c->sz.n_merged)});
  return ran(c, n);
}
cudaError_t launch_unmerge(const litevggt_ctx* c, const litevggt_plan* p, const __nv_bfloat16* ym, const __nv_bfloat16* res, __nv_bfloat16* out,
                           cudaStream_t s, int* n) {
  touch(s, {rows(ym, c->sz.n_merged), rows(res, c->sz.n_tokens), {p->dst_of, 4 * c->sz.n_tokens}}, {rows(out, c->sz.n_tokens)});
  return ran(c, n);
}
cudaError_t launch_unmerge_rows(const litevggt_ctx* c, const int* dst_of, const int* kept, const int* off, const int* src, const __nv_bfloat16* ym,
                                const __nv_bfloat16* res, __nv_bfloat16* out, long long row0, long long row1, cudaStream_t s, int* n) {
  const Sizes& z = c->sz;
  ++g_rows_written;
  touch(s, {rows(ym + row0 * 1024, row1 - row0), rows(res, z.n_tokens), {dst_of, 4 * z.n_tokens}, {kept, 4 * z.n_merged}, {off, 4 * (z.n_merged + 1)},
            {src, 4 * z.n_remove}}, {rows(out, z.n_tokens), {c->ws.status, 4}});  // (its bounds checks)
  return ran(c, n);
}
cudaError_t launch_linear_scaled(litevggt_ctx* c, const __nv_bfloat16* a, long long m, long long, const __nv_bfloat16*, long long,
                                 const __nv_bfloat16*, int, int, float, const LinearStat& st, __nv_bfloat16* out, cudaStream_t s, int* n) {
  touch(s, {rows(a, m)}, {rows(out, 3 * m)});
  if (st.key_norm != nullptr) {  // raises every norm and value to 4, as an atomic maximum would
    const long long words = m / st.seq_len * 2 * 16;
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
cudaError_t launch_linear(litevggt_ctx* c, const __nv_bfloat16* a, long long m, long long, const __nv_bfloat16*, long long,
                          const __nv_bfloat16*, const ZeroWords& z, __nv_bfloat16* out, cudaStream_t s, int* n) {
  touch(s, {rows(a, m)}, {rows(out, m)});
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
cudaError_t launch_flash_attention(litevggt_ctx* c, const __nv_bfloat16* qkv, long long m, int n_seq, __nv_bfloat16* o, cudaStream_t s, int* n) {
  touch(s, {rows(qkv, 3 * m * n_seq)}, {rows(o, m * n_seq)});
  return ran(c, n);
}
cudaError_t launch_flash_attention_rows(litevggt_ctx* c, const __nv_bfloat16* qkv, long long m, long long row0, long long row1, __nv_bfloat16* o,
                                        cudaStream_t s, int* n) {
  touch(s, {rows(qkv, 3 * m)}, {rows(o + row0 * 1024, row1 - row0)});
  return ran(c, n);
}
cudaError_t launch_qkv_quantize(litevggt_ctx* c, const __nv_bfloat16*, long long, bool, cudaStream_t, int* n) { return ran(c, n); }
cudaError_t launch_flash_attention_fp8(litevggt_ctx* c, long long, __nv_bfloat16*, cudaStream_t, int* n) { return ran(c, n); }
}  // namespace lv

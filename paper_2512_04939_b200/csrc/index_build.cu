// Selection of the src tokens to merge and construction of the cached index arrays.
//
// Inputs: per src token (ascending token order) its best anchor and cosine.  The R most
// similar src tokens are merged (ties towards the lower token index); every other token
// keeps its own row, rows follow ascending token order.  Outputs: dst_of[N], size[M],
// kept_idx[M] and a CSR (seg_off[M+1], seg_src[R]) listing, per merged row, the absorbed
// src tokens in ascending token order - the order the merge kernel sums them in.
//
// Everything here is integer work on ~1 M elements, bound by launches and latency, so the aim is few
// passes and no sort:
//   select    the R-th largest cosine by its ordered bits, 11 + 11 + 10 of them at a time: histogram,
//             then every block of the next pass finds the bin that holds the R-th for itself;
//   number    one scan over the tokens counts those above the threshold and those equal to it
//             before each token; both the row of a kept token and the rank of a merged one follow;
//   group     merged tokens count into their rows (the count's old value is a slot), a scan over the
//             rows gives the segments, each token goes to its slot and then to its rank among its
//             segment's tokens.  Which slot a token got depends on scheduling, its rank does not.
// Ten launches, or - up to kSmallTokens tokens, where a launch costs more than what it does -
// one launch of one block.  The two bitonic sorts of 64-bit keys that came before took 92 launches at 200
// frames of 28 x 37 (418 us, 77 now) and 23 at four of 16 x 16 (82 us; 19 now, 50 as ten launches, events included).
// No host synchronisation: all counts follow from the config.
#include "common.cuh"
#include "runtime.h"

namespace lv {

constexpr int kIdxThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanChunk = kIdxThreads * kScanItems;  // <= 4 Mi elements in <= 1024 blocks, whose sums one block can add
constexpr int kSelBins = 2048;
// A token's rank in a segment of up to this many tokens comes from comparing it with each of them, at
// most R x 1024 loads; longer ones, of which there are at most R / 1024, each take a block that walks
// over all R merged tokens in order.
constexpr int kLongSegment = 1024;
constexpr int kLongBlocks = 148;
constexpr long long kSmallTokens = 8192;

// bits [shift, shift + bits) of a key select its bin in pass 0, 1, 2
__host__ __device__ constexpr int sel_shift(int pass) { return pass == 0 ? 21 : pass == 1 ? 10 : 0; }
__host__ __device__ constexpr int sel_bins(int pass) { return pass == 2 ? 1024 : 2048; }

__device__ __forceinline__ unsigned sim_bits(float f) {  // monotone float -> unsigned
  const unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Inclusive scan over the block's threads; scratch holds one value per warp.
template <class T>
__device__ __forceinline__ T block_scan_inclusive(T v, T* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  __syncthreads();
  if (lane == 31) scratch[warp] = v;
  __syncthreads();
  if (warp == 0) {
    T w = scratch[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T t = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += t;
    }
    scratch[lane] = w;
  }
  __syncthreads();
  return warp > 0 ? v + scratch[warp - 1] : v;
}

// The selection so far: keys above `prefix` (its fixed high bits) are in, `need` more come from those
// that share it.
struct Selection {
  unsigned prefix;
  unsigned need;
};

// Everything the phases read and write.  No pointer is __restrict__: one phase reads what an earlier one
// wrote, in the same launch where one block runs them all.
struct IndexArgs {
  const unsigned long long* match_key;  // [|Src|] the matching's result
  const int* dst_list;
  const float* inv_norm_src;
  const int* src_pos;                   // [N]
  int* best_dst;                        // [|Src|]
  float* best_sim;                      // [|Src|]
  int *dst_of, *size, *kept_idx, *seg_off, *seg_src;
  unsigned* hist;                       // 3 histograms of kSelBins
  Selection* sel;                       // [3] the selection after every pass
  unsigned long long* token_sums;       // per block of kScanChunk tokens
  int* row_sums;                        // per block of kScanChunk rows
  unsigned* key;                        // [|Src|] ordered bits of best_sim
  int* long_rows;                       // [0] number of long segments, then their rows
  int* count;                           // [M] merged tokens of a row
  int *rem_token, *rem_anchor, *rem_row, *rem_slot, *seg_tmp;  // [R] merged tokens; tokens by slot
  long long n_src, n_dst, n_tokens, n_merged, n_remove;
  uint32_t* status;
  Stamp stamp;
};

// Fixes the bits of pass `pass` from its histogram.  Called by a whole block of kIdxThreads threads.
template <int pass>
__device__ __forceinline__ Selection select_bin(const unsigned* hist, Selection before) {
  __shared__ unsigned scratch[32];
  __shared__ Selection found;
  constexpr int bins = sel_bins(pass), per = bins / kIdxThreads;
  unsigned c[per], sum = 0;
#pragma unroll
  for (int i = 0; i < per; ++i) {  // from the highest bin downwards
    c[i] = hist[bins - 1 - (threadIdx.x * per + i)];
    sum += c[i];
  }
  unsigned above = block_scan_inclusive(sum, scratch) - sum;
#pragma unroll
  for (int i = 0; i < per; ++i) {
    if (above < before.need && above + c[i] >= before.need) {
      found.prefix = before.prefix | ((unsigned)(bins - 1 - (threadIdx.x * per + i)) << sel_shift(pass));
      found.need = before.need - above;
    }
    above += c[i];
  }
  __syncthreads();
  return found;
}

// Adds 1 to hist[bin] for the lanes with `on`; cosines crowd into few bins, so equal ones go together.
__device__ __forceinline__ void hist_add(unsigned* hist, unsigned bin, bool on) {
  const unsigned active = __ballot_sync(0xffffffffu, on);
  if (on) {
    const unsigned same = __match_any_sync(active, bin);
    if ((threadIdx.x & 31) == (unsigned)(__ffs(same) - 1)) atomicAdd(&hist[bin], (unsigned)__popc(same));
  }
}

// ---- the phases; block `block` of `blocks`, kIdxThreads threads each

// Pass 0 also takes the matching's keys apart: anchor token and cosine of every src row.
template <int pass>
__device__ __forceinline__ void phase_select(int block, int blocks, const IndexArgs& a) {
  __shared__ unsigned bins[kSelBins];
  const bool selects = a.n_remove < a.n_src;  // else all are merged
  if (selects)
    for (int i = threadIdx.x; i < kSelBins; i += kIdxThreads) bins[i] = 0u;
  Selection so_far{0u, (unsigned)a.n_remove};
  if constexpr (pass > 0) {
    if constexpr (pass == 2) so_far = a.sel[0];
    so_far = select_bin<pass - 1>(a.hist + (pass - 1) * kSelBins, so_far);
    if (block == 0 && threadIdx.x == 0) a.sel[pass - 1] = so_far;
  }
  __syncthreads();
  for (long long base = (long long)block * kIdxThreads; base < a.n_src; base += (long long)blocks * kIdxThreads) {
    const long long i = base + threadIdx.x;
    unsigned k = 0;
    bool on = i < a.n_src;
    if (on) {
      if constexpr (pass == 0) {
        const unsigned long long mk = a.match_key[i];
        unsigned col = ~(unsigned)mk;
        if (col >= a.n_dst) {
          atomicOr(a.status, kStatusBounds);
          col = 0;
        }
        const unsigned v = (unsigned)(mk >> 32);  // the cosine before the src row's own norm, as ordered bits
        const float sim = __uint_as_float((v & 0x80000000u) ? (v & 0x7fffffffu) : ~v) * a.inv_norm_src[i];
        a.best_dst[i] = a.dst_list[col];
        a.best_sim[i] = sim;
        k = sim_bits(sim);
        a.key[i] = k;
      } else {
        k = a.key[i];
        on = (k >> sel_shift(pass - 1)) == (so_far.prefix >> sel_shift(pass - 1));
      }
    }
    if (selects) hist_add(bins, (k >> sel_shift(pass)) & (unsigned)(sel_bins(pass) - 1), on);
  }
  if (!selects) return;
  __syncthreads();
  for (int i = threadIdx.x; i < sel_bins(pass); i += kIdxThreads)
    if (bins[i] != 0u) atomicAdd(&a.hist[pass * kSelBins + i], bins[i]);
}

// Tokens above the threshold (low word) and equal to it (high word) among a thread's kScanItems.
__device__ __forceinline__ unsigned long long token_counts(const IndexArgs& a, unsigned threshold, long long base,
                                                           int (&pos)[kScanItems], unsigned long long (&c)[kScanItems]) {
  unsigned long long sum = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    pos[i] = base + i < a.n_tokens ? a.src_pos[base + i] : -1;
    c[i] = 0ull;
    if (pos[i] >= 0) {
      const unsigned k = a.key[pos[i]];
      c[i] = k > threshold ? 1ull : k == threshold ? 1ull << 32 : 0ull;
    }
    sum += c[i];
  }
  return sum;
}

// With every src token merged the threshold lies below all keys.  Called by a whole block.
__device__ __forceinline__ Selection selection_after_histograms(const IndexArgs& a) {
  return a.n_remove == a.n_src ? Selection{0u, (unsigned)a.n_src} : select_bin<2>(a.hist + 2 * kSelBins, a.sel[1]);
}

// Threshold (from the last histogram) and the counts of every block of tokens.
__device__ __forceinline__ void phase_count_removed(int block, const IndexArgs& a) {
  __shared__ unsigned long long scratch[32];
  const Selection s = selection_after_histograms(a);
  if (block == 0 && threadIdx.x == 0) a.sel[2] = s;
  int pos[kScanItems];
  unsigned long long c[kScanItems];
  const long long base = (long long)block * kScanChunk + (long long)threadIdx.x * kScanItems;
  const unsigned long long incl = block_scan_inclusive(token_counts(a, s.prefix, base, pos, c), scratch);
  if (threadIdx.x == kIdxThreads - 1) a.token_sums[block] = incl;
}

// Sum of the first `count` (<= kIdxThreads) block sums, in every thread.
template <class T>
__device__ __forceinline__ T sum_of_blocks_before(const T* block_sums, int count, T* scratch) {
  __shared__ T total;
  const T incl = block_scan_inclusive((int)threadIdx.x < count ? block_sums[threadIdx.x] : T(0), scratch);
  if (threadIdx.x == kIdxThreads - 1) total = incl;
  __syncthreads();
  return total;
}

// Rows of the kept tokens, and the merged tokens with their anchors in ascending token order.  With
// n_remove = 0 every token is kept.
__device__ __forceinline__ void phase_number_tokens(int block, const IndexArgs& a) {
  __shared__ unsigned long long scratch[32];
  const long long base = (long long)block * kScanChunk + (long long)threadIdx.x * kScanItems;
  int pos[kScanItems];
  unsigned long long c[kScanItems], before = 0;
  unsigned need = 0;
  if (a.n_remove > 0) {
    const Selection s = a.sel[2];
    need = s.need;
    const unsigned long long prefix = block > 0 ? sum_of_blocks_before(a.token_sums, block, scratch) : 0ull;
    const unsigned long long sum = token_counts(a, s.prefix, base, pos, c);
    before = prefix + block_scan_inclusive(sum, scratch) - sum;
  } else {
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) c[i] = 0ull;
  }
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i >= a.n_tokens) break;
    const unsigned above = (unsigned)before, equal = (unsigned)(before >> 32);
    const long long removed = (long long)above + (equal < need ? equal : need);
    if ((unsigned)c[i] != 0u || ((unsigned)(c[i] >> 32) != 0u && equal < need)) {
      if (removed < a.n_remove) {
        a.rem_token[removed] = (int)(base + i);
        a.rem_anchor[removed] = a.best_dst[pos[i]];
      }
    } else {
      const long long row = base + i - removed;
      if (row < a.n_merged) {
        a.dst_of[base + i] = (int)row;
        a.kept_idx[row] = (int)(base + i);
      } else {
        atomicOr(a.status, kStatusBounds);
      }
    }
    before += c[i];
  }
}

// Merged tokens take their anchor's row and a slot in it.
__device__ __forceinline__ void phase_assign_removed(int block, const IndexArgs& a) {
  const long long i = (long long)block * kIdxThreads + threadIdx.x;
  if (i >= a.n_remove) return;
  const int token = a.rem_token[i], anchor = a.rem_anchor[i];
  int row = anchor >= 0 && anchor < a.n_tokens ? a.dst_of[anchor] : -1;
  if (token < 0 || token >= a.n_tokens || row < 0 || row >= a.n_merged) {
    atomicOr(a.status, kStatusBounds);
    row = 0;
  } else {
    a.dst_of[token] = row;
  }
  a.rem_row[i] = row;
  a.rem_slot[i] = atomicAdd(&a.count[row], 1);
}

__device__ __forceinline__ void phase_row_sums(int block, const IndexArgs& a) {
  __shared__ int scratch[32];
  const long long base = (long long)block * kScanChunk + (long long)threadIdx.x * kScanItems;
  int sum = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) sum += base + i < a.n_merged ? a.count[base + i] : 0;
  const int incl = block_scan_inclusive(sum, scratch);
  if (threadIdx.x == kIdxThreads - 1) a.row_sums[block] = incl;
}

// Row sizes, segment offsets and the list of long segments.
__device__ __forceinline__ void phase_segments(int block, const IndexArgs& a) {
  __shared__ int scratch[32];
  const long long base = (long long)block * kScanChunk + (long long)threadIdx.x * kScanItems;
  const int prefix = block > 0 ? sum_of_blocks_before(a.row_sums, block, scratch) : 0;
  int c[kScanItems], sum = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    c[i] = base + i < a.n_merged ? a.count[base + i] : 0;
    sum += c[i];
  }
  int off = prefix + block_scan_inclusive(sum, scratch) - sum;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i >= a.n_merged) break;
    a.size[base + i] = 1 + c[i];
    a.seg_off[base + i] = off;
    if (c[i] > kLongSegment) a.long_rows[1 + atomicAdd(&a.long_rows[0], 1)] = (int)(base + i);
    off += c[i];
    if (base + i == a.n_merged - 1) a.seg_off[a.n_merged] = (int)a.n_remove;
  }
}

__device__ __forceinline__ void phase_slot_tokens(int block, const IndexArgs& a) {
  const long long i = (long long)block * kIdxThreads + threadIdx.x;
  if (i < a.n_remove) a.seg_tmp[a.seg_off[a.rem_row[i]] + a.rem_slot[i]] = a.rem_token[i];
}

// A thread per merged token: its rank among its segment's tokens.
__device__ __forceinline__ void phase_rank(int block, const IndexArgs& a) {
  const long long i = (long long)block * kIdxThreads + threadIdx.x;
  if (i >= a.n_remove) return;
  const int row = a.rem_row[i], len = a.count[row];
  if (len > kLongSegment) return;
  const int token = a.rem_token[i], off = a.seg_off[row];
  int rank = 0;
  for (int k = 0; k < len; ++k) rank += a.seg_tmp[off + k] < token ? 1 : 0;
  a.seg_src[off + rank] = token;
}

// A block per long segment: all merged tokens in order, those of the segment's row in the order met.
__device__ __forceinline__ void phase_long_segments(int block, int blocks, const IndexArgs& a) {
  __shared__ int scratch[32];
  __shared__ int met;
  const int n_long = a.long_rows[0];
  for (int l = block; l < n_long; l += blocks) {
    const int row = a.long_rows[1 + l];
    int at = a.seg_off[row];
    for (long long base = 0; base < a.n_remove; base += kIdxThreads) {
      const bool mine = base + threadIdx.x < a.n_remove && a.rem_row[base + threadIdx.x] == row;
      const int incl = block_scan_inclusive(mine ? 1 : 0, scratch);
      if (mine) a.seg_src[at + incl - 1] = a.rem_token[base + threadIdx.x];
      if (threadIdx.x == kIdxThreads - 1) met = incl;
      __syncthreads();
      at += met;
      __syncthreads();
    }
  }
}

enum Phase { kSelect0, kSelect1, kSelect2, kCountRemoved, kNumberTokens, kAssignRemoved, kRowSums, kSegments, kSlotTokens, kOrder };

template <int phase>
__device__ __forceinline__ void run_phase(int block, int blocks, const IndexArgs& a) {
  if constexpr (phase == kSelect0) phase_select<0>(block, blocks, a);
  if constexpr (phase == kSelect1) phase_select<1>(block, blocks, a);
  if constexpr (phase == kSelect2) phase_select<2>(block, blocks, a);
  if constexpr (phase == kCountRemoved) phase_count_removed(block, a);
  if constexpr (phase == kNumberTokens) phase_number_tokens(block, a);
  if constexpr (phase == kAssignRemoved) phase_assign_removed(block, a);
  if constexpr (phase == kRowSums) phase_row_sums(block, a);
  if constexpr (phase == kSegments) phase_segments(block, a);
  if constexpr (phase == kSlotTokens) phase_slot_tokens(block, a);
  if constexpr (phase == kOrder) {
    const int rank_blocks = (int)((a.n_remove + kIdxThreads - 1) / kIdxThreads);
    if (block < rank_blocks) phase_rank(block, a);
    else phase_long_segments(block - rank_blocks, blocks - rank_blocks, a);
  }
}

// Blocks of a phase; 0: nothing to do.
static __host__ __device__ inline int phase_blocks(int phase, const IndexArgs& a, int select_blocks) {
  auto per = [](long long n, int each) { return (int)((n + each - 1) / each); };
  const bool merges = a.n_remove > 0;
  if (phase == kSelect0) return a.n_src > 0 ? select_blocks : 0;
  if (phase == kNumberTokens) return per(a.n_tokens, kScanChunk);
  if (phase == kRowSums || phase == kSegments) return per(a.n_merged, kScanChunk);
  if (!merges) return 0;
  if (phase == kSelect1 || phase == kSelect2) return a.n_remove == a.n_src ? 0 : select_blocks;  // all of them: nothing to select
  if (phase == kCountRemoved) return per(a.n_tokens, kScanChunk);
  return per(a.n_remove, kIdxThreads) + (phase == kOrder && a.n_remove > kLongSegment ? (select_blocks > 1 ? kLongBlocks : 1) : 0);
}

template <int phase>
__global__ void __launch_bounds__(kIdxThreads) index_phase_kernel(const IndexArgs a) {
  const Span span(a.stamp);
  run_phase<phase>(blockIdx.x, gridDim.x, a);
}

// All phases in one block: what the blocks of a launch would do, one block after the other.  Sums over blocks that come before
// are not asked for where there is one, nor histograms where every src token is merged (four frames of 16 x 16: 8.3 us,
// 11.0 with both); the threshold, which counting the tokens leaves behind, is.
template <int phase>
__device__ __forceinline__ void run_phases_from(const IndexArgs& a) {
  const int blocks = phase_blocks(phase, a, 1);
  if (phase == kCountRemoved && blocks == 1) {
    const Selection s = selection_after_histograms(a);
    if (threadIdx.x == 0) a.sel[2] = s;
    __syncthreads();
  } else if (phase != kRowSums || blocks > 1) {
    for (int b = 0; b < blocks; ++b) {
      run_phase<phase>(b, blocks, a);
      __syncthreads();
    }
  }
  if constexpr (phase < kOrder) run_phases_from<phase + 1>(a);
}
__global__ void __launch_bounds__(kIdxThreads, 1) index_small_kernel(const IndexArgs a, int* zeroed, int zeroed_words) {
  const Span span(a.stamp);
  // (the histograms come first)
  for (int i = threadIdx.x + (a.n_remove < a.n_src ? 0 : 3 * kSelBins); i < zeroed_words; i += kIdxThreads) zeroed[i] = 0;
  __syncthreads();
  run_phases_from<kSelect0>(a);
}

template <int phase>
static cudaError_t launch_phases_from(const litevggt_ctx* ctx, IndexArgs& a, int select_blocks, cudaStream_t s, int* launches) {
  const int blocks = phase_blocks(phase, a, select_blocks);
  if (blocks > 0) {
    a.stamp = next_stamp(ctx);
    const cudaError_t e = launch(index_phase_kernel<phase>, dim3((unsigned)blocks), kIdxThreads, 0, s, a);
    if (e != cudaSuccess) return e;
    ++*launches;
  }
  if constexpr (phase < kOrder) return launch_phases_from<phase + 1>(ctx, a, select_blocks, s, launches);
  return cudaSuccess;
}

// [ 3 histograms | long segments: count, rows | merged tokens per row ], first in the scratch array and zero
// when a plan's build starts
static long long zero_words(const Sizes& z) { return 3 * kSelBins + 1 + z.n_remove / kLongSegment + 1 + z.n_merged; }

// Words of the index build's scratch array.
long long index_scratch_words(const Sizes& z) {
  return round_up(zero_words(z), 4) + 8 + 2 * kIdxThreads + kIdxThreads + round_up(z.n_src, 4) + 5 * round_up(z.n_remove, 4);
}

ZeroWords index_zero_words(const litevggt_ctx* ctx) {
  if (ctx->sz.n_tokens <= kSmallTokens) return ZeroWords{};  // the single block does it
  return ZeroWords{reinterpret_cast<uint32_t*>(ctx->ws.index_scratch), zero_words(ctx->sz)};
}

cudaError_t launch_index_build(litevggt_ctx* ctx, litevggt_plan* plan, cudaStream_t s, int* launches) {
  const Sizes& z = ctx->sz;
  Workspace& ws = ctx->ws;
  const long long r = z.n_remove;
  int* w = ws.index_scratch;
  auto take = [&w](long long words) {
    int* p = w;
    w += words;
    return p;
  };
  IndexArgs a;
  a.match_key = ws.match_keys;
  a.dst_list = ws.dst_list;
  a.inv_norm_src = ws.inv_norm_src;
  a.src_pos = ws.src_pos;
  a.best_dst = plan->best_dst;
  a.best_sim = plan->best_sim;
  a.dst_of = plan->dst_of;
  a.size = plan->size;
  a.kept_idx = plan->kept_idx;
  a.seg_off = plan->seg_off;
  a.seg_src = plan->seg_src;
  const long long zeroed = zero_words(z);
  int* zero = take(round_up(zeroed, 4));
  a.hist = reinterpret_cast<unsigned*>(zero);
  a.long_rows = zero + 3 * kSelBins;
  a.count = a.long_rows + 1 + r / kLongSegment + 1;
  a.sel = reinterpret_cast<Selection*>(take(8));
  a.token_sums = reinterpret_cast<unsigned long long*>(take(2 * kIdxThreads));
  a.row_sums = take(kIdxThreads);
  a.key = reinterpret_cast<unsigned*>(take(round_up(z.n_src, 4)));
  a.rem_token = take(round_up(r, 4));
  a.rem_anchor = take(round_up(r, 4));
  a.rem_row = take(round_up(r, 4));
  a.rem_slot = take(round_up(r, 4));
  a.seg_tmp = take(round_up(r, 4));
  a.n_src = z.n_src;
  a.n_dst = z.n_dst;
  a.n_tokens = z.n_tokens;
  a.n_merged = z.n_merged;
  a.n_remove = r;
  a.status = ws.status;
  if (z.n_tokens <= kSmallTokens) {
    a.stamp = next_stamp(ctx);
    ++*launches;
    return launch(index_small_kernel, dim3(1), kIdxThreads, 0, s, a, zero, (int)zeroed);
  }
  if (z.n_src == 0) {  // no matching ran
    cudaError_t e = cudaMemsetAsync(zero, 0, (size_t)zeroed * 4, s);
    if (e != cudaSuccess) return e;
  }
  // at most as many blocks as run at a time, and at least two (one means the single-block kernel): each
  // flushes a histogram
  long long select_blocks = (z.n_src + 4 * kIdxThreads - 1) / (4 * kIdxThreads);
  if (select_blocks > 2 * ctx->num_sms) select_blocks = 2 * ctx->num_sms;
  if (select_blocks < 2) select_blocks = 2;
  return launch_phases_from<kSelect0>(ctx, a, (int)select_blocks, s, launches);
}

}  // namespace lv

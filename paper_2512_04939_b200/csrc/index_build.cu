// Selection of the src tokens to merge and construction of the cached index arrays.
//
// Inputs: per src token (ascending token order) its best anchor and cosine.  The R most
// similar src tokens are merged (ties towards the lower token index); every other token
// keeps its own row, rows follow ascending token order.  Outputs: dst_of[N], size[M],
// kept_idx[M] and a CSR (seg_off[M+1], seg_src[R]) listing, per merged row, the absorbed
// src tokens in ascending token order - the order the merge kernel sums them in.
//
// Everything here is integer work on at most ~1 M elements, bound by latency: dependent loads and the
// steps that need the whole of the step before.  So there is no sort, and what used to be boundaries between launches (4.3 us
// each, of which there were ten) are barriers (0.7 us) of one cluster of blocks, each with a run of the src tokens (and the
// tokens from its first to the next block's first) and a run of the rows.  A short sequence is the work of one block
// that holds in its shared memory what one step hands to the next (four frames of 16 x 16: 9.7 us, 5 so); in a long one the
// steps behind the numbers of its tokens are launches over the chip, in a very long one all are.  (launch_index_build has the figures.)
//   select    the R-th largest cosine by its ordered bits, eight of them at a time: every block makes a
//             histogram of its own keys in shared memory, and after a barrier adds up those of all blocks
//             and finds the bin that holds the R-th for itself.  What the histograms of the blocks before it hold
//             over and at the threshold is all that a block needs to number its tokens;
//   number    one scan over the block's tokens, from there on: the row of a kept token, the place
//             of a merged one;
//   group     merged tokens count into their rows (the count's old value is a slot), a scan over the
//             rows gives the segments, each token goes to its slot and then to its rank among its
//             segment's tokens.  Which slot a token got depends on scheduling, its rank does not.
#include "common.cuh"
#include "runtime.h"

namespace lv {

// Every step ends in scans and barriers whose instructions all warps issue, so fewer are sooner through: a block of 512 threads where
// it has few tokens (577 tokens in one block 31.0 us, 32.0 with 1024, 3,360 50.4, 51.4, 56.3 with 256), 1024 where it has many.
constexpr int kIdxThreads = 512;
constexpr int kIdxWideThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kSelBins = 256;
constexpr int kSelPasses = 4;
constexpr int kIdxMaxBlocks = 16, kIdxPortableBlocks = 8;  // of a cluster
constexpr int kIdxParts = 128;     // runs of rows of a long sequence
// Sequences of more tokens than this are numbered by launches over the chip too, their keys selected 11 + 11 + 10 bits at a
// time by histograms in global memory: what the cluster's 16 SMs do for all tokens grows beyond five launches (index build, us,
// cluster / launches: 66,624 tokens 36 / 44, 189,000 58 / 45, 208,200 67 / 45, 1,041,000 238 / 77).
constexpr long long kManyTokens = 98304;
constexpr int kLongBins = 2048, kLongThreads = 1024, kLongChunk = kLongThreads * kScanItems;  // <= 4 Mi tokens in <= 1024 chunks
// A token's rank in a segment of up to this many tokens comes from comparing it with each of them, at
// most R x 1024 loads; longer ones, of which there are at most R / 1024, each take a block that walks
// over all R merged tokens in order.
constexpr int kLongSegment = 1024;
constexpr int kLongBlocks = 148;

__host__ __device__ constexpr int sel_shift(int pass) { return 24 - 8 * pass; }  // of the bits that select a key's bin in pass 0 to 3

__device__ __forceinline__ unsigned sim_bits(float f) {  // monotone float -> unsigned
  const unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ int threads() { return (int)blockDim.x; }

// Inclusive scan over the block's threads; scratch holds one value per warp, in the end the sums up to and with it.
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
    T w = lane < threads() / 32 ? scratch[lane] : T(0);
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
// that share it.  Of the keys of the blocks before this one, `above` are over it and (after the last pass) `equal` at it.
struct Selection {
  unsigned prefix, need, above, equal;
};

// Everything the steps read and write.  No pointer is __restrict__: one step reads what an earlier one
// wrote, in the same launch.
struct IndexArgs {
  const unsigned long long* match_key;  // [|Src|] the matching's result
  const int *src_list, *dst_list;
  const float* inv_norm_src;
  const int* src_pos;                   // [N]
  int* best_dst;                        // [|Src|]
  float* best_sim;                      // [|Src|]
  int *dst_of, *size, *kept_idx, *seg_off, *seg_src;
  unsigned* key;                        // [|Src|] ordered bits of best_sim
  int* long_rows;                       // [0] number of long segments, then their rows
  int* count;                           // [M] merged tokens of a row
  int* part_sums;                       // [kIdxParts] merged tokens by run of rows, where the steps are launches
  unsigned* hist;                       // [3][kLongBins], zero when the build of a very long sequence starts
  Selection* sel;                       // [3] its selection after every pass
  unsigned long long* token_sums;       // its counts of every kLongChunk tokens
  int *rem_token, *rem_anchor, *rem_row, *rem_slot, *seg_tmp;  // [R] merged tokens; tokens by slot
  int *row_of, *offset, *anchor_of;     // dst_of, seg_off and best_dst, for reading: copies where the block keeps such in shared memory
  long long n_src, n_dst, n_tokens, n_merged, n_remove;
  uint32_t* status;
  Stamp stamp;
  __host__ __device__ bool selects() const { return n_remove > 0 && n_remove < n_src; }  // else none or all are merged
};

// Lays what the steps hand on over `words`: [ long segments: count, rows | merged tokens per row | keys | five words a merged
// token ], and the copies of what they read back where `copies`.  Returns the words it takes.
__host__ __device__ inline long long lay_scratch(IndexArgs& a, int* words, bool copies) {
  long long at = 0;
  auto take = [&](long long count) {
    int* p = words + at;
    at += (count + 3) / 4 * 4;
    return p;
  };
  a.long_rows = take(1 + a.n_remove / kLongSegment + 1);
  a.count = take(a.n_merged);
  a.part_sums = take(kIdxParts);
  a.hist = reinterpret_cast<unsigned*>(take(a.n_tokens > kManyTokens ? 3 * kLongBins : 0));
  a.sel = reinterpret_cast<Selection*>(take(a.n_tokens > kManyTokens ? 3 * 4 : 0));
  a.token_sums = reinterpret_cast<unsigned long long*>(take(a.n_tokens > kManyTokens ? 2 * (a.n_tokens / kLongChunk + 1) : 0));
  a.key = reinterpret_cast<unsigned*>(take(a.n_src));
  a.rem_token = take(a.n_remove);
  a.rem_anchor = take(a.n_remove);
  a.rem_row = take(a.n_remove);
  a.rem_slot = take(a.n_remove);
  a.seg_tmp = take(a.n_remove);
  a.row_of = copies ? take(a.n_tokens) : a.dst_of;
  a.offset = copies ? take(a.n_merged) : a.seg_off;
  a.anchor_of = copies ? take(a.n_src) : a.best_dst;
  return at;
}

// Shared memory that the other blocks of the cluster read.
struct IndexShared {
  alignas(16) unsigned hist[kSelPasses][kSelBins];
  unsigned part[kIdxMaxBlocks];  // this block's merged tokens by the block that has their row
};

__device__ __forceinline__ unsigned ld_cluster(uint32_t addr) {
  unsigned v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

// Fixes the bits of pass `pass` from the histograms of all blocks.  `sums` [kSelBins] serves one pass.
template <int pass, bool kLocal>
__device__ __forceinline__ Selection select_bin(const unsigned* hist, uint2* sums, int block, int blocks, const Selection& before) {
  constexpr int per = kSelBins / 32;
  if (threadIdx.x < kSelBins) {
    const uint32_t at = smem_u32(hist + threadIdx.x);
    uint2 sum = make_uint2(kLocal ? hist[threadIdx.x] : 0u, 0u);  // of all blocks, of those before this one
    int q = block;  // every block starts with another one, or all would queue up for the first one's memory
#pragma unroll 16
    for (int i = 0; i < (kLocal ? 0 : blocks); ++i) {
      const unsigned v = ld_cluster(mapa_u32(at, q));
      sum.x += v;
      sum.y += q < block ? v : 0u;
      q = q + 1 == blocks ? 0 : q + 1;
    }
    sums[threadIdx.x % per * 32 + threadIdx.x / per] = sum;  // (so that lanes read side by side)
  }
  __syncthreads();
  // every warp finds the bin for itself, a lane looks at eight, lane 31 at the lowest
  const int lane = threadIdx.x & 31, top = kSelBins - 1 - lane * per;
  uint2 c[per];
  unsigned all = 0;
#pragma unroll
  for (int i = 0; i < per; ++i) {
    c[i] = sums[(per - 1 - i) * 32 + 31 - lane];
    all += c[i].x;
  }
  unsigned over = all;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, over, o);
    if (lane >= o) over += t;
  }
  const int owner = __ffs(__ballot_sync(0xffffffffu, over >= before.need)) - 1;  // the highest bins that reach it
  over -= all;
  unsigned mine = 0, bin = 0, need = 0, equal = 0;  // mine: over the bin, of the blocks before this one
  bool found = false;
#pragma unroll
  for (int i = 0; i < per; ++i) {
    if (!found && (lane < owner || over + c[i].x < before.need)) mine += lane <= owner ? c[i].y : 0u;
    if (lane == owner && !found && over + c[i].x >= before.need) {
      found = true;
      bin = (unsigned)(top - i);
      need = before.need - over;
      equal = c[i].y;
    }
    over += c[i].x;
  }
  return Selection{before.prefix | __shfl_sync(0xffffffffu, bin, owner) << sel_shift(pass), __shfl_sync(0xffffffffu, need, owner),
                   before.above + __reduce_add_sync(0xffffffffu, mine), __shfl_sync(0xffffffffu, equal, owner)};
}

template <bool kLocal>
__device__ __forceinline__ void all_blocks() {
  if constexpr (kLocal) {
    __syncthreads();
  } else {
    __syncwarp();  // the barrier wants whole warps
    cluster_sync();
  }
}

// Adds 1 to hist[bin] for the lanes with `on`; cosines crowd into few bins, so equal ones go together.
__device__ __forceinline__ void hist_add(unsigned* hist, unsigned bin, bool on) {
  const unsigned active = __ballot_sync(0xffffffffu, on);
  if (on) {
    const unsigned same = __match_any_sync(active, bin);
    if ((threadIdx.x & 31) == (unsigned)(__ffs(same) - 1)) atomicAdd(&hist[bin], (unsigned)__popc(same));
  }
}

// The matching's key of src token i taken apart into anchor token and cosine, whose ordered bits it returns.
template <bool kLocal>
__device__ __forceinline__ unsigned take_match(const IndexArgs& a, int i, unsigned long long match, float inv_norm) {
  unsigned col = ~(unsigned)match;
  if (col >= a.n_dst) {
    atomicOr(a.status, kStatusBounds);
    col = 0;
  }
  const unsigned v = (unsigned)(match >> 32);  // the cosine before the src row's own norm, as ordered bits
  const float sim = __uint_as_float((v & 0x80000000u) ? (v & 0x7fffffffu) : ~v) * inv_norm;
  const int anchor = a.dst_list[col];
  a.best_dst[i] = anchor;
  if constexpr (kLocal) a.anchor_of[i] = anchor;
  a.best_sim[i] = sim;
  return a.key[i] = sim_bits(sim);
}

// The block's src tokens [p0, p1): the matching's keys taken apart into anchor token and cosine, whose ordered bits a thread
// holds for its first kHeld tokens and finds in memory for others; and the first histogram.
constexpr int kHeld = 4;
template <bool kLocal>
__device__ __forceinline__ void read_matches(const IndexArgs& a, int p0, int p1, bool selects, unsigned* hist, unsigned (&held)[kHeld]) {
  for (int base = p0; base < p1; base += kHeld * threads()) {
    unsigned long long match[kHeld];
    float inv_norm[kHeld];
#pragma unroll
    for (int j = 0; j < kHeld; ++j) {
      const int i = base + j * threads() + (int)threadIdx.x;
      match[j] = i < p1 ? a.match_key[i] : 0ull;
      inv_norm[j] = i < p1 ? a.inv_norm_src[i] : 0.0f;
    }
#pragma unroll
    for (int j = 0; j < kHeld; ++j) {
      const int first = base + j * threads(), i = first + (int)threadIdx.x;
      if (first >= p1) break;
      const unsigned k = i < p1 ? take_match<kLocal>(a, i, match[j], inv_norm[j]) : 0u;
      if (base == p0) held[j] = k;
      if (selects) hist_add(hist, k >> sel_shift(0), i < p1);
    }
  }
}
// The histogram of pass `pass` over the keys whose higher bits are the selection's.
template <int pass>
__device__ __forceinline__ void count_keys(const IndexArgs& a, int p0, int p1, const Selection& so_far, unsigned* hist,
                                           const unsigned (&held)[kHeld]) {
  auto count = [&](unsigned k, bool on) {
    hist_add(hist, (k >> sel_shift(pass)) & (unsigned)(kSelBins - 1),
             on && (k >> sel_shift(pass - 1)) == (so_far.prefix >> sel_shift(pass - 1)));
  };
#pragma unroll
  for (int j = 0; j < kHeld; ++j)
    if (p0 + j * threads() < p1) count(held[j], p0 + j * threads() + (int)threadIdx.x < p1);
  for (int base = p0 + kHeld * threads(); base < p1; base += kHeld * threads()) {
    unsigned k[kHeld];
#pragma unroll
    for (int j = 0; j < kHeld; ++j) {
      const int i = base + j * threads() + (int)threadIdx.x;
      k[j] = i < p1 ? a.key[i] : 0u;
    }
#pragma unroll
    for (int j = 0; j < kHeld; ++j)
      if (base + j * threads() < p1) count(k[j], base + j * threads() + (int)threadIdx.x < p1);
  }
}

// A thread's tokens of the block's chunk that starts at `chunk`: their places among the src tokens (-1: none, or none is merged)
// and keys.
struct TokenKeys {
  int pos[kScanItems];
  unsigned key[kScanItems];
  __device__ __forceinline__ void load_places(const IndexArgs& a, int chunk, int t1) {
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
      const int t = chunk + (int)threadIdx.x * kScanItems + i;
      pos[i] = t < t1 && a.n_remove > 0 ? a.src_pos[t] : -1;
    }
  }
  __device__ __forceinline__ void load_keys(const IndexArgs& a) {
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) key[i] = pos[i] >= 0 ? a.key[pos[i]] : 0u;
  }
};
// Rows of the block's kept tokens, and its merged tokens with their anchors, in ascending token order.  `before`: the
// keys of the blocks before it that are over (low word) and at (high word) the threshold.  `next` holds the first chunk.
template <bool kLocal>
__device__ __forceinline__ void number_tokens(const IndexArgs& a, int t0, int t1, unsigned threshold, unsigned need,
                                              unsigned long long before, TokenKeys& next) {
  __shared__ unsigned long long scratch[32];
  for (int chunk = t0; chunk < t1; chunk += threads() * kScanItems) {
    int p[kScanItems];
    unsigned long long c[kScanItems], sum = 0ull;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
      p[i] = next.pos[i];
      c[i] = p[i] < 0 ? 0ull : next.key[i] > threshold ? 1ull : next.key[i] == threshold ? 1ull << 32 : 0ull;
      sum += c[i];
    }
    if (chunk + threads() * kScanItems < t1) {  // on their way while these are scanned
      next.load_places(a, chunk + threads() * kScanItems, t1);
      next.load_keys(a);
    }
    unsigned long long at = before + block_scan_inclusive(sum, scratch) - sum;
    before += scratch[31];
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
      const int t = chunk + (int)threadIdx.x * kScanItems + i;
      if (t >= t1) break;
      const unsigned above = (unsigned)at, equal = (unsigned)(at >> 32);
      const long long removed = (long long)above + (equal < need ? equal : need);
      if ((unsigned)c[i] != 0u || ((unsigned)(c[i] >> 32) != 0u && equal < need)) {
        if (removed < a.n_remove) {
          a.rem_token[removed] = t;
          a.rem_anchor[removed] = a.anchor_of[p[i]];
        }
      } else {
        const long long row = t - removed;
        if (row >= 0 && row < a.n_merged) {
          a.dst_of[t] = (int)row;
          if constexpr (kLocal) a.row_of[t] = (int)row;
          a.kept_idx[row] = t;
        } else {
          atomicOr(a.status, kStatusBounds);
        }
      }
      at += c[i];
    }
  }
}

// Merged tokens take their anchor's row and a slot in it, kItems at a time, each being a chain of loads: two in a cluster, one where
// the threads of a launch are enough for all (1,099,200 random tokens: 20.4 us, two at a time 28.5).
template <int kItems>
__device__ __forceinline__ void assign_removed(int block, int blocks, const IndexArgs& a, int rows_per_block, unsigned* part) {
  const int stride = blocks * threads();
  for (int i0 = block * threads() + (int)threadIdx.x; i0 < a.n_remove; i0 += kItems * stride) {
    int token[kItems], anchor[kItems], row[kItems];
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const bool on = i0 + j * stride < a.n_remove;
      token[j] = on ? a.rem_token[i0 + j * stride] : -1;
      anchor[j] = on ? a.rem_anchor[i0 + j * stride] : -1;
    }
#pragma unroll
    for (int j = 0; j < kItems; ++j) row[j] = anchor[j] >= 0 && anchor[j] < a.n_tokens ? a.row_of[anchor[j]] : -1;
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const int i = i0 + j * stride;
      if (i >= a.n_remove) break;
      if (token[j] < 0 || token[j] >= a.n_tokens || row[j] < 0 || row[j] >= a.n_merged) {
        atomicOr(a.status, kStatusBounds);
        row[j] = 0;
      } else {
        a.dst_of[token[j]] = row[j];
      }
      a.rem_row[i] = row[j];
      a.rem_slot[i] = atomicAdd(&a.count[row[j]], 1);
      atomicAdd(&part[row[j] / rows_per_block], 1u);
    }
  }
}

// Sizes, segment offsets and the list of long segments, of rows [r0, r1); rows_before() merged tokens have rows before them.
template <bool kLocal, class Before>
__device__ __forceinline__ void lay_segments(const IndexArgs& a, int r0, int r1, const Before& rows_before) {
  __shared__ int scratch[32];
  int c[kScanItems], off = 0;
  auto load = [&](int chunk) {
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
      const int r = chunk + (int)threadIdx.x * kScanItems + i;
      c[i] = r < r1 ? a.count[r] : 0;
    }
  };
  load(r0);
  off = rows_before();
  for (int chunk = r0; chunk < r1; chunk += threads() * kScanItems) {
    const int base = chunk + (int)threadIdx.x * kScanItems;
    int n[kScanItems], sum = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
      n[i] = c[i];
      sum += n[i];
    }
    if (chunk + threads() * kScanItems < r1) load(chunk + threads() * kScanItems);
    int at = off + block_scan_inclusive(sum, scratch) - sum;
    off += scratch[31];
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
      if (base + i >= r1) break;
      a.size[base + i] = 1 + n[i];
      a.seg_off[base + i] = at;
      if constexpr (kLocal) a.offset[base + i] = at;
      if (n[i] > kLongSegment) a.long_rows[1 + atomicAdd(&a.long_rows[0], 1)] = base + i;
      at += n[i];
      if (base + i == a.n_merged - 1) a.seg_off[a.n_merged] = (int)a.n_remove;
    }
  }
}

__device__ __forceinline__ void slot_token(int i, const IndexArgs& a) {
  a.seg_tmp[a.offset[a.rem_row[i]] + a.rem_slot[i]] = a.rem_token[i];
}

// A merged token's rank among its segment's tokens.
__device__ __forceinline__ void rank_token(int i, const IndexArgs& a) {
  const int row = a.rem_row[i], len = a.count[row];
  if (len > kLongSegment) return;
  const int token = a.rem_token[i], off = a.offset[row];
  int rank = 0;
  for (int k = 0; k < len; ++k) rank += a.seg_tmp[off + k] < token ? 1 : 0;
  a.seg_src[off + rank] = token;
}

// A block per long segment: all merged tokens in order, those of the segment's row in the order met.  A chain of scans, so
// four tokens a thread to each (the launch that does it, 208,200 equal tokens, one segment of 124,920: 76 us, 162 with one; 103 with one
// and 1024 threads, which make the ranks of many middling segments slower: 65,952 tokens of 40 kinds 45 -> 75 us).
__device__ __forceinline__ void order_long_segments(int block, int blocks, const IndexArgs& a) {
  __shared__ int scratch[32];
  const int n_long = a.long_rows[0], n_remove = (int)a.n_remove;
  for (int l = block; l < n_long; l += blocks) {
    const int row = a.long_rows[1 + l];
    int at = a.offset[row];
    for (int base = 0; base < n_remove; base += threads() * kScanItems) {
      const int first = base + (int)threadIdx.x * kScanItems;
      bool mine[kScanItems];
      int sum = 0;
#pragma unroll
      for (int i = 0; i < kScanItems; ++i) {
        mine[i] = first + i < n_remove && a.rem_row[first + i] == row;
        sum += mine[i] ? 1 : 0;
      }
      int to = at + block_scan_inclusive(sum, scratch) - sum;
#pragma unroll
      for (int i = 0; i < kScanItems; ++i)
        if (mine[i]) a.seg_src[to++] = a.rem_token[first + i];
      at += scratch[31];
    }
  }
}

// kLocal: one block, which keeps in shared memory what the steps hand on.  kNumber: as far as the numbers of the tokens.
template <bool kLocal, bool kNumber>
__global__ void __launch_bounds__(kLocal || kNumber ? kIdxWideThreads : kIdxThreads, 1) index_build_kernel(const IndexArgs args) {
  IndexArgs a = args;
  extern __shared__ int local_words[];
  if constexpr (kLocal) lay_scratch(a, local_words, true);
  __shared__ IndexShared sh;
  __shared__ uint2 sums[2][kSelBins];
  const int block = kLocal ? 0 : blockIdx.x, blocks = kLocal ? 1 : gridDim.x;  // one cluster
  const bool selects = a.selects();
  for (int i = threadIdx.x; i < kSelPasses * kSelBins; i += threads()) sh.hist[0][i] = 0u;
  if (threadIdx.x < kIdxMaxBlocks) sh.part[threadIdx.x] = 0u;
  __syncthreads();
  const Span span(a.stamp);
  // runs of src tokens and of rows; a block's tokens go from its first src token to the next block's
  auto src_at = [&](int b) { return (int)(a.n_src * b / blocks); };
  auto token_at = [&](int b) {
    if (b == 0) return 0;
    if (b == blocks) return (int)a.n_tokens;
    const long long t = src_at(b) < a.n_src ? a.src_list[src_at(b)] : a.n_tokens * b / blocks;
    return (int)(t < 0 ? 0 : t < a.n_tokens ? t : a.n_tokens);
  };
  const int p0 = src_at(block), p1 = src_at(block + 1), t0 = token_at(block), t1 = token_at(block + 1);
  TokenKeys tokens;
  tokens.load_places(a, t0, t1);
  const int rows_per_block = (int)((a.n_merged + blocks - 1) / blocks);
  for (int i = block * threads() + (int)threadIdx.x; i < a.n_merged; i += blocks * threads()) a.count[i] = 0;
  if (block == 0 && threadIdx.x == 0) a.long_rows[0] = 0;
  if (kNumber && block == 0 && threadIdx.x < kIdxParts) a.part_sums[threadIdx.x] = 0;

  // (with every src token merged the threshold lies below all keys)
  Selection sel{0u, (unsigned)a.n_remove, selects || a.n_remove == 0 ? 0u : (unsigned)p0, 0u};
  unsigned held[kHeld] = {};
  read_matches<kLocal>(a, p0, p1, selects, sh.hist[0], held);
  if (selects) {
    all_blocks<kLocal>();
    sel = select_bin<0, kLocal>(sh.hist[0], sums[0], block, blocks, sel);
    count_keys<1>(a, p0, p1, sel, sh.hist[1], held);
    all_blocks<kLocal>();
    sel = select_bin<1, kLocal>(sh.hist[1], sums[1], block, blocks, sel);
    count_keys<2>(a, p0, p1, sel, sh.hist[2], held);
    all_blocks<kLocal>();
    tokens.load_keys(a);
    sel = select_bin<2, kLocal>(sh.hist[2], sums[0], block, blocks, sel);
    count_keys<3>(a, p0, p1, sel, sh.hist[3], held);
    all_blocks<kLocal>();
    sel = select_bin<3, kLocal>(sh.hist[3], sums[1], block, blocks, sel);
  } else {
    __syncthreads();
    tokens.load_keys(a);
  }
  number_tokens<kLocal>(a, t0, t1, sel.prefix, sel.need, (unsigned long long)sel.equal << 32 | sel.above, tokens);
  all_blocks<kLocal>();  // (also: no block ends while another reads its shared memory)
  if constexpr (kNumber) return;
  if (a.n_remove > 0) {
    assign_removed<2>(block, blocks, a, rows_per_block, sh.part);
    all_blocks<kLocal>();
  }
  __shared__ int rows_before;
  const long long r0 = (long long)rows_per_block * block, r1 = r0 + rows_per_block;
  lay_segments<kLocal>(a, (int)r0, (int)(r1 < a.n_merged ? r1 : a.n_merged), [&]() -> int {
    if (threadIdx.x < 32) {
      unsigned sum = 0;
      if constexpr (!kLocal) {
#pragma unroll 8
        for (int i = threadIdx.x; i < blocks * block; i += 32) sum += ld_cluster(mapa_u32(smem_u32(&sh.part[i % block]), i / block));
      }
      sum = __reduce_add_sync(0xffffffffu, sum);
      if (threadIdx.x == 0) rows_before = (int)sum;
    }
    __syncthreads();
    return rows_before;
  });
  all_blocks<kLocal>();
  if (a.n_remove == 0) return;
  for (int i = block * threads() + (int)threadIdx.x; i < a.n_remove; i += blocks * threads()) slot_token(i, a);
  all_blocks<kLocal>();
  for (int i = block * threads() + (int)threadIdx.x; i < a.n_remove; i += blocks * threads()) rank_token(i, a);
  order_long_segments(block, blocks, a);
}

// ---- the selection and the numbers of very long sequences, launches of kLongThreads threads a block
__host__ __device__ constexpr int long_shift(int pass) { return pass == 0 ? 21 : pass == 1 ? 10 : 0; }
__host__ __device__ constexpr int long_bins(int pass) { return pass == 2 ? 1024 : 2048; }

// Fixes the bits of pass `pass` from its histogram.
template <int kShift, int kBins>
__device__ __forceinline__ Selection long_select_bin(const unsigned* hist, const Selection& before) {
  __shared__ unsigned scratch[32];
  __shared__ Selection found;
  constexpr int per = kBins / kLongThreads;
  unsigned c[per], sum = 0;
#pragma unroll
  for (int i = 0; i < per; ++i) {  // from the highest bin downwards
    c[i] = hist[kBins - 1 - (threadIdx.x * per + i)];
    sum += c[i];
  }
  unsigned above = block_scan_inclusive(sum, scratch) - sum;
#pragma unroll
  for (int i = 0; i < per; ++i) {
    if (above < before.need && above + c[i] >= before.need)
      found = Selection{before.prefix | (unsigned)(kBins - 1 - (threadIdx.x * per + i)) << kShift, before.need - above, 0u, 0u};
    above += c[i];
  }
  __syncthreads();
  return found;
}

// kShift, kBins: this pass's; kShiftBefore, kBinsBefore: those of the one before, or 0 in the first, which takes the matching's
// keys apart.
template <int kPass, int kShift, int kBins, int kShiftBefore, int kBinsBefore>
__global__ void __launch_bounds__(kLongThreads) index_select_kernel(const IndexArgs a) {
  const Span span(a.stamp);
  __shared__ unsigned bins[kLongBins];
  const bool selects = a.selects();
  for (int i = threadIdx.x; i < kLongBins; i += kLongThreads) bins[i] = 0u;
  Selection so_far{0u, (unsigned)a.n_remove, 0u, 0u};
  if constexpr (kPass > 0) {
    if constexpr (kPass == 2) so_far = a.sel[0];
    so_far = long_select_bin<kShiftBefore, kBinsBefore>(a.hist + (kPass - 1) * kLongBins, so_far);
    if (blockIdx.x == 0 && threadIdx.x == 0) a.sel[kPass - 1] = so_far;
  } else {
    for (long long i = (long long)blockIdx.x * kLongThreads + threadIdx.x; i < a.n_merged; i += (long long)gridDim.x * kLongThreads) a.count[i] = 0;
    if (blockIdx.x == 0 && threadIdx.x < kIdxParts) a.part_sums[threadIdx.x] = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) a.long_rows[0] = 0;
  }
  __syncthreads();
  for (long long base = (long long)blockIdx.x * kLongThreads; base < a.n_src; base += (long long)gridDim.x * kLongThreads) {
    const int i = (int)base + (int)threadIdx.x;
    bool on = i < a.n_src;
    unsigned k = 0;
    if (on) {
      if constexpr (kPass == 0) {
        k = take_match<false>(a, i, a.match_key[i], a.inv_norm_src[i]);
      } else {
        k = a.key[i];
        on = (k >> kShiftBefore) == (so_far.prefix >> kShiftBefore);
      }
    }
    if (selects) hist_add(bins, (k >> kShift) & (unsigned)(kBins - 1), on);
  }
  if (!selects) return;
  __syncthreads();
  for (int i = threadIdx.x; i < kBins; i += kLongThreads)
    if (bins[i] != 0u) atomicAdd(&a.hist[kPass * kLongBins + i], bins[i]);
}

// Threshold (from the last histogram; below all keys where every src token is merged) and the counts of every chunk of tokens.
__global__ void __launch_bounds__(kLongThreads) index_count_kernel(const IndexArgs a) {
  const Span span(a.stamp);
  __shared__ unsigned long long scratch[32];
  TokenKeys t;  // (on its way while the bin is found)
  t.load_places(a, blockIdx.x * kLongChunk, (int)a.n_tokens);
  t.load_keys(a);
  const Selection s = a.n_remove == a.n_src ? Selection{0u, (unsigned)a.n_src, 0u, 0u}
                                            : long_select_bin<long_shift(2), long_bins(2)>(a.hist + 2 * kLongBins, a.sel[1]);
  if (blockIdx.x == 0 && threadIdx.x == 0) a.sel[2] = s;
  unsigned long long sum = 0ull;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i)
    sum += t.pos[i] < 0 ? 0ull : t.key[i] > s.prefix ? 1ull : t.key[i] == s.prefix ? 1ull << 32 : 0ull;
  const unsigned long long incl = block_scan_inclusive(sum, scratch);
  if (threadIdx.x == kLongThreads - 1) a.token_sums[blockIdx.x] = incl;
}

__global__ void __launch_bounds__(kLongThreads) index_number_kernel(const IndexArgs a) {
  const Span span(a.stamp);
  __shared__ unsigned long long scratch[32];
  Selection s{};
  unsigned long long before = 0ull;
  TokenKeys t;
  const int first = blockIdx.x * kLongChunk;
  t.load_places(a, first, (int)a.n_tokens);
  t.load_keys(a);
  if (a.n_remove > 0) {
    s = a.sel[2];
    block_scan_inclusive((int)threadIdx.x < (int)blockIdx.x ? a.token_sums[threadIdx.x] : 0ull, scratch);
    before = scratch[31];
  }
  number_tokens<false>(a, first, (int)min((long long)first + kLongChunk, a.n_tokens), s.prefix, s.need, before, t);
}

// The steps behind the numbers as launches over the chip.
__global__ void __launch_bounds__(kIdxThreads) index_assign_kernel(const IndexArgs a, int rows_per_part) {
  __shared__ unsigned part[kIdxParts];
  if (threadIdx.x < kIdxParts) part[threadIdx.x] = 0u;
  __syncthreads();
  const Span span(a.stamp);
  assign_removed<1>(blockIdx.x, gridDim.x, a, rows_per_part, part);
  __syncthreads();
  if (threadIdx.x < kIdxParts && part[threadIdx.x] != 0u) atomicAdd(&a.part_sums[threadIdx.x], (int)part[threadIdx.x]);
}
__global__ void __launch_bounds__(kIdxWideThreads) index_lay_kernel(const IndexArgs a, int rows_per_part) {
  const Span span(a.stamp);
  __shared__ int rows_before;
  const long long r0 = (long long)rows_per_part * blockIdx.x, r1 = r0 + rows_per_part;
  lay_segments<false>(a, (int)r0, (int)(r1 < a.n_merged ? r1 : a.n_merged), [&]() -> int {
    if (threadIdx.x < 32) {
      int sum = 0;
      for (int i = threadIdx.x; i < (int)blockIdx.x; i += 32) sum += a.part_sums[i];
      sum = __reduce_add_sync(0xffffffffu, sum);
      if (threadIdx.x == 0) rows_before = sum;
    }
    __syncthreads();
    return rows_before;
  });
}
__global__ void __launch_bounds__(kIdxThreads) index_slot_kernel(const IndexArgs a) {
  const Span span(a.stamp);
  const int i = blockIdx.x * threads() + (int)threadIdx.x;
  if (i < a.n_remove) slot_token(i, a);
}
__global__ void __launch_bounds__(kIdxThreads) index_order_kernel(const IndexArgs a) {
  const Span span(a.stamp);
  const int rank_blocks = (int)((a.n_remove + threads() - 1) / threads()), i = blockIdx.x * threads() + (int)threadIdx.x;
  if ((int)blockIdx.x >= rank_blocks) order_long_segments(blockIdx.x - rank_blocks, gridDim.x - rank_blocks, a);
  else if (i < a.n_remove) rank_token(i, a);
}

static IndexArgs index_sizes(const Sizes& z) {
  IndexArgs a = {};
  a.n_src = z.n_src;
  a.n_dst = z.n_dst;
  a.n_tokens = z.n_tokens;
  a.n_merged = z.n_merged;
  a.n_remove = z.n_remove;
  return a;
}
// Words of the index build's scratch array.
long long index_scratch_words(const Sizes& z) {
  IndexArgs a = index_sizes(z);
  return lay_scratch(a, nullptr, false);
}

// Which form, by what a plan's build on new features and the merge behind it take (us):
//   one block up to kLocalTokens, which keep in its shared memory what it hands on (one block / the cluster): 3,360 tokens 47.7 / 53.7, 4,050
//     55.3 / 58.6, 5,040 68.2 / 68.2, 6,300 69.7 / 67.5, 7,203 78.3 / 74.3, 8,820 93.4 / 82.2; of 40 kinds, each token's rank counted
//     among many, 5,040 83.9 / 80.1, 6,300 107 / 98, 8,820 155 / 127;
//   one cluster, while what its 16 SMs do for all tokens is less than the launches: 12,600 tokens 120 (as launches 122);
//   launches behind the numbers of the tokens: 43,968 tokens 568 (in the cluster 572), 66,624 1148 (1159);
//   launches throughout, from kManyTokens on.
constexpr long long kLocalTokens = 5120;
constexpr int kLocalBytes = 164 * 1024;
static_assert(kLocalTokens * 8 * 4 + 2048 <= kLocalBytes, "at most eight words a token (all src, all merged) and the fixed ones");
constexpr long long kWideTokens = 4096;  // (kIdxThreads above; 4,164 tokens 56.4 with 512 threads, 54.9 with 1024)
constexpr long long kClusterTokens = 32768;

// Blocks of the cluster: 16 SMs where the device has that many together (more than the eight that every one has to offer).
static int cluster_blocks(const void* kernel, int threads, std::atomic<unsigned long long>& asked, std::atomic<unsigned long long>& fits) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return kIdxPortableBlocks;
  const unsigned long long bit = 1ull << (dev & 63);
  if ((asked.load(std::memory_order_acquire) & bit) == 0) {
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = kIdxMaxBlocks;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kIdxMaxBlocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0)
      fits.fetch_or(bit, std::memory_order_release);
    else
      (void)cudaGetLastError();
    asked.fetch_or(bit, std::memory_order_release);
  }
  return (fits.load(std::memory_order_acquire) & bit) != 0 ? kIdxMaxBlocks : kIdxPortableBlocks;
}

// The histograms of a very long sequence, which have to be zero before launch_index_build where it selects; the matching sees to it.
ZeroWords index_zero_words(const litevggt_ctx* ctx) {
  IndexArgs a = index_sizes(ctx->sz);
  lay_scratch(a, ctx->ws.index_scratch, false);
  return a.n_tokens > kManyTokens && a.selects() ? ZeroWords{a.hist, 3 * kLongBins} : ZeroWords{};
}

cudaError_t launch_index_build(litevggt_ctx* ctx, litevggt_plan* plan, cudaStream_t s, int* launches) {
  Workspace& ws = ctx->ws;
  IndexArgs a = index_sizes(ctx->sz);
  a.match_key = ws.match_keys;
  a.src_list = ws.src_list;
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
  a.status = ws.status;
  const long long local_bytes = 4 * lay_scratch(a, ws.index_scratch, true);
  lay_scratch(a, ws.index_scratch, false);
  auto stamped = [&]() -> const IndexArgs& {
    a.stamp = next_stamp(ctx);
    ++*launches;
    return a;
  };
  if (a.n_tokens <= kLocalTokens) {
    const auto build = index_build_kernel<true, false>;
    static std::atomic<unsigned long long> smem_set{0};
    const cudaError_t e = set_max_dynamic_smem_once(reinterpret_cast<const void*>(build), kLocalBytes, smem_set);
    if (e != cudaSuccess) return e;
    return launch(build, dim3(1), a.n_tokens > kWideTokens ? kIdxWideThreads : kIdxThreads, (size_t)local_bytes, s, stamped());
  }
  const bool wide = a.n_tokens > kClusterTokens, many = a.n_tokens > kManyTokens;
  const auto build = wide ? index_build_kernel<false, true> : index_build_kernel<false, false>;
  const int threads = wide ? kIdxWideThreads : kIdxThreads;
  static std::atomic<unsigned long long> asked[2], fits[2];
  const int cluster = cluster_blocks(reinterpret_cast<const void*>(build), threads, asked[wide], fits[wide]);
  cudaError_t e = cudaSuccess;
  if (!many) e = launch_clusters(cluster, true, build, dim3((unsigned)cluster), (unsigned)threads, 0, s, stamped());
  if (many) {
    // at most as many blocks as run at a time: each flushes a histogram
    const bool selects = a.selects();
    long long blocks = (a.n_src + 4 * kLongThreads - 1) / (4 * kLongThreads);
    const dim3 select((unsigned)(blocks < 1 ? 1 : blocks < 2 * ctx->num_sms ? blocks : 2 * ctx->num_sms));
    const dim3 chunks((unsigned)((a.n_tokens + kLongChunk - 1) / kLongChunk));
    e = launch(index_select_kernel<0, long_shift(0), long_bins(0), 0, 0>, select, kLongThreads, 0, s, stamped());
    if (e == cudaSuccess && selects)
      e = launch(index_select_kernel<1, long_shift(1), long_bins(1), long_shift(0), long_bins(0)>, select, kLongThreads, 0, s, stamped());
    if (e == cudaSuccess && selects)
      e = launch(index_select_kernel<2, long_shift(2), long_bins(2), long_shift(1), long_bins(1)>, select, kLongThreads, 0, s, stamped());
    if (e == cudaSuccess && a.n_remove > 0) e = launch(index_count_kernel, chunks, kLongThreads, 0, s, stamped());
    if (e == cudaSuccess) e = launch(index_number_kernel, chunks, kLongThreads, 0, s, stamped());
  }
  if (e != cudaSuccess || !wide) return e;
  const int rows_per_part = (int)((a.n_merged + kIdxParts - 1) / kIdxParts);
  const unsigned blocks = (unsigned)((a.n_remove + kIdxThreads - 1) / kIdxThreads);
  if (blocks > 0) e = launch(index_assign_kernel, dim3(blocks), kIdxThreads, 0, s, stamped(), rows_per_part);
  // (1024 threads where they make it one scan a block: 1,041,000 tokens 14.2 -> 8.5 us)
  const int lay_threads = rows_per_part > kIdxThreads * kScanItems ? kIdxWideThreads : kIdxThreads;
  if (e == cudaSuccess) e = launch(index_lay_kernel, dim3(kIdxParts), lay_threads, 0, s, stamped(), rows_per_part);
  if (e == cudaSuccess && blocks > 0) e = launch(index_slot_kernel, dim3(blocks), kIdxThreads, 0, s, stamped());
  if (e == cudaSuccess && blocks > 0)
    e = launch(index_order_kernel, dim3(blocks + (a.n_remove > kLongSegment ? kLongBlocks : 0)), kIdxThreads, 0, s, stamped());
  return e;
}

}  // namespace lv

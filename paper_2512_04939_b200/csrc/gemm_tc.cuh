// Persistent bf16 GEMM mainloop on the 5th-generation tensor cores:
//   C[m, n] = sum_k A[m, k] * B[n, k]        (both operands K-major, fp32 accumulate)
// with a pluggable epilogue that consumes the accumulator straight out of tensor memory.
//
// Used by (a) the projection layers of the attention block (plain epilogue: + bias,
// round to bf16, store) and (b) the src->anchor cosine matching (epilogue keeps a
// running row argmax, so the |Src| x |Dst| score matrix never exists in memory).
//
// Mostly two CTAs (a cluster, the two SMs of a TPC) share a tile of 256 rows x kBN columns: each holds its
// own 128 rows of A and half of the tile's rows of B, and one tcgen05.mma.cta_group::2 per 16 of K
// reads both halves of B from both SMs.  What bounds the mainloop is the stream from L2 into shared
// memory, and a pair needs 32 KB per CTA and k-block of a 256-column tile where a CTA of its own
// needs 48 KB for the same arithmetic: 1322 -> 1434 TFLOP/s on 52,050 rows x 1024 x 3072, 1465 -> 1535 at
// k = 4096 and 104 K rows.  Narrow tiles fill the chip where rows are few (543 rows x 1024 x 1024: 10.1 -> 7.6 us).
// A CTA of its own with 128 x 256 tiles (kCtas = 1) remains
// where its finer rows save a wave (3360 rows x 1024 x 4096: 23.6 us against 27.1) and for short k,
// where the epilogue bounds the launch and a pair would drain in step.
//
// Shape of one CTA of the pair:
//   warp 0      TMA producer (one elected lane): A tile 128 x 64 and B tile kBN/2 x 64 per
//               k-block into a shared-memory ring (128-byte swizzle); both CTAs' loads count
//               towards the `full` barrier of the leader (the CTA of even rank)
//   warp 1      leader only: MMA issuer (one elected lane), 4 x tcgen05.mma M256 K16 per k-block
//               into one of two kBN-column fp32 accumulators in both SMs' tensor memory; its
//               commits arrive on the barriers of both CTAs
//   warps 2..   epilogue: each thread owns one accumulator row (one TMEM lane) and
//               walks its columns in chunks while the issuer already fills the other
//               accumulator.  An epilogue with per-row state (the argmax) runs on four
//               warps, one per 32-lane quarter, over all columns.  An epilogue that
//               writes a matrix runs on eight (two per quarter, every other 64 columns) and
//               hands every 64-column chunk back as bf16; the warp parks its 32 x 64
//               block in shared memory (128-byte swizzle) and one lane sends it to
//               global memory as a TMA store, so rows leave the SM as whole 128-byte
//               lines
// Tile order.  With a row-state epilogue each pair owns a block of 256 rows at a time and
// sweeps all column tiles in ascending order (the state stays in registers); all pairs sweep
// in step, so a tile of B comes from HBM once for all of them.  Row blocks are handed out
// round-robin as long as there is one for every pair; the rest, a last wave that would
// leave most of the chip idle (1 block for 74 pairs at 200 frames of 28 x 37, 32 at 32 of 37 x 37), is dealt
// out in equal runs of column tiles, and the epilogue combines what it found in parts of a
// row's sweep.  With a matrix epilogue tiles are numbered row block major and dealt
// round-robin, so the CTAs running at one moment share a few row blocks of A and the whole
// of B stays in L2 - with the row-block order and K = 4096 the resident A panels outgrew L2.
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "gemm_tiles.h"

namespace lv {

constexpr int kGemmBK = 64;
constexpr int kGemmMaxThreads = 320;  // 2 + 8 warps
// Threads of a launch: TMA warp + MMA warp + 4 (row-state epilogue) or 8 (matrix epilogue) warps.
template <class Epi>
constexpr int gemm_threads() {
  return 64 + (Epi::kTileOut ? 256 : 128);
}
constexpr int kGemmTileABytes = kGemmBM * kGemmBK * 2;
constexpr int kGemmOutChunkCols = 64;                                   // columns per staged output block
constexpr int kGemmOutBlockBytes = 32 * kGemmOutChunkCols * 2;          // one warp's 32 rows x 64 columns
constexpr int kGemmOutBytes = 8 * kGemmOutBlockBytes;                   // one block per epilogue warp

// Ring geometry of a tile of kBN columns shared by kCtas CTAs.
template <int kBN, int kCtas>
struct GemmShape {
  static constexpr int kTileBBytes = kBN / kCtas * kGemmBK * 2;
  static constexpr int kStageBytes = kGemmTileABytes + kTileBBytes;
  static constexpr int kStages = 6 * 32768 / kStageBytes;  // a pair: 6 at 256 columns, 9 at 64; one CTA: 4 at 256
  static constexpr uint32_t kTmemCols = kBN > 128 ? 512 : 2 * kBN;  // two accumulators, a power of two
  static constexpr int kSmemBytes = kStages * kStageBytes + kGemmOutBytes + 512 + 1024;  // + barriers + slack
};

template <int kStages>
struct GemmBarriers {
  uint64_t full[kStages];   // used in the leader
  uint64_t empty[kStages];
  uint64_t tmem_full[2];
  uint64_t tmem_empty[2];   // used in the leader
  uint64_t teardown;
  uint32_t tmem_base;
  uint32_t abort_flag;
};

// The i-th tile of a pair (or of a CTA of its own); false once it has run out of tiles.  `first` / `last`:
// the tile begins / ends the pair's run through this row block.
struct GemmTile {
  int mb, nt;
  bool first, last;
};
template <bool kRoundRobinTiles>
__device__ __forceinline__ bool gemm_tile_at(int i, int pair, int pairs, int num_m_blocks, int num_n_tiles, GemmTile& tile) {
  if constexpr (kRoundRobinTiles) {
    const long long t = (long long)pair + (long long)i * pairs;
    if (t >= (long long)num_m_blocks * num_n_tiles) return false;
    tile.mb = (int)(t / num_n_tiles);
    tile.nt = (int)(t % num_n_tiles);
    return true;
  } else {
    const int full = num_m_blocks / pairs;  // sweeps with a row block for every pair
    if (i < full * num_n_tiles) {
      tile.mb = pair + i / num_n_tiles * pairs;
      tile.nt = i % num_n_tiles;
      tile.first = tile.nt == 0;
      tile.last = tile.nt == num_n_tiles - 1;
      return true;
    }
    const long long rest = (long long)(num_m_blocks - full * pairs) * num_n_tiles;
    const long long lo = rest * pair / pairs, hi = rest * (pair + 1) / pairs;
    const long long t = lo + (i - full * num_n_tiles);
    if (t >= hi) return false;
    tile.mb = full * pairs + (int)(t / num_n_tiles);
    tile.nt = (int)(t % num_n_tiles);
    tile.first = tile.nt == 0 || t == lo;
    tile.last = tile.nt == num_n_tiles - 1 || t == hi - 1;
    return true;
  }
}

template <class Epi, int kBN, int kCtas>
__global__ void __launch_bounds__(kGemmMaxThreads, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
               const __grid_constant__ CUtensorMap tmap_out, int m_rows, int n_cols, int k_dim, Epi epi,
               uint32_t* status, ZeroWords zero, Stamp stamp) {
  using Shape = GemmShape<kBN, kCtas>;
  constexpr int kStages = Shape::kStages;
  constexpr bool kPair = kCtas == 2;
  static_assert(kPair || Epi::kTileOut, "the row-state epilogue runs on pairs");
  static_assert(!kPair || (kBN % 32 == 0 && kBN <= 256), "columns of an instruction of a pair");
  static_assert(kBN % kGemmOutChunkCols == 0 || (kBN % kGemmOutChunkCols == 32 && Epi::kTileOut), "");
  extern __shared__ uint8_t smem_raw[];
  // the same offset in both CTAs of a pair: the leader's descriptors address the other CTA's tiles too
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* smem_a = smem;
  uint8_t* smem_b = smem + kStages * kGemmTileABytes;
  uint8_t* smem_out = smem + kStages * Shape::kStageBytes;
  GemmBarriers<kStages>* bars = reinterpret_cast<GemmBarriers<kStages>*>(smem_out + kGemmOutBytes);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = kPair ? cluster_ctarank() : 0u;
  const bool leader = rank == 0;
  const int pair = blockIdx.x / kCtas, pairs = gridDim.x / kCtas;
  const int num_m_blocks = (m_rows + kCtas * kGemmBM - 1) / (kCtas * kGemmBM);
  const int num_n_tiles = (n_cols + kBN - 1) / kBN;
  const int num_kb = k_dim / kGemmBK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bars->tmem_full[b], 1);
      mbar_init(&bars->tmem_empty[b], (Epi::kTileOut ? 8 : 4) * kCtas);  // the epilogue warps of both CTAs
    }
    mbar_init(&bars->teardown, 1);
    bars->abort_flag = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tmap_a);
    tma_prefetch_desc(&tmap_b);
    if constexpr (Epi::kTileOut) tma_prefetch_desc(&tmap_out);
  }
  if (warp == 1) {
    if constexpr (kPair) {
      tmem_alloc_pair(&bars->tmem_base, Shape::kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(&bars->tmem_base, Shape::kTmemCols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  if constexpr (kPair) cluster_sync(); else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = bars->tmem_base;
  const WaitCtl ctl{&bars->abort_flag, status};
  const Span span(stamp);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < zero.count; i += (long long)gridDim.x * blockDim.x)
    zero.words[i] = 0u;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      uint32_t issued = 0;
      bool ok = true;
      GemmTile tile;
      for (int i = 0; ok && gemm_tile_at<Epi::kTileOut>(i, pair, pairs, num_m_blocks, num_n_tiles, tile); ++i) {
        const int row = (kCtas * tile.mb + (int)rank) * kGemmBM, col = tile.nt * kBN + (int)rank * (kBN / kCtas);
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!mbar_wait(&bars->empty[stage], phase ^ 1u, ctl)) { ok = false; break; }
          if (leader) mbar_expect_tx(&bars->full[stage], kCtas * Shape::kStageBytes);
          uint8_t* dst_a = smem_a + stage * kGemmTileABytes;
          uint8_t* dst_b = smem_b + stage * Shape::kTileBBytes;
          if constexpr (kPair) {
            const uint32_t full = mapa_u32(smem_u32(&bars->full[stage]), 0);
            tma_load_2d_pair(dst_a, &tmap_a, full, kb * kGemmBK, row);
            tma_load_2d_pair(dst_b, &tmap_b, full, kb * kGemmBK, col);
          } else {
            tma_load_2d(dst_a, &tmap_a, &bars->full[stage], kb * kGemmBK, row);
            tma_load_2d(dst_b, &tmap_b, &bars->full[stage], kb * kGemmBK, col);
          }
          ++issued;
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
      // Drain: every load this thread issued must have landed and been consumed (and the commit that says
      // so have arrived here) before the CTA may exit; a pair that gave up still waits for its loads.
      const uint32_t n_drain = issued < (uint32_t)kStages ? issued : (uint32_t)kStages;
      for (uint32_t i = 0; i < n_drain; ++i) {
        // walk back over the most recently used stages
        int s = stage - 1 - (int)i;
        uint32_t ph = phase;
        while (s < 0) { s += kStages; ph ^= 1u; }
        const long long t0 = clock64();
        while (!mbar_try_wait(&bars->empty[s], ph)) {
          // (the other CTA's barrier counts this one's bytes: without it, give them a million cycles)
          if (*ctl.abort_flag != 0u && (leader ? mbar_try_wait(&bars->full[s], ph) : clock64() - t0 > (1ll << 20))) break;
          if (clock64() - t0 > kTimeoutCycles) { atomicOr(status, kStatusTimeout); break; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (leader && elect_one()) {
      constexpr uint32_t idesc = umma_idesc_bf16(kCtas * kGemmBM, kBN, false, false);
      auto commit = [](uint64_t* bar, uint16_t ctas) {
        if constexpr (kPair) umma_commit_pair(bar, ctas); else umma_commit(bar);
      };
      const uint64_t a_desc0 = smem_desc_sw128(smem_u32(smem_a), 16, 1024);
      const uint64_t b_desc0 = smem_desc_sw128(smem_u32(smem_b), 16, 1024);
      int stage = 0;
      uint32_t phase = 0;
      uint32_t tile_iter = 0;
      bool ok = true;
      GemmTile tile;
      for (int i = 0; ok && gemm_tile_at<Epi::kTileOut>(i, pair, pairs, num_m_blocks, num_n_tiles, tile); ++i, ++tile_iter) {
        const uint32_t ab = tile_iter & 1u;
        const uint32_t ab_phase = (tile_iter >> 1) & 1u;
        if (!mbar_wait(&bars->tmem_empty[ab], ab_phase ^ 1u, ctl)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + ab * kBN;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!mbar_wait(&bars->full[stage], phase, ctl)) { ok = false; break; }
          tc_fence_after();
          // the descriptors are linear in the shared-memory address (16-byte units in the low bits)
          const uint64_t a_desc = a_desc0 + (uint64_t)(stage * (kGemmTileABytes >> 4));
          const uint64_t b_desc = b_desc0 + (uint64_t)(stage * (Shape::kTileBBytes >> 4));
#pragma unroll
          for (int k = 0; k < kGemmBK / 16; ++k) {
            // +32 bytes along K inside the swizzled row = +2 in descriptor units
            if constexpr (kPair) umma_ss_pair(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
            else umma_ss(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
          }
          commit(&bars->empty[stage], 3);
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        if (ok) commit(&bars->tmem_full[ab], 3);
      }
      if (!ok) {
        // make sure no MMA is still in flight before tensor memory is released
        commit(&bars->teardown, 1);
        const long long t0 = clock64();
        while (!mbar_try_wait(&bars->teardown, 0)) {
          if (clock64() - t0 > kTimeoutCycles) break;
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue warps
    const uint32_t quarter = warp & 3u;  // TMEM lanes 32*quarter .. 32*quarter+31
    const int half = (warp - 2) >> 2;    // even or odd 64-column chunks (matrix epilogue only)
    const int row_in_tile = quarter * 32 + lane;
    uint32_t tile_iter = 0;
    uint32_t chunk_iter = 0;
    typename Epi::State st;
    GemmTile tile;
    for (int i = 0; gemm_tile_at<Epi::kTileOut>(i, pair, pairs, num_m_blocks, num_n_tiles, tile); ++i, ++tile_iter) {
      const int row0 = (kCtas * tile.mb + (int)rank) * kGemmBM;
      const int row = row0 + row_in_tile;
      if constexpr (!Epi::kTileOut) {
        if (tile.first) epi.begin(st, row);
      }
      const uint32_t ab = tile_iter & 1u;
      const uint32_t ab_phase = (tile_iter >> 1) & 1u;
      if (!mbar_wait_warp_in_line(&bars->tmem_full[ab], ab_phase, ctl)) break;
      tc_fence_after();
      const uint32_t t_addr = tmem_base + ((quarter * 32u) << 16) + ab * kBN;
      if constexpr (Epi::kTileOut) {
        const int warp_row0 = row0 + (int)quarter * 32;
        uint8_t* block = smem_out + (warp - 2) * kGemmOutBlockBytes;
#pragma unroll 1
        for (int c = half; c < (kBN + kGemmOutChunkCols - 1) / kGemmOutChunkCols; c += 2) {
          const int col0 = tile.nt * kBN + c * kGemmOutChunkCols;
          if (col0 >= n_cols || warp_row0 >= m_rows) break;  // nothing of this block exists (warp-uniform)
          int r = row;
          // Worked out for every chunk: held over the loop, the row's addresses spill (12 bytes at 224 columns, 8 at 160; both
          // layers of an MLP of 1,153 rows 30.5 us, 30.0 so, 1,777 34.0 and 33.4).  Other widths have the registers.
          if constexpr (kBN % kGemmOutChunkCols != 0) asm volatile("" : "+r"(r));
          uint32_t acc[64];  // (where the tile ends before, what lies behind it is read and not used)
          tmem_ld32(t_addr + c * 64, reinterpret_cast<uint32_t(&)[32]>(acc[0]));
          tmem_ld32(t_addr + c * 64 + 32, reinterpret_cast<uint32_t(&)[32]>(acc[32]));
          tmem_ld_wait();
          uint32_t packed[32];
          if constexpr (kBN % kGemmOutChunkCols != 0) {
            // The end of such a tile, or of the matrix within one: 32 columns, two whole sectors that the row's thread stores.
            if (min(kBN - c * kGemmOutChunkCols, n_cols - col0) < kGemmOutChunkCols) {
              epi.template convert<4>(r, col0, acc, packed);
              if (r < m_rows) {
                uint4* dst = reinterpret_cast<uint4*>(epi.out + (long long)r * n_cols + col0);
#pragma unroll
                for (int q = 0; q < 4; ++q) dst[q] = make_uint4(packed[4 * q], packed[4 * q + 1], packed[4 * q + 2], packed[4 * q + 3]);
              }
              continue;
            }
          }
          epi.transform(r, col0, acc, packed);
          // The previous store out of this warp's staging block must be done reading it.
          if (chunk_iter != 0) {
            if (lane == 0) bulk_wait_group_read<0>();
            __syncwarp();
          }
          // Row `lane` of the block, its eight 16-byte units permuted the way the 128-byte swizzle
          // of the store's tensor map expects (unit u of row r sits at u ^ (r mod 8)).
          uint8_t* my_row = block + lane * 128;
#pragma unroll
          for (int u = 0; u < 8; ++u)
            *reinterpret_cast<uint4*>(my_row + ((u ^ (lane & 7)) << 4)) =
                make_uint4(packed[4 * u], packed[4 * u + 1], packed[4 * u + 2], packed[4 * u + 3]);
          fence_proxy_async_shared();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&tmap_out, block, col0, warp_row0);
            bulk_commit_group();
          }
          ++chunk_iter;
        }
      } else {
#pragma unroll 1
        for (int c = 0; c < kBN / 32; ++c) {
          uint32_t acc[32];
          tmem_ld32(t_addr + c * 32, acc);
          tmem_ld_wait();
          epi.consume(st, row, tile.nt * kBN + c * 32, acc);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if constexpr (kPair) mbar_arrive_cluster(mapa_u32(smem_u32(&bars->tmem_empty[ab]), 0));
        else mbar_arrive(&bars->tmem_empty[ab]);
      }
      if constexpr (!Epi::kTileOut) {
        if (tile.last) epi.finish(st, row);
      }
    }
    // Shared memory must outlive every store that still reads it.
    if constexpr (Epi::kTileOut) {
      if (lane == 0) bulk_wait_group_all();
    }
  }

  // neither CTA may exit while the other can still arrive on its barriers or its tiles are being read
  __syncwarp();
  tc_fence_before();
  if constexpr (kPair) cluster_sync(); else __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    if constexpr (kPair) tmem_dealloc_pair(tmem_base, Shape::kTmemCols); else tmem_dealloc(tmem_base, Shape::kTmemCols);
  }
}

// One launch of the mainloop on at most one CTA per SM; `work` bounds the pairs (or CTAs) that find something
// to do.
template <class Epi, int kBN, int kCtas>
cudaError_t gemm_launch(const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& out, long long m, long long n,
                        long long k, const Epi& epi, long long work, int num_sms, uint32_t* status,
                        const ZeroWords& zero, const Stamp& stamp, cudaStream_t s) {
  using Shape = GemmShape<kBN, kCtas>;
  static std::atomic<unsigned long long> smem_set{0};
  cudaError_t e = set_max_dynamic_smem_once(reinterpret_cast<const void*>(gemm_tc_kernel<Epi, kBN, kCtas>), Shape::kSmemBytes,
                                            smem_set);
  if (e != cudaSuccess) return e;
  const long long groups = work < num_sms / kCtas ? work : num_sms / kCtas;
  return launch_clusters(kCtas, true, gemm_tc_kernel<Epi, kBN, kCtas>, dim3((unsigned)(kCtas * groups)), gemm_threads<Epi>(),
                         Shape::kSmemBytes, s, a, b, out, (int)m, (int)n, (int)k, epi, status, zero, stamp);
}

// ----------------------------------------------------------------------------------------
// Statistics of a projected Q/K/V matrix that the attention needs before it starts, taken from the
// rounded values while they are still in the epilogue's registers (a chunk of 64 columns is one
// head of one tensor): a pass over the matrix of its own cost 19 us (key norms, 22 K rows) to 66 us
// (208 K rows, 200 sequences), and 184 us for the magnitudes of 22 K rows, whose atomics met on 48 words.
// Here a warp reduces its 32 rows and sends one atomic per sequence that they touch.
enum : int { kStatNone = 0, kStatKeyNorm = 1, kStatValues = 2, kStatAmax = 3 };

// Epilogue: out[row, col] = bf16(acc + bias[col])
struct LinearEpilogue {
  static constexpr bool kTileOut = true;
  struct State {};
  const __nv_bfloat16* bias;  // may be null
  __nv_bfloat16* out;
  int m_rows;
  int n_cols;
  int scale_begin, scale_end;  // output columns [scale_begin, scale_end) are multiplied by `scale`
  float scale;
  // kStatKeyNorm: stat[seq][0][head] = largest |row|^2 over the head's 64 columns, for the columns [scale_begin, scale_end)
  //               (K) and sequences of seq_len rows, stat[seq][1][head] = largest magnitude of as many columns behind them (V);
  // kStatValues: the magnitudes only;
  // kStatAmax:    stat[col / 64] = largest magnitude of those 64 columns.  Both start at zero.
  int stat_kind;
  int seq_len;
  float* stat;

  __device__ __forceinline__ static float largest(const uint32_t (&packed)[32]) {
    float a = 0.0f;  // fmaxf drops a NaN
#pragma unroll
    for (int i = 0; i < 32; ++i) a = fmaxf(a, fmaxf(fabsf(bf16_lo(packed[i])), fabsf(bf16_hi(packed[i]))));
    return a;
  }
  // 64 accumulator columns of one row -> 32 bf16 pairs
  __device__ __forceinline__ void transform(int row, int col0, const uint32_t (&acc)[64], uint32_t (&packed)[32]) const {
    convert<8>(row, col0, acc, packed);
    if (stat_kind == kStatAmax) {
      const uint32_t best = __reduce_max_sync(0xffffffffu, row < m_rows ? __float_as_uint(largest(packed)) : 0u);
      if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned int*>(stat) + col0 / 64, best);
    } else if (stat_kind != kStatNone && col0 >= (stat_kind == kStatValues ? scale_end : scale_begin) && col0 < 2 * scale_end - scale_begin) {
      const bool is_v = col0 >= scale_end;
      float what;  // (NaN counts as 0)
      if (is_v) {
        what = largest(packed);
      } else {
        float sum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          sum[i & 3] = fmaf(bf16_lo(packed[i]), bf16_lo(packed[i]), sum[i & 3]);
          sum[i & 3] = fmaf(bf16_hi(packed[i]), bf16_hi(packed[i]), sum[i & 3]);
        }
        what = fmaxf(0.0f, (sum[0] + sum[1]) + (sum[2] + sum[3]));
      }
      // non-negative floats order like their bit patterns; the warp's first row is live (see the caller)
      const int row0 = row - (int)(threadIdx.x & 31);
      const int mine = row < m_rows ? row / seq_len : -1;
      const int last = (row0 + 31 < m_rows ? row0 + 31 : m_rows - 1) / seq_len;
      const int heads = (scale_end - scale_begin) / 64, at = (col0 - scale_begin) / 64;  // K's heads, then V's
      for (int seq = row0 / seq_len; seq <= last; ++seq) {
        const uint32_t best = __reduce_max_sync(0xffffffffu, mine == seq ? __float_as_uint(what) : 0u);
        if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned int*>(stat) + seq * 2 * heads + at, best);
      }
    }
  }
  // the first kEights x 8 of them, which lie on one side of the scale's borders
  template <int kEights>
  __device__ __forceinline__ void convert(int, int col0, const uint32_t (&acc)[64], uint32_t (&packed)[32]) const {
    const float sc = (col0 >= scale_begin && col0 < scale_end) ? scale : 1.0f;
    if (bias != nullptr) {
      const uint4* bp = reinterpret_cast<const uint4*>(bias + col0);
#pragma unroll
      for (int q = 0; q < kEights; ++q) {
        const uint4 b = __ldg(bp + q);
        const uint32_t bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float lo = (__uint_as_float(acc[q * 8 + 2 * i]) + bf16_lo(bw[i])) * sc;
          const float hi = (__uint_as_float(acc[q * 8 + 2 * i + 1]) + bf16_hi(bw[i])) * sc;
          packed[q * 4 + i] = pack_bf16(lo, hi);
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4 * kEights; ++i)
        packed[i] = pack_bf16(__uint_as_float(acc[2 * i]) * sc, __uint_as_float(acc[2 * i + 1]) * sc);
    }
  }
};

// GELU with the error function, x Phi(x) = 0.5 x (1 + erf(x / sqrt 2)).  erf comes from the five-term
// rational approximation of Abramowitz & Stegun (7.1.26): for z >= 0, 1 - erf(z) = P(t) exp(-z^2) with
// t = 1 / (1 + p z), absolute error below 1.5e-7 - three orders of magnitude under the bf16 rounding
// of the result.  With h = P(t) exp(-z^2) / 2, z = |x| / sqrt 2, the result is max(x, 0) - |x| h, so the
// negative side has no cancellation and neither side a branch.  Two values at a time, in packed arithmetic, 1 / sqrt 2
// and the 1/2 in the constants: about 9 issue slots a value where the scalar form took 16, in an epilogue that shares
// them with nobody but draws on the same power (the kernels of an MLP of 208,200 rows 2.75 -> 2.68 ms, of 3,360 rows 55.6 -> 54.8 us, in
// whole passes within their noise: local half of 200 frames 5.97 -> 5.93 ms, block of 7 frames 257 us either way;
// largest error against 64 bits over [-12, 12] 3.3e-7, scalar 4.2e-7).  |x| counts as 64 at most, where h is long zero, so
// that an infinite x meets no infinity times zero; a NaN stays one.
__device__ __forceinline__ float2 gelu_erf(float2 x) {
  auto both = [](float c) { return make_float2(c, c); };
  const float2 m = make_float2(fmax_nan(-fabsf(x.x), -64.0f), fmax_nan(-fabsf(x.y), -64.0f));  // -|x|
  const float2 d = __ffma2_rn(m, both(-0.3275911f * 0.70710678118654752f), both(1.0f));
  float2 t, ex;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t.x) : "f"(d.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t.y) : "f"(d.y));
  float2 p = __ffma2_rn(both(0.5f * 1.061405429f), t, both(0.5f * -1.453152027f));
  p = __ffma2_rn(p, t, both(0.5f * 1.421413741f));
  p = __ffma2_rn(p, t, both(0.5f * -0.284496736f));
  p = __ffma2_rn(p, t, both(0.5f * 0.254829592f));
  p = __fmul2_rn(p, t);
  const float2 y = __fmul2_rn(m, both(0.84932180028801907f));  // sqrt(log2(e) / 2): 2^(-y^2) = exp(-z^2)
  const float2 y2 = __fmul2_rn(y, y);
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex.x) : "f"(-y2.x));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex.y) : "f"(-y2.y));
  return __ffma2_rn(m, __fmul2_rn(p, ex), make_float2(fmaxf(x.x, 0.0f), fmaxf(x.y, 0.0f)));
}

// Epilogue of the MLP layers: out[row, col] = bf16(act(acc + bias[col]) + residual[row, col]) with
// act = erf-GELU (0.5 x (1 + erf(x / sqrt 2))) or the identity, residual optional.
struct MlpEpilogue {
  static constexpr bool kTileOut = true;
  struct State {};
  const __nv_bfloat16* bias;      // may be null
  const __nv_bfloat16* residual;  // may be null, same shape as the output with pitch ld_res
  __nv_bfloat16* out;
  int m_rows;
  int n_cols;
  long long ld_res;
  int gelu;

  __device__ __forceinline__ void transform(int row, int col0, const uint32_t (&acc)[64], uint32_t (&packed)[32]) const {
    convert<8>(row, col0, acc, packed);
  }
  // the first kEights x 8 columns
  template <int kEights>
  __device__ __forceinline__ void convert(int row, int col0, const uint32_t (&acc)[64], uint32_t (&packed)[32]) const {
    const bool has_res = residual != nullptr && row < m_rows;
    const uint4* bp = reinterpret_cast<const uint4*>(bias + col0);
    const uint4* rp = reinterpret_cast<const uint4*>(residual + (long long)row * ld_res + col0);
#pragma unroll
    for (int q = 0; q < kEights; ++q) {
      float v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(acc[q * 8 + i]);
      if (bias != nullptr) {
        const uint4 b = __ldg(bp + q);
        const uint32_t bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          v[2 * i] += bf16_lo(bw[i]);
          v[2 * i + 1] += bf16_hi(bw[i]);
        }
      }
      if (gelu) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 g = gelu_erf(make_float2(v[2 * i], v[2 * i + 1]));
          v[2 * i] = g.x;
          v[2 * i + 1] = g.y;
        }
      }
      if (has_res) {
        const uint4 r = rp[q];
        const uint32_t rw[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          v[2 * i] += bf16_lo(rw[i]);
          v[2 * i + 1] += bf16_hi(rw[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) packed[q * 4 + i] = pack_bf16(v[2 * i], v[2 * i + 1]);
    }
  }
};

// Epilogue: running argmax over columns of acc[row, col] * inv_norm_b[col].  What a pair found in its
// run through a row block's columns goes into key[row] by an atomic maximum: the value's bits in an
// order-preserving form above the complement of the column, so the largest value wins and of equal
// ones the lowest column, whatever the runs and their order.  Keys start at zero, below every
// value.  Within a run columns are visited in ascending order and only a strictly larger value replaces
// the current best.
__host__ __device__ __forceinline__ unsigned ordered_bits(unsigned u) {  // monotone float bits -> unsigned
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
struct ArgmaxEpilogue {
  static constexpr bool kTileOut = false;
  struct State {
    float best;
    int best_col;
  };
  const float* inv_norm_b;  // [n_cols rounded up to 256], padding = 0
  unsigned long long* key;  // [m_rows]
  int m_rows;
  int n_cols;

  __device__ __forceinline__ void begin(State& st, int) const {
    st.best = -INFINITY;
    st.best_col = 0;
  }
  __device__ __forceinline__ void consume(State& st, int, int col0, const uint32_t (&acc)[32]) const {
    const int valid = n_cols - col0;  // columns of this chunk that exist
    if (valid <= 0) return;
    const float4* np = reinterpret_cast<const float4*>(inv_norm_b + col0);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 w = __ldg(np + q);
      const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = q * 4 + i;
        const float v = __uint_as_float(acc[c]) * wv[i];
        if (c < valid && v > st.best) {
          st.best = v;
          st.best_col = col0 + c;
        }
      }
    }
  }
  __device__ __forceinline__ void finish(State& st, int row) const {
    if (row >= m_rows) return;
    const float v = st.best + 0.0f;  // -0 and +0 are the same value
    atomicMax(&key[row], (unsigned long long)ordered_bits(__float_as_uint(v)) << 32 | (unsigned)~st.best_col);
  }
};

}  // namespace lv

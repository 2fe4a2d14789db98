// Global self-attention over the merged token sequence (Sec. 3.1: the frame-global
// attention layer; after merging it runs over M instead of N tokens).  Per head
//   O = softmax(Q K^T / sqrt(64)) V,      non-causal, no mask,
// computed flash-style: scores never leave the SM.
//
// One CTA = 256 query rows (two tiles of 128) of one head, sweeping all keys in tiles of
// 128 that are consumed as two halves of 64 ("steps").  Sequences of up to kFaOneTileRows rows
// take CTAs of one tile instead, two to an SM, with half of everything below: the set-up and the
// write-back of one CTA then run under the sweep of the other, and a sequence pays for ceil(rows /
// 128) tiles and not for an even number of them.  What a sequence of 1041 rows (a 28 x 37 frame) spends
// outside its nine key tiles bounded it; the frame-local layer of 200 such frames, projections
// included, went from 3.09 to 2.58 ms.  The pair of tiles reads every K/V tile once for 256 rows and
// is the faster one when the sweep is longer: 41 us (one tile) against 49 at 2.6 K rows, 67 each at 3.6 K, 121 against 118
// at 5.2 K.  Warp roles of the pair (19 warps):
//   warps 0-15  softmax.  Warp w works on query tile t = w / 8 and TMEM lane quarter w % 4 (one
//               thread = one query row); the two warps of a (tile, quarter), c = (w / 4) % 2, either
//               take every other step whole or share each, 32 of its 64 scores per row and warp
//               (see the sweep in the kernel).  In the online form, which shares, the two threads of
//               a row swap their partial row maxima through shared memory once per step.  Four
//               softmax warps per scheduler keep the special-function unit busy while others wait.
//               (Steps of 48 keys in three score buffers, so that no warp waits for the scores to be
//               refilled, measured 7 % slower: what a step costs besides its scores counts more.)
//   warp  16    MMA issuer of tile 0 (one elected lane):  S_h = Q K_jh^T  and  O += P_h V_jh
//   warp  17    TMA producer (one elected lane): K_j / V_j through two 4-stage shared-memory rings
//   warp  18    MMA issuer of tile 1 (issuing costs tens of cycles per instruction, so one
//               thread cannot feed both tiles)
// One CTA of two tiles sits on an SM, so nothing would run under the set-up, the first loads and the write-back of the
// next: a launch is one such CTA per SM, and each works off jobs (256 rows of one head) until they run out.  The
// K/V ring goes on from job to job; the next job's queries have come to shared memory by the time the last scores of this
// one have, take the old ones' place in tensor memory then, and the next scores are under way before this job's rows are
// written.  Whole layers: 4,386 rows 153 -> 148 us, 15,932 rows 1.15 -> 1.09 ms, 31,751 rows 3.64 -> 3.60; from 83 K rows
// on, at the power cap, nothing (251,872 rows 241.9 -> 243.4).  What the softmax warps do themselves between two jobs is
// what is left: with queries and rows going row by row between global memory and registers (4096 and 2048 lines for the
// load unit, twice that for a part's rows) 4.3 us from a job's last probabilities to the next one's first scores, 3.4 as
// it is, and the first job's queries in 2.1 us, not 3.4: the core at 5,205 rows 109.5 -> 105.7 us, at 8,244 250.5 ->
// 242.6, whole layers 180.9 -> 178.9, 346.3 -> 339.8, 10,410 rows 492.7 -> 487.9, 31,751 (query weights x 16) 4.27 ->
// 4.21 ms.  Jobs come off a counter, late in the job before: with a fixed stride, or taken a whole job ahead, rows in the
// online form left 3 % of 31,751 rows' time to a few CTAs at the end.  With one tile, two CTAs an SM run under each other
// anyway, and jobs measured 3 % slower.
// Tensor memory (512 columns allocated, 480 used):
//   [0,256)    S/P: tile t, half h at column t*128 + h*64.  S_th is 128 x 64 fp32.  A softmax
//              thread reads its 32 columns and writes its 32 probabilities (16 columns of bf16
//              pairs) over the start of the same 32 columns, so P_th sits in columns [0,16) and
//              [32,48) of the half and no thread writes where another one reads; the second MMA
//              takes its A operand from there, 8 columns (16 keys) per instruction.
//   [256,416)  O_0, O_1 (fp32, 80 columns each: 64 output channels, then the row sum - the second
//              MMA's B operand carries a column of ones next to V, so the tensor core adds up
//              exactly the bf16 probabilities that it multiplies with V - and 15 unused columns)
//   [416,480)  Q_0, Q_1 (bf16 pairs, 32 columns each), written once by the softmax threads:
//              Q is the A operand of the first MMA from tensor memory, so the MMAs read only K and V tiles
//              from shared memory.
// The two halves of a tile double-buffer the scores: while the softmax threads work on
// half h the tensor core already runs O += P V of the other half and the next Q K^T into
// it.  The MMAs are issued in order, which is what makes the S/P aliasing safe: Q K^T for
// step n+2 is issued after the P V that reads the same columns.
// V tiles are consumed as an MN-major B operand, K tiles as a K-major one, so neither
// needs a transpose.
//
// Softmax arithmetic.  At head dim 64 every score costs 256 tensor flops and one
// exponential, and the special-function unit issues only 16 ex2 per clock per SM (the packed
// bf16x2 / f16x2 forms issue at half the rate, so they give the same 16 results per clock), half of
// what the tensor cores would need.  A fixed share of the exponentials of every row is therefore
// evaluated on the FMA pipes instead: round-to-nearest split x = n + f, |f| <= 1/2, a cubic
// for 2^f (relative error 7.5e-5, far below the bf16 rounding of P) and n added into the
// exponent field.  The share is a build-time constant, kFaPolyPairs of the 16 pairs of scores a
// thread handles per step; 7 measured best in the kernel (on register data alone, 4 warps per
// scheduler: 6 pairs take 182 clocks per 32 scores against 257 with the special-function unit only,
// 8 pairs 220).
// Shared memory: K ring, V ring, behind the V ring a 2 KB block that holds the ones column of
// the P V operand (see the kernel), and with two tiles room for the next queries and the rows on their way out.
//
// Key chunks.  All CTAs of a head stream the same K/V, but they drift apart, so their combined
// working set is the head's whole K/V; beyond about a quarter of the L2 that no longer stays
// resident and every CTA would pull its tiles from HBM (measured: 2.4 TB per launch at 520 K
// keys).  Long sequences are therefore swept in chunks of at most kFaChunkTiles key tiles, one
// launch per chunk: a chunk's K/V of one head (16 MiB) stays in L2 while all query blocks pass
// over it.  Every launch starts its accumulators from zero and, at its end, adds its partial
// output rows, row sums and reference to what the earlier chunks left in global memory (fp32,
// round to nearest; a few GB of traffic per launch).  That also bounds the chain of additions
// into one tensor-memory accumulator: carried through all 4067 key tiles of a 520 K-key sweep,
// the accumulator picked up an error that grew in proportion to the number of keys (2.9e-3 of
// the output's RMS at 252 K keys, 5.0e-3 at 520 K, against 2e-4 at 1.5 K).
//
// Softmax reference.  Any per-row constant m may be subtracted from the scores before the
// exponential: the division by the row sum removes it again.  It only has to keep 2^(s - m)
// inside the range of bf16 / fp32, it does not have to be the row maximum.  By Cauchy-Schwarz
// every score of a row is at most B = |q| max_k |k| (K carrying the softmax scale: base-2 units), so
// with m = B all exponents lie in [-2B, 0]; while 2B stays well inside the exponent range of
// fp32 nothing underflows, every probability keeps its 8 significant bits and the fp32
// accumulators their 24.  The pass that rounds K last leaves max_k |k|^2 per head behind, each
// softmax thread takes |q|^2 of its row while loading Q, and a warp pair whose rows all have
// B <= kFaFixedRefLimit runs the sweep with a constant reference (in fact with none: the constant
// cancels, see the kernel): no row maximum, no exchange between the two threads of a row, no
// rescaling, and - the softmax scale 1/sqrt(64) log2(e) arriving folded into K - no arithmetic
// between the tensor core's scores and the exponential.
// Rows with larger B need a reference other than zero, but seldom a running one: the largest score s0
// among the first 64 keys bounds the row maximum from below as B does from above, and wherever a
// whole number m lies close enough to both (fa_shift_up, fa_shift_down) it serves the whole sweep - the
// shifted form, at the cost of a subtraction or a clamp per score, both of which the bound spares the
// fixed form.  Trained projections attend that sharply (query weights x 16 on the generator's tokens:
// B up to 213): 31,751 rows went from 4.81 to 4.41 ms there.
// What remains takes the online form: base-2 softmax with a lazily updated reference
// maximum, the running output rescaled only when a row maximum grows far over the
// reference (the threads then first wait until the tile's last P V has retired).  All three equal
// the plain softmax up to rounding.
#include <type_traits>

#include "common.cuh"
#include "runtime.h"

namespace lv {

constexpr int kFaSoftmaxWarps = 16;
constexpr int kFaThreads = (kFaSoftmaxWarps + 3) * 32;
constexpr int kFaTileBytes = kFaTileKeys * 64 * 2;
constexpr int kFaOnesBytes = 16 * 128;  // 16 key rows of the ones column block
constexpr uint32_t kFaOCols = 80;  // 64 output channels, the row sum, 15 unused columns
// The online form's reference is set kFaAhead over the maximum found so far and serves until the row maximum lies more than
// kFaRescaleThreshold over it; then the row is rescaled, and its warp with it, which waits for the tensor core and reads
// and writes its output.  Sums over 2^22 keys times |v| <= 2^20 stay below 2^82; keys more than 126 - 32 under the maximum
// are lost, 2^-72 of the row at most.  (Layer of 31,751 rows at query weights x 64, all of them online: 5.30 ms with the
// reference at the maximum and rescaling beyond 2^8, 5.23 beyond 2^22, 5.13 with the reference 16 ahead, 4.95 as it stands.)
constexpr float kFaRescaleThreshold = 40.0f;
constexpr float kFaAhead = 32.0f;
// Largest Cauchy-Schwarz bound B on the base-2 scores of a row for which the fixed reference is
// used.  With the reference left out the probabilities lie in [2^-B, 2^B]: at B = 80 their products
// with |v| >= 2^-20 are normal fp32 numbers (>= 2^-100), and a row sum over 2^20 keys times
// |v| <= 2^20 stays below 2^120, inside fp32; the polynomial exponential is valid to +-120.
#ifndef LV_FA_FIXED_REF_LIMIT
#define LV_FA_FIXED_REF_LIMIT 80.0f
#endif
constexpr float kFaFixedRefLimit = LV_FA_FIXED_REF_LIMIT;
// Of the 16 pairs of scores a thread handles per step, this many take the polynomial exponential
// (fixed-reference form only, where every argument lies in [-kFaFixedRefLimit, kFaFixedRefLimit]).
#ifndef LV_FA_POLY_PAIRS
#define LV_FA_POLY_PAIRS 7
#endif
constexpr int kFaPolyPairs = LV_FA_POLY_PAIRS;
// The same in the shifted-reference form, whose polynomial pairs also need a clamp and whose other
// pairs a subtraction, and which takes the polynomial of degree 6 (the running maximum that served these
// rows before is as good as the special-function unit).  Layers at query weights x 16, 2 / 3 / 4 / 5 pairs: 10,410 rows 557 / 543 /
// 544 / 541 us, 31,751 4.17 / 4.07 ms, 62,460 16.10 / 15.84 / 16.14 / 16.00; x 8: 31,751 3.83 / 3.80, 62,460 14.56 / 14.51 / 14.61 /
// 14.61.  (Three measured no better than two while the waits had their loops in line.)
#ifndef LV_FA_SHIFT_POLY_PAIRS
#define LV_FA_SHIFT_POLY_PAIRS 3
#endif
constexpr int kFaShiftPolyPairs = LV_FA_SHIFT_POLY_PAIRS;
// Shifted reference m of a row with score bound B and a known score s0, both limits by the sequence's length (its binary
// logarithm, rounded up).  B - m <= fa_shift_up: row sums over that many keys, times the head's largest |v| where that is over
// 2^20, stay below 2^126.  m - s0 <= fa_shift_down: what lies more than 126 under m is off by up to 2^-126 a key (flushed
// to zero by the special-function unit, held up at 2^-126 by the polynomial's clamp), the row's largest probability
// is at least 2^-fa_shift_down, so all such keys together are off by 2^-24 of the row's mass at most - no more than one
// fp32 rounding of the row sum.  (With 84 up, the limit of 2^22 keys and |v| <= 2^20, at every length, a seventh of the
// 256-row tiles of 31,751 rows at query weights x 16 had a row in the online form, a tenth with 91: 4.53 -> 4.49 ms.)
static float key_bits(long long keys) {
  int bits = 0;
  while ((1ll << bits) < keys) ++bits;
  return (float)bits;
}
__device__ __forceinline__ float fa_shift_up(float bits, float v_max) {
  const int v_bits = (int)(__float_as_uint(v_max) >> 23) - 126;  // |v| < 2^v_bits; 129 where it is infinite
  return 126.0f - bits - fmaxf((float)v_bits, 20.0f);
}
__device__ __forceinline__ float fa_shift_down(float bits) { return 126.0f - 24.0f - bits; }

// The jobs of a launch, one query block of one head of one sequence each, query blocks fastest.  Those that the last
// round would leave alone on the chip are split along the keys: ids from `full` on are (job, part) with
// `parts` parts to a job, and leave partial rows for combine_parts_kernel.
struct FaJobs {
  int q_first, q_blocks, heads, count, full, parts;
  float* o;   // [slot][16][256][4] partial output rows, four channels at a time, slot = id - full
  float* ml;  // [slot][256]{reference, row sum}
  int* taken; // how many jobs beyond the CTAs' first ones have been taken; zero when the launch starts
};
struct FaTiles {
  int begin, end;  // a job's key tiles
};
__device__ __forceinline__ FaTiles fa_tiles(const FaJobs& jobs, int id, int tile_begin, int tile_end) {
  const int slot = id - jobs.full;
  if (slot < 0) return FaTiles{tile_begin, tile_end};
  const int part = slot % jobs.parts;
  return FaTiles{(int)((long long)tile_end * part / jobs.parts), (int)((long long)tile_end * (part + 1) / jobs.parts)};
}
struct FaJob {
  int q_block, head, seq, slot;  // slot < 0: a whole job
};
__device__ __forceinline__ FaJob fa_job(const FaJobs& jobs, int id) {
  const int slot = id - jobs.full, job = slot < 0 ? id : jobs.full + slot / jobs.parts;
  const int rest = job / jobs.q_blocks;
  return FaJob{jobs.q_first + job % jobs.q_blocks, rest % jobs.heads, rest / jobs.heads, slot};
}
// This thread's 32 channels of row r (0..255) of the job; rows side by side, 4 channels of each at a time, so that a warp's store
// is 512 bytes in a row (a row of its own after the other they took 2.4 to 3.8 us).
__device__ __forceinline__ void fa_store_part(const FaJobs& split, int slot, int r, int c, const uint32_t (&acc)[32], float scale,
                                              float m_ref, float row_sum) {
  float4* dst = reinterpret_cast<float4*>(split.o) + ((size_t)slot * 16 + c * 8) * 256 + r;
#pragma unroll
  for (int i = 0; i < 8; ++i)
    dst[i * 256] = make_float4(__uint_as_float(acc[4 * i]) * scale, __uint_as_float(acc[4 * i + 1]) * scale,
                         __uint_as_float(acc[4 * i + 2]) * scale, __uint_as_float(acc[4 * i + 3]) * scale);
  if (c == 0) *reinterpret_cast<float2*>(split.ml + ((size_t)slot * 256 + r) * 2) = make_float2(m_ref, row_sum);
}

template <int kTiles, int kStages>
struct FaBarriers {
  uint64_t k_full[kStages], k_empty[kStages];
  uint64_t v_full[kStages], v_empty[kStages];
  uint64_t q_ready[kTiles], s_full[kTiles][2], p_ready[kTiles][2], pv_done[kTiles], o_done[kTiles], o_free[kTiles];
  uint64_t teardown[kTiles];
  uint64_t q_full[kTiles], q_empty[kTiles];  // the queries' way through shared memory
  uint64_t job_full[2], job_empty[2];
  int job[2];  // the CTA's next jobs
  uint32_t tmem_base;
  uint32_t abort_flag;
};
// what the two warps of a pair tell each other about their 32 rows: [tile][warp of the pair][row]
template <int kTiles>
struct FaPairs {
  float first_max[kTiles][2][128];
  float row_max[2][kTiles][2][128];  // of either half of a key tile
  uint32_t left[kTiles][2][4];       // [tile][warp of the pair][quarter]: has given up and gone
};
// What differs between the CTA of two query tiles (one CTA per SM) and that of one (two per SM).
template <int kTiles>
struct FaShape {
  static constexpr int kSoftmaxWarps = 8 * kTiles;
  static constexpr int kThreads = (kSoftmaxWarps + 1 + kTiles) * 32;
  static constexpr int kStages = kTiles == 2 ? 4 : 3;
  static constexpr uint32_t kTmemCols = 256 * kTiles;
  static constexpr uint32_t kColS = 0, kColO = 128 * kTiles, kColQ = (128 + 80) * kTiles;
  // queries on their way in and rows on their way out: where V and K tiles will be and have been, or, where the ring goes on
  // from job to job, of their own
  static constexpr int kRowBytes = kTiles == 2 ? 2 * kTiles * kFaTileBytes : 0;
  static constexpr int kSmemBytes =
      2 * kStages * kFaTileBytes + kRowBytes + kFaOnesBytes + (int)sizeof(FaPairs<kTiles>) + 512 + 1024;
};

constexpr int kFaAloneBytes = 120 * 1024;  // shared memory that keeps a second CTA off the SM
static_assert(kFaAloneBytes >= FaShape<1>::kSmemBytes, "");

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 2^d for a whole number d <= 0, exact; zero under 2^-126.
__device__ __forceinline__ float exp2_whole(float d) { return __uint_as_float((uint32_t)((int)fmaxf(d, -127.0f) + 127) << 23); }

// 2^(x - m) for a pair of arguments on the FMA pipes, `magic` = 1.5 * 2^23 - m with m a whole number.
// Adding it rounds x to the nearest integer and leaves n = that integer - m in the low mantissa
// bits; the fraction's power comes from a polynomial fitted on [-1/2, 1/2] and n is added to the exponent
// field; of a NaN that makes a number beyond the largest bf16, so its row still ends up not finite.
// Valid for x - m in [-126, 120].  The cubic is good to 7.5e-5 relative.  With kFull the degree is 6 and
// the result, rounding included, within 6.6e-8 of 2^(x - m): closer than the special-function unit,
// whose ex2.approx was measured at up to 1.45e-7 (5.4e-8 against 2.6e-8 in the mean square).
template <bool kFull>
__device__ __forceinline__ float2 poly_exp2_pair(float2 x, float2 magic, float2 neg_magic) {
  const float2 t = __fadd2_rn(x, magic);
  const float2 n = __fadd2_rn(t, neg_magic);
  const float2 f = __ffma2_rn(n, make_float2(-1.0f, -1.0f), x);
  auto horner = [&](float2 p, float c) { return __ffma2_rn(p, f, make_float2(c, c)); };
  float2 p;
  if constexpr (kFull) {
    p = horner(make_float2(1.5820509e-4f, 1.5820509e-4f), 1.341820345e-3f);
    p = horner(p, 9.617063217e-3f);
    p = horner(p, 5.55027239e-2f);
    p = horner(p, 0.2402265519f);
    p = horner(p, 0.6931472421f);
    p = horner(p, 1.0f);
  } else {
    p = horner(make_float2(0.0551716648f, 0.0551716648f), 0.2426111251f);
    p = horner(p, 0.6932609677f);
    p = horner(p, 0.9999280572f);
  }
  float2 r;
  r.x = __uint_as_float(__float_as_uint(p.x) + (__float_as_uint(t.x) << 23));
  r.y = __uint_as_float(__float_as_uint(p.y) + (__float_as_uint(t.y) << 23));
  return r;
}
__device__ __forceinline__ float2 poly_exp2_pair(float2 x) {
  return poly_exp2_pair<false>(x, make_float2(12582912.0f, 12582912.0f), make_float2(-12582912.0f, -12582912.0f));
}

// Wait until the most recent loads into a ring (up to one per stage) have landed.
// `issued` counts the loads issued into the ring so far; load i uses stage i % kStages and
// completes the phase with parity (i / kStages) & 1.  Not sensitive to the abort flag: the
// copies are in flight and must finish before the shared memory can be given up.
template <int kStages>
__device__ __forceinline__ void drain_ring(uint64_t* full, uint32_t issued, uint32_t* status) {
  const uint32_t n_drain = issued < (uint32_t)kStages ? issued : (uint32_t)kStages;
  for (uint32_t i = 0; i < n_drain; ++i) {
    const uint32_t idx = issued - 1 - i;
    const long long t0 = clock64();
    while (!mbar_try_wait(&full[idx % kStages], (idx / kStages) & 1u)) {
      if (clock64() - t0 > kTimeoutCycles) { atomicOr(status, kStatusTimeout); break; }
    }
  }
}

// Exponentials of 32 scores of a row, which arrive scaled, with no reference to subtract: p = 2^s, packed to bf16 pairs (the
// row sum is formed by the tensor core from these rounded values).  The first kPoly of the 16 pairs take the
// polynomial on the FMA pipes (callers guarantee arguments above -120 for them), the others the
// special-function unit.
template <int kPoly>
__device__ __forceinline__ void exp2_chunk(const uint32_t (&s)[32], uint32_t (&packed)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float2 x = make_float2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1]));
    float2 p;
    if (i < kPoly) {
      p = poly_exp2_pair(x);
    } else {
      p.x = fast_exp2(x.x);
      p.y = fast_exp2(x.y);
    }
    packed[i] = pack_bf16(p.x, p.y);
  }
}

// The same for a reference m that is a whole number, |m| <= 2^20: p = 2^(s - m).  For the polynomial
// pairs the subtraction is free, m being part of the constant that rounds to the nearest integer; they
// clamp at m - 126, below which the exponent field would wrap.
template <int kPoly>
__device__ __forceinline__ void exp2_chunk_shifted(const uint32_t (&s)[32], float m, uint32_t (&packed)[16]) {
  const float2 neg_m = make_float2(-m, -m);
  const float floor_s = m - 126.0f, magic = 12582912.0f - m;  // exact: 1.5 * 2^23 -+ 2^20 keeps its exponent
  const float2 magic2 = make_float2(magic, magic), neg_magic2 = make_float2(-magic, -magic);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float2 p;
    if (i < kPoly) {
      const float2 x = make_float2(fmax_nan(__uint_as_float(s[2 * i]), floor_s), fmax_nan(__uint_as_float(s[2 * i + 1]), floor_s));
      p = poly_exp2_pair<true>(x, magic2, neg_magic2);
    } else {
      const float2 x = __fadd2_rn(make_float2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), neg_m);
      p.x = fast_exp2(x.x);
      p.y = fast_exp2(x.y);
    }
    packed[i] = pack_bf16(p.x, p.y);
  }
}

// Largest of a thread's 32 scores.
__device__ __forceinline__ float max32(const uint32_t (&s)[32]) {
  float mx[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const uint32_t* sc = &s[g * 8];
    mx[g] = fmax3(__uint_as_float(sc[0]), __uint_as_float(sc[1]), __uint_as_float(sc[2]));
    mx[g] = fmax3(mx[g], __uint_as_float(sc[3]), __uint_as_float(sc[4]));
    mx[g] = fmax3(mx[g], __uint_as_float(sc[5]), __uint_as_float(sc[6]));
    mx[g] = fmaxf(mx[g], __uint_as_float(sc[7]));
  }
  return fmaxf(fmax3(mx[0], mx[1], mx[2]), mx[3]);
}

// The two warps of one (tile, lane quarter).  In a job that has such barriers (one, and in the online form one a step) a warp that
// gives up goes on to meet its partner at all of them, so no step has to ask.  A warp that leaves between jobs says so and
// arrives without waiting, which lets the partner through the next job's first barrier, behind which it finds out.
__device__ __forceinline__ void pair_barrier(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_barrier_leave(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// (out of line: it runs only where a wait was given up)
__device__ __noinline__ void meet_partner(int id, int met, int n_steps) {
  for (; met < n_steps; ++met) pair_barrier(id);
}

// kFirst / kLast: this launch holds the first / the last key chunk of the sweep.
// kTiles: query tiles of the CTA.
template <int kTiles, bool kFirst, bool kLast>
__global__ void __launch_bounds__(FaShape<kTiles>::kThreads, kTiles == 2 ? 1 : 2)
flash_attention_kernel(const __grid_constant__ CUtensorMap tmap_qkv, __nv_bfloat16* __restrict__ o,
                       float* __restrict__ o_state, float* __restrict__ ml_state, const float* __restrict__ kv_max,
                       float key_bits, int seq_len, int dim, int tile_begin, int tile_end, FaJobs jobs, uint32_t* status, Stamp stamp) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* smem_k = smem;
  using Shape = FaShape<kTiles>;
  constexpr int kStages = Shape::kStages;
  uint8_t* smem_v = smem_k + kStages * kFaTileBytes;
  uint8_t* smem_ones = smem_v + kStages * kFaTileBytes;  // see below
  uint8_t* smem_rows = smem_ones + kFaOnesBytes;
  uint8_t* smem_q = kTiles == 2 ? smem_rows : smem_ones - kFaTileBytes;  // [tile], queries; with one tile until V needs its last stage
  uint8_t* smem_o = kTiles == 2 ? smem_rows + kTiles * kFaTileBytes : smem_k;  // [warp] 32 rows of 64 bytes
  FaPairs<kTiles>* pairs = reinterpret_cast<FaPairs<kTiles>*>(smem_rows + Shape::kRowBytes);
  FaBarriers<kTiles, kStages>* bars = reinterpret_cast<FaBarriers<kTiles, kStages>*>(pairs + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr bool first_chunk = kFirst;
  constexpr bool last_chunk = kLast;
  // Every role walks over the CTA's jobs by itself; where a CTA has only one it is the block's own.
  constexpr bool kJobs = kTiles == 2;
  // The first is the block's own too, the others come off a counter, so that CTAs whose rows need a slower form
  // of the softmax take fewer.
  const int id0 = kJobs ? (int)blockIdx.x : 0, id_end = kJobs ? jobs.count : 1;
  auto job_at = [&](int id) {
    if constexpr (kJobs) return fa_job(jobs, id);
    else return FaJob{(int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z, -1};
  };
  // A job covers key tiles [begin, end) of ceil(seq_len / 128); its step n is half n % 2 of its tile n / 2.
  auto tiles_at = [&](int id) {
    if constexpr (kJobs) return fa_tiles(jobs, id, tile_begin, tile_end);
    else return FaTiles{tile_begin, tile_end};
  };
  auto keys_of = [&](const FaTiles& kv) { return (kLast ? seq_len : kv.end * kFaTileKeys) - kv.begin * kFaTileKeys; };  // at least one
  // a last key tile with at most 64 keys has no second half
  auto steps_of = [&](const FaTiles& kv) { return min(2 * (kv.end - kv.begin), (keys_of(kv) + 63) / 64); };
  // a tile without rows takes no part
  auto tile_live = [&](int id, int t) { return t == 0 || job_at(id).q_block * (128 * kTiles) + 128 < seq_len; };

  // (by many threads at once: a CTA of a short sequence lives for few microseconds)
  if (threadIdx.x < kStages) {
    mbar_init(&bars->k_full[threadIdx.x], 1);
    mbar_init(&bars->k_empty[threadIdx.x], kTiles);  // every tile's MMA issuer releases a stage
    mbar_init(&bars->v_full[threadIdx.x], 1);
    mbar_init(&bars->v_empty[threadIdx.x], kTiles);
    mbar_fence_init();
  } else if (threadIdx.x >= 32 && threadIdx.x < 32 + 2 * kTiles) {
    const int t = (threadIdx.x - 32) >> 1, h = threadIdx.x & 1;
    mbar_init(&bars->s_full[t][h], 1);
    mbar_init(&bars->p_ready[t][h], 8);
    if (h == 0) {
      mbar_init(&bars->q_ready[t], 8);
      mbar_init(&bars->o_done[t], 1);
      mbar_init(&bars->teardown[t], 1);
      mbar_init(&bars->q_full[t], 1);
    } else {
      mbar_init(&bars->o_free[t], 8);
      mbar_init(&bars->pv_done[t], 1);
      mbar_init(&bars->q_empty[t], 8);
    }
    mbar_fence_init();
  } else if (threadIdx.x == 96) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->job_full[i], 1);
      mbar_init(&bars->job_empty[i], Shape::kSoftmaxWarps + kTiles);
    }
    mbar_fence_init();
    bars->abort_flag = 0;
    for (int i = 0; i < 8 * kTiles; ++i) (&pairs->left[0][0][0])[i] = 0u;
    tma_prefetch_desc(&tmap_qkv);
  }
  // The row sums come out of the second MMA: its B operand is 80 columns wide, V's 64 channels and,
  // one descriptor stride further on, a block whose first column is 1 and whose other columns are 0,
  // so accumulator column 64 collects sum_k P[row, k] of exactly the bf16 probabilities that multiply
  // V.  The block is 16 key rows (one instruction's worth) laid out like a V tile (128-byte rows,
  // 16-byte chunks XOR-swizzled with the row index modulo 8); every instruction's descriptor carries
  // the stride from its own V rows to this one block.
  if (threadIdx.x < kFaOnesBytes / 16) {
    const int r = threadIdx.x >> 3, chunk = threadIdx.x & 7;  // 128-byte row, 16-byte chunk within it
    const uint32_t first = chunk == (r & 7) ? 0x00003f80u : 0u;  // bf16 1.0 in logical column 0
    reinterpret_cast<uint4*>(smem_ones)[threadIdx.x] = make_uint4(first, 0u, 0u, 0u);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes, read by the MMA
  constexpr int kIssuerWarp = Shape::kSoftmaxWarps;  // of tile 0; then the TMA producer, the issuer of tile 1
  if (warp == kIssuerWarp) {
    tmem_alloc(&bars->tmem_base, Shape::kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = bars->tmem_base;
  const WaitCtl ctl{&bars->abort_flag, status};
  const Span span(stamp);

  // `turn` (0..3, in the low bits): the CTA's jobs so far; id_end or more where there is no further one, or on a wait given up
  auto job_after = [&](uint32_t turn, bool one_lane, bool& ok) -> int {
    if constexpr (kJobs) {
      ok = one_lane ? mbar_wait(&bars->job_full[turn & 1u], turn >> 1 & 1u, ctl) : mbar_wait_warp(&bars->job_full[turn & 1u], turn >> 1 & 1u, ctl);
      if (!ok) return id_end;
      int id = *reinterpret_cast<volatile int*>(&bars->job[turn & 1u]);
      // (from one lane, so that the compiler knows it to be the same in all and a job's loops not to diverge)
      if (!one_lane) id = __shfl_sync(0xffffffffu, id, 0);
      if (one_lane || lane == 0) mbar_arrive(&bars->job_empty[turn & 1u]);
      return id;
    } else {
      return id_end;
    }
  };
  if (warp == kIssuerWarp + 1) {
    // ------------------------------------------------------------------ TMA producer
    if (elect_one()) {
      uint32_t k_issued = 0, v_issued = 0, phase = 0;
      int stage = 0;
      bool ok = true;
      uint32_t turn = 0;
      uint32_t q_sent[kTiles] = {};
      // A job's queries, of the tiles that have rows, once the ones before have been read.
      auto send_q = [&](int id) -> bool {
        const FaJob job = job_at(id);
#pragma unroll
        for (int t = 0; t < kTiles; ++t) {
          if (!tile_live(id, t)) continue;
          if (q_sent[t] != 0 && !mbar_wait(&bars->q_empty[t], (q_sent[t] - 1) & 1u, ctl)) return false;
          mbar_expect_tx(&bars->q_full[t], kFaTileBytes);
          tma_load_2d(smem_q + t * kFaTileBytes, &tmap_qkv, &bars->q_full[t], job.head * 64, job.seq * seq_len + (job.q_block * kTiles + t) * 128);
          ++q_sent[t];
        }
        return true;
      };
      if (id0 < id_end) ok = send_q(id0);
      for (int id = id0; id < id_end && ok;) {
        const FaJob job = job_at(id);
        const FaTiles kv = tiles_at(id);
        int next_id = id_end;
        const int row0 = job.seq * seq_len, col = job.head * 64;
        for (int j = kv.begin; j < kv.end; ++j) {
          if (kJobs && j == max(kv.begin, kv.end - 2)) {
            // The next job, to everybody; late, so that it is not kept waiting here while another CTA has nothing to do, and
            // early enough for the counter's answer to come before these tiles are through.
            if (turn >= 2 && !mbar_wait(&bars->job_empty[turn & 1u], (turn >> 1 & 1u) ^ 1u, ctl)) { ok = false; break; }
            next_id = (int)gridDim.x + atomicAdd(jobs.taken, 1);
            bars->job[turn & 1u] = next_id;
            mbar_arrive(&bars->job_full[turn & 1u]);
            ++turn;
            if (next_id < id_end && !send_q(next_id)) { ok = false; break; }
          }
          if (!mbar_wait(&bars->k_empty[stage], phase ^ 1u, ctl)) { ok = false; break; }
          mbar_expect_tx(&bars->k_full[stage], kFaTileBytes);
          tma_load_2d(smem_k + stage * kFaTileBytes, &tmap_qkv, &bars->k_full[stage], dim + col, row0 + j * kFaTileKeys);
          ++k_issued;
          if (!mbar_wait(&bars->v_empty[stage], phase ^ 1u, ctl)) { ok = false; break; }
          if (!kJobs && v_issued == kStages - 1 && !mbar_wait(&bars->q_ready[0], 0, ctl)) { ok = false; break; }  // the queries lie there
          mbar_expect_tx(&bars->v_full[stage], kFaTileBytes);
          tma_load_2d(smem_v + stage * kFaTileBytes, &tmap_qkv, &bars->v_full[stage], 2 * dim + col, row0 + j * kFaTileKeys);
          ++v_issued;
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        id = next_id;
      }
#pragma unroll
      for (int t = 0; t < kTiles; ++t) drain_ring<1>(&bars->q_full[t], q_sent[t], status);
      // every load issued by this thread must have landed before the CTA may exit
      drain_ring<kStages>(bars->k_full, k_issued, status);
      drain_ring<kStages>(bars->v_full, v_issued, status);
    }
  } else if (warp == kIssuerWarp || (kTiles == 2 && warp == kIssuerWarp + 2)) {
    // ------------------------------------------------------------------ MMA issuer of tile t
    if (elect_one()) {
      const int t = warp == kIssuerWarp ? 0 : 1;
      constexpr uint32_t idesc_qk = umma_idesc_bf16(128, 64, false, false);
      constexpr uint32_t idesc_pv = umma_idesc_bf16(128, kFaOCols, false, true);
      const uint32_t s_col = tmem_base + Shape::kColS + t * 128;
      const uint32_t o_col = tmem_base + Shape::kColO + t * kFaOCols;
      const uint32_t q_col = tmem_base + Shape::kColQ + t * 32;
      // S_h = Q (tensor memory) x K[64h .. 64h+63]^T (shared memory, K-major); 4 steps of 16 channels
      // the descriptors are linear in the shared-memory address (its 16-byte units sit in the low
      // bits and cannot carry out of their field), so a stage / half is one addition away
      const uint64_t k_desc0 = smem_desc_sw128(smem_u32(smem_k), 16, 1024);
      const uint64_t v_desc0 = smem_desc_sw128(smem_u32(smem_v), kStages * kFaTileBytes, 1024);
      // x 16-byte units into the V ring: the address grows and the stride to the ones block (bits
      // 16-29, never below zero because that block lies behind the ring) shrinks by the same amount
      auto v_desc_at = [&](uint32_t x) { return v_desc0 + (uint64_t)x - ((uint64_t)x << 16); };
      auto issue_qk = [&](int h, int stage) {
        const uint64_t b_desc = k_desc0 + (uint64_t)((stage * kFaTileBytes + h * 8192) >> 4);
#pragma unroll
        for (int k = 0; k < 4; ++k) umma_ts(s_col + h * 64, q_col + k * 8, b_desc + 2 * k, idesc_qk, k != 0 ? 1u : 0u);
        umma_commit(&bars->s_full[t][h]);
      };
      // the rings and the barriers' phases go on from job to job
      int stage = 0;
      uint32_t phase = 0, round = 0;              // round: jobs of this tile so far
      uint32_t turn = 0;                          // parities of the two halves' barriers when a job starts, a bit each
      bool ok = true;
      uint32_t jobs_done = 0;
      for (int id = id0; id < id_end && ok; id = ok ? job_after(jobs_done++, true, ok) : id_end) {
        const FaTiles kv = tiles_at(id);
        const int n_kv = kv.end - kv.begin, n_steps = steps_of(kv);
        if (!tile_live(id, t)) {
          for (int j = 0; j < n_kv && ok; ++j) {  // the stages go by
            ok = mbar_wait(&bars->k_full[stage], phase, ctl);
            if (ok) mbar_arrive(&bars->k_empty[stage]);
            if (ok) ok = mbar_wait(&bars->v_full[stage], phase, ctl);
            if (ok) mbar_arrive(&bars->v_empty[stage]);
            if (++stage == kStages) { stage = 0; phase ^= 1u; }
          }
          continue;
        }
        ok = mbar_wait(&bars->q_ready[t], round & 1u, ctl);
        if (ok) ok = mbar_wait(&bars->k_full[stage], phase, ctl);
        if (ok) {
          tc_fence_after();
          issue_qk(0, stage);
          if (n_steps > 1) issue_qk(1, stage);
          umma_commit(&bars->k_empty[stage]);
        }
        for (int j = 0; j < n_kv && ok; ++j) {
          int next_stage = stage + 1;
          uint32_t next_phase = phase;
          if (next_stage == kStages) { next_stage = 0; next_phase ^= 1u; }
          const bool last = j + 1 == n_kv;
          if (!mbar_wait(&bars->v_full[stage], phase, ctl)) { ok = false; break; }
          if (!last && !mbar_wait(&bars->k_full[next_stage], next_phase, ctl)) { ok = false; break; }
          // the previous job's output has been read
          if (j == 0 && round != 0 && !mbar_wait(&bars->o_free[t], (round - 1) & 1u, ctl)) { ok = false; break; }
          for (int h = 0; h < 2; ++h) {
            const int n = 2 * j + h;
            if (n == n_steps) break;
            if (!mbar_wait(&bars->p_ready[t][h], ((turn >> h) ^ (uint32_t)j) & 1u, ctl)) { ok = false; break; }
            tc_fence_after();
            // 64 keys of V_j (64 rows of 128 bytes = 8192 bytes per half), 16 keys per instruction:
            // 8 TMEM columns of P (keys 0-31 in columns [0,16) of the half, keys 32-63 in [32,48)),
            // 2048 bytes of V; second 64-column block of B = the ones block
            const uint32_t v_at = (uint32_t)((stage * kFaTileBytes + h * 8192) >> 4);
#pragma unroll
            for (int k = 0; k < 4; ++k)
              umma_ts(o_col, s_col + h * 64 + (k >> 1) * 32 + (k & 1) * 8, v_desc_at(v_at + 128 * k), idesc_pv,
                      (j | h | k) != 0 ? 1u : 0u);  // every job starts its accumulators from zero
            if (n + 2 < n_steps) {
              issue_qk(h, next_stage);  // where these probabilities were
            } else {
              // no Q K^T follows whose completion would tell the softmax threads that this P V has retired; they
              // ask for the last but one (a job of one step counts too)
              if (n + 2 == n_steps || n_steps == 1) umma_commit(&bars->pv_done[t]);
              if (n + 1 == n_steps) umma_commit(&bars->o_done[t]);
            }
          }
          if (!ok) break;
          umma_commit(&bars->v_empty[stage]);
          if (!last) umma_commit(&bars->k_empty[next_stage]);
          stage = next_stage;
          phase = next_phase;
        }
        turn ^= ((uint32_t)(n_steps + 1) >> 1 & 1u) | ((uint32_t)n_steps & 2u);
        ++round;
      }
      if (!ok) {
        umma_commit(&bars->teardown[t]);
        const long long t0 = clock64();
        while (!mbar_try_wait(&bars->teardown[t], 0)) {
          if (clock64() - t0 > kTimeoutCycles) break;
        }
      }
    }
  } else if (warp < Shape::kSoftmaxWarps) {
    // ------------------------------------------------------------------ softmax warps
    const int t = warp >> 3;
    const int c = (warp >> 2) & 1;
    const uint32_t quarter = warp & 3u;
    const int row_in_tile = (int)quarter * 32 + lane;
    const uint32_t lane_base = (quarter * 32u) << 16;
    const uint32_t s_addr = tmem_base + lane_base + Shape::kColS + t * 128;
    const uint32_t o_row = tmem_base + lane_base + Shape::kColO + t * kFaOCols, o_addr = o_row + c * 32;

    auto row_of = [&](const FaJob& job) { return job.q_block * (128 * kTiles) + t * 128 + row_in_tile; };  // within the sequence
    // The queries come by TMA: loaded row by row, every load of a warp touches 32 lines, 4096 in all for two tiles, 2 us
    // (a CTA of one tile, four frames of 16 x 16: layer 32.3 -> 31.7 us; local half of 200 frames of 28 x 37 5.18 -> 5.15
    // ms).  This thread's half (32 channels) of its row goes to tensor memory, in the place of the queries before, all of
    // whose Q K^T must have retired.  Returns the Cauchy-Schwarz bound on the whole row's scores (K carries the
    // softmax scale, so they are in base-2 units already), or -1 where a wait was given up.
    auto take_q = [&](const FaJob& job, uint32_t parity) -> float {
      const float k_norm2 = kv_max[job.seq * 2 * (dim / 64) + job.head];
      if (!mbar_wait_warp(&bars->q_full[t], parity, ctl)) return -1.0f;
      const bool live = row_of(job) < seq_len;
      uint32_t qreg[16];
      float q_norm2 = 0.0f;
#pragma unroll
      for (int i = 0; i < 8; ++i) {  // in the same order in both threads of a row, so that they find the same bound
        uint4 v = *reinterpret_cast<const uint4*>(smem_q + t * kFaTileBytes + row_in_tile * 128 + ((i ^ (row_in_tile & 7)) << 4));
        if (!live) v = make_uint4(0u, 0u, 0u, 0u);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          q_norm2 = fmaf(bf16_hi(w[e]), bf16_hi(w[e]), fmaf(bf16_lo(w[e]), bf16_lo(w[e]), q_norm2));
          if (i < 4 || c == 1) qreg[4 * (i & 3) + e] = w[e];
        }
      }
      tmem_st16(tmem_base + lane_base + Shape::kColQ + t * 32 + c * 16, qreg);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&bars->q_ready[t]);
        if (kJobs) mbar_arrive(&bars->q_empty[t]);
      }
      return sqrtf(q_norm2 * k_norm2);
    };
    bool ok = true;
    // Phases that go on from job to job, a bit each: of half 0's and half 1's barriers when a job starts, of the job's own
    // barriers;
    uint32_t turn = 0;  // and from bit 4 on the CTA's jobs so far
    auto next_job = [&](int id) -> int {  // the first from `id` on that has rows in this tile
      while (id < id_end && !tile_live(id, t)) {
        id = job_after(turn >> 4, false, ok);
        turn += 16u;
      }
      return id;
    };
    const int barrier_id = 1 + t * 4 + (int)quarter;
    int id = next_job(id0);
    float score_bound = 0.0f;
    if (id < id_end) {
      score_bound = take_q(job_at(id), 0u);
      if (score_bound < 0.0f) id = id_end;
    }
    while (id < id_end) {
      const FaTiles kv = tiles_at(id);
      const int n_keys = keys_of(kv), n_steps = steps_of(kv), last = kv.end - kv.begin - 1;
      const bool warp_live = kTiles * 128 * job_at(id).q_block + t * 128 + (int)quarter * 32 < seq_len;
      // both warps of a pair vote over the same 32 rows, so they agree on the form they run
      const bool fixed_ref = __all_sync(0xffffffffu, score_bound <= kFaFixedRefLimit ? 1 : 0) != 0;
      float m_ref = -INFINITY;  // reference, in the scores' own (base-2) units
      auto masked = [&](uint32_t (&s)[32], int valid) {
#pragma unroll
        for (int k = 0; k < 32; ++k)
          if (k >= valid) s[k] = 0xff800000u;  // -inf: probability 0
      };
      auto scores_in = [&](int h, uint32_t parity) -> bool { return mbar_wait_warp(&bars->s_full[t][h], parity & 1u, ctl); };
      // of half h of the job's key tile j
      auto scores_of = [&](int h, int j) -> bool { return scores_in(h, kJobs ? (turn >> h) ^ (uint32_t)j : (uint32_t)j); };
      auto give_p = [&](int h, uint32_t count) {
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_count(&bars->p_ready[t][h], count);
      };
      // The sweep of a row whose reference stays what it is: `exps` turns 32 scores into 16 bf16 pairs.  The two
      // warps of a pair need nothing from each other here, so in the CTA of two tiles (kWide) each takes every
      // other step whole - one wait and one hand-over for 64 scores a thread where sharing a step pays for
      // both twice: 1.85 -> 1.79 ms at 22 K rows, 3.73 -> 3.62 at 32 K, 11.2 -> 10.7 at 52 K, 28.9 -> 27.9 at
      // 83 K.  With one tile, where a sweep is short, sharing gives the shorter step: 286 us either way at 8.3
      // K rows, 20.4 against 21.7 at 1.8 K.  (Loading 16 or 32 scores ahead of the exponentials
      // measured the same or, where it spilled, less.)
      // Only the last tile of a job can reach past the sequence, so the steps before it need no masking;
      // shared steps are written out per half so that barrier and tensor-memory addresses are constants of
      // the loop.
      constexpr bool kWide = kTiles == 2;
      auto sweep = [&](auto exps) {
        auto step = [&](uint32_t parity, int h, bool may_mask) -> bool {
          if (!scores_in(h, parity)) return false;
          tc_fence_after();
#pragma unroll
          for (int i = 0; i < (kWide ? 2 : 1); ++i) {
            const int g = kWide ? i : c;  // columns [32 g, 32 g + 32) of the half
            const uint32_t addr = s_addr + h * 64 + g * 32;
            uint32_t s[32], packed[16];
            tmem_ld32(addr, s);
            tmem_ld_wait();
            const int valid = may_mask ? n_keys - (2 * last + h) * 64 - g * 32 : 32;
            if (may_mask && valid < 32) {
              masked(s, valid);
              exps(s, packed, std::true_type{});
            } else {
              exps(s, packed, std::false_type{});
            }
            tmem_st16(addr, packed);  // over the start of the columns just read
          }
          give_p(h, kWide ? 2 : 1);
          return true;
        };
        if constexpr (kWide) {
          // the counter carries the parity
          uint32_t j = (turn >> c) & 1u;
          const uint32_t end = j + (uint32_t)last;
          for (; j < end && ok; ++j) ok = step(j, c, false);
          if (ok && 2 * last + c < n_steps) ok = step(end, c, true);
        } else {
          for (uint32_t j = 0; j < (uint32_t)last && ok; ++j) ok = step(j, 0, false) && step(j, 1, false);
          if (ok) ok = step(last, 0, true) && (2 * last + 1 == n_steps || step(last, 1, true));
        }
      };
      if (!warp_live) {
        // ---- no live row in this warp (nor in its partner): the issuer needs the hand-over, nobody the result
        for (int n = c; n < n_steps && ok; n += 2) {
          ok = scores_of(c, n >> 1);
          if (ok && lane == 0) mbar_arrive_count(&bars->p_ready[t][c], 2);
        }
      } else if (fixed_ref) {
        // ---- fixed reference.  The scores all lie inside [-score_bound, score_bound]; the constant
        // 2^-score_bound that would bring the exponents to [-2 score_bound, 0] cancels between numerator
        // and row sum, so it is not applied: reference 0, and the scores go into the exponential as
        // they come out of the tensor core.
        m_ref = 0.0f;
        sweep([](const uint32_t (&s)[32], uint32_t (&packed)[16], auto mask) {
          exp2_chunk<decltype(mask)::value ? 0 : kFaPolyPairs>(s, packed);  // (the polynomial cannot take -inf)
        });
      } else {
        // ---- a reference that is not zero.  The first step's scores are looked at once (they stay where
        // they are for the sweep): their maximum is a lower bound of the row maximum, score_bound an upper one.
        bool shifted = false;
        ok = scores_of(0, 0);
        float mx_own = INFINITY;  // of a warp that gives up: sends the partner to the form that keeps meeting it
        if (ok) {
          tc_fence_after();
          uint32_t s[32];
          tmem_ld32(s_addr + c * 32, s);
          tmem_ld_wait();
          masked(s, n_keys - c * 32);
          mx_own = max32(s);
        }
        pairs->first_max[t][c][row_in_tile] = mx_own;
        pair_barrier(barrier_id);
        int met = 0;  // pair barriers of the online form that this warp has been at, where it gives up
        const volatile uint32_t* partner_left = &pairs->left[t][c ^ 1][quarter];
        if (__any_sync(0xffffffffu, *partner_left != 0u ? 1 : 0)) break;
        const float mx_first = fmaxf(mx_own, pairs->first_max[t][c ^ 1][row_in_tile]);
        const FaJob job = job_at(id);
        const float v_max = kv_max[(job.seq * 2 + 1) * (dim / 64) + job.head];
        const float m = ceilf(fmaxf(score_bound - fa_shift_up(key_bits, v_max), mx_first));
        shifted = __all_sync(0xffffffffu, m - mx_first <= fa_shift_down(key_bits) && fabsf(m) <= 1048576.0f ? 1 : 0) != 0;
        if (shifted) m_ref = m;
        if (ok && shifted) {
          // ---- shifted reference, kept for the whole launch: a whole number m (see fa_shift_up) under which
          // nothing overflows and the row's largest probability is not small, so no running maximum is
          // needed.
          const float m = m_ref;
          sweep([m](const uint32_t (&s)[32], uint32_t (&packed)[16], auto mask) {
            exp2_chunk_shifted<decltype(mask)::value ? 0 : kFaShiftPolyPairs>(s, m, packed);
          });
        } else if (ok) {
          // ---- online form.  Both threads of a row share every step, half of its scores each, and tell each other their
          // maxima.
          auto step = [&](int j, int h, bool may_mask) -> bool {
            if (!scores_of(h, j)) {
              met = 2 * j + h;
              return false;
            }
            tc_fence_after();
            const uint32_t addr = s_addr + h * 64 + c * 32;
            uint32_t s[32], packed[16];
            auto load = [&] {
              tmem_ld32(addr, s);
              tmem_ld_wait();
              if (may_mask) masked(s, n_keys - (2 * j + h) * 64 - c * 32);
            };
            load();
            const float mx_own = max32(s);
            pairs->row_max[h][t][c][row_in_tile] = mx_own;
            pair_barrier(barrier_id);
            const float mx = fmaxf(mx_own, pairs->row_max[h][t][c ^ 1][row_in_tile]);
            if ((j | h) == 0) {
              m_ref = ceilf(mx) + kFaAhead;  // whole numbers, like the other forms'
            } else {
              const bool grow = mx > m_ref + kFaRescaleThreshold;
              if (__any_sync(0xffffffffu, grow ? 1 : 0)) {
                // O_t may still be the target of the previous step's P V.  The issuer follows that P V
                // with the Q K^T that refills the other half's scores, so their arrival tells that it
                // has retired; where nothing follows (the job's last step), pv_done does.
                const bool waited = 2 * j + h + 1 < n_steps ? scores_of(h ^ 1, j + h)
                                                            : mbar_wait_warp(&bars->pv_done[t], (turn >> 2) & 1u, ctl);
                if (!waited) {
                  met = 2 * j + h + 1;
                  return false;
                }
                tc_fence_after();
                const float m_new = grow ? ceilf(mx) + kFaAhead : m_ref;
                const float alpha = exp2_whole(m_ref - m_new);
                m_ref = m_new;
                uint32_t acc[32], sum;  // this thread's 32 of the row's 64 output channels; one of the two has the row sum too
                tmem_ld32(o_addr, acc);
                tmem_ld1(o_row + 64, sum);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 32; ++i) acc[i] = __float_as_uint(__uint_as_float(acc[i]) * alpha);
                tmem_st32(o_addr, acc);
                if (c == 1) tmem_st1(o_row + 64, __float_as_uint(__uint_as_float(sum) * alpha));
                load();  // again: held beside the output they would spill
              }
            }
            exp2_chunk_shifted<0>(s, m_ref, packed);
            tmem_st16(addr, packed);  // over the start of the columns just read
            give_p(h, 1);
            return true;
          };
          for (int j = 0; j < last && ok; ++j) ok = step(j, 0, false) && step(j, 1, false);
          if (ok) ok = step(last, 0, true) && (2 * last + 1 == n_steps || step(last, 1, true));
        }
        if (!ok && !shifted) meet_partner(barrier_id, met, n_steps);
      }
      if (!ok) break;
      // The next job's queries take the old ones' place, and the next scores are under way, while the tensor cores finish this
      // one's last P V and its rows are written.
      if constexpr (kJobs) asm volatile("" : "+r"(id));  // the job is worked out again: nothing of it is held over the sweep
      const int after = job_after(turn >> 4, false, ok);
      turn += 16u;
      const int next_id = next_job(after);
      if (!ok) break;
      if (next_id < id_end) {
        const int last_step = steps_of(tiles_at(id)) - 1;  // its scores came behind all others
        if (!scores_of(last_step & 1, last_step >> 1)) break;
        tc_fence_after();
        score_bound = take_q(job_at(next_id), ((turn >> 2) & 1u) ^ 1u);
        if (score_bound < 0.0f) break;
      }
      if (!mbar_wait_warp(&bars->o_done[t], (turn >> 2) & 1u, ctl)) break;
      tc_fence_after();
      uint32_t acc[32], sum;
      tmem_ld32(o_addr, acc);
      tmem_ld1(o_row + 64, sum);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (kJobs && lane == 0) mbar_arrive(&bars->o_free[t]);
      const FaJob job = job_at(id);
      // A part of a row leaves with its sum between 1 and 2 and the reference that goes with it: references chosen for a
      // launch lie up to a hundred binades over or under what a part holds, which would be lost beside another part.
      if (!(kFirst && kLast) || job.slot >= 0) {
        const uint32_t e = min(max(sum >> 23 & 255u, 1u), 253u);
        const float scale = __uint_as_float((254u - e) << 23);
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i] = __float_as_uint(__uint_as_float(acc[i]) * scale);
        sum = __float_as_uint(__uint_as_float(sum) * scale);
        m_ref += (float)((int)e - 127);
      }
      const int row = job.seq * seq_len + row_of(job);  // global row of qkv / o
      uint8_t* my_rows = smem_o + warp * 2048;  // 32 rows of 64 bytes, 16-byte unit u of row r at u ^ (r / 2 mod 4)
      if (row_of(job) < seq_len) {
        if (job.slot >= 0) {
          fa_store_part(jobs, job.slot, t * 128 + row_in_tile, c, acc, 1.0f, m_ref, __uint_as_float(sum));
        } else {
          float row_sum = __uint_as_float(sum);
          // each of the row's two threads keeps its own copy of {reference, row sum} in the state
          float* ml_mine = ml_state + ((size_t)row * (dim / 64) + job.head) * 4 + 2 * c;
          if (!first_chunk) {
            // add what the earlier chunks left for this row, in fp32 with round-to-nearest: partial
            // output, row sum and their reference; the weights are powers of two
            const float m_old = ml_mine[0], l_old = ml_mine[1];
            float a_old = 1.0f, a_new = 1.0f;
            if (m_old != m_ref) {
              const float m_tot = fmaxf(m_old, m_ref);
              a_old = exp2_whole(m_old - m_tot);
              a_new = exp2_whole(m_ref - m_tot);
              m_ref = m_tot;
            }
            const uint4* src = reinterpret_cast<const uint4*>(o_state + (size_t)row * dim + job.head * 64 + c * 32);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const uint4 v = src[i];
              const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
              for (int e = 0; e < 4; ++e)
                acc[4 * i + e] = __float_as_uint(fmaf(__uint_as_float(acc[4 * i + e]), a_new, __uint_as_float(w[e]) * a_old));
            }
            row_sum = fmaf(row_sum, a_new, l_old * a_old);
          }
          if (last_chunk) {
            const float inv = 1.0f / row_sum;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint4 w;
              w.x = pack_bf16(__uint_as_float(acc[q * 8 + 0]) * inv, __uint_as_float(acc[q * 8 + 1]) * inv);
              w.y = pack_bf16(__uint_as_float(acc[q * 8 + 2]) * inv, __uint_as_float(acc[q * 8 + 3]) * inv);
              w.z = pack_bf16(__uint_as_float(acc[q * 8 + 4]) * inv, __uint_as_float(acc[q * 8 + 5]) * inv);
              w.w = pack_bf16(__uint_as_float(acc[q * 8 + 6]) * inv, __uint_as_float(acc[q * 8 + 7]) * inv);
              *reinterpret_cast<uint4*>(my_rows + lane * 64 + ((q ^ (lane >> 1 & 3)) << 4)) = w;
            }
          } else {
            // leave the sum over the chunks so far for the next launch
            uint4* dst = reinterpret_cast<uint4*>(o_state + (size_t)row * dim + job.head * 64 + c * 32);
#pragma unroll
            for (int i = 0; i < 8; ++i) dst[i] = make_uint4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
            ml_mine[0] = m_ref;
            ml_mine[1] = row_sum;
          }
        }
      }
      if (last_chunk && job.slot < 0) {
        // four lanes a row: a store of the warp's covers 8 lines, where a row of its own for every lane makes it 32
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = i * 8 + (lane >> 2), in_seq = job.q_block * (128 * kTiles) + t * 128 + (int)quarter * 32 + r;
          const uint4 v = *reinterpret_cast<const uint4*>(my_rows + r * 64 + (((lane & 3) ^ (r >> 1 & 3)) << 4));
          if (in_seq < seq_len)
            *reinterpret_cast<uint4*>(o + (size_t)(job.seq * seq_len + in_seq) * dim + job.head * 64 + c * 32 + (lane & 3) * 8) = v;
        }
        __syncwarp();
      }
      const uint32_t steps = (uint32_t)steps_of(tiles_at(id));
      turn ^= ((steps + 1) >> 1 & 1u) | (steps & 2u) | 4u;
      id = next_id;
    }
    if (__any_sync(0xffffffffu, *ctl.abort_flag != 0u ? 1 : 0)) {
      *const_cast<volatile uint32_t*>(&pairs->left[t][c][quarter]) = 1u;
      pair_barrier_leave(barrier_id);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kIssuerWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, Shape::kTmemCols);
  }
}

// ------------------------------------------------------------------------------------------------
// E4M3 variant (qkv_dtype = 1).  Same CTA shape, warp roles, barriers and tensor-memory map as the
// bf16 kernel above; what differs:
//   * Q, K and V arrive as E4M3 bytes with one scale per (tensor, head); both products run as
//     kind::f8f6f4 (K = 32 per instruction: two instructions per step and product instead of four);
//   * K tiles are 128 keys x 64 bytes (64-byte swizzle); V comes transposed, 64 channel rows x 128
//     key bytes per tile, K-major like K, followed in shared memory by 16 rows of which the first
//     holds 1.0 in every byte: as rows 64..79 of the B operand they make accumulator column 64 the sum
//     of the very E4M3 probabilities that multiply V;
//   * the probabilities are rounded to E4M3, whose values reach from 2^-9 to 448 only, so they must
//     sit at the top of that range: every row runs the online form with the reference kept 8 below
//     the running row maximum (the largest probability of a row is 2^8 when the reference is set
//     and may grow to 2^8.75 before the row is rescaled), which leaves 17 binades below the row
//     maximum before a probability is rounded to zero; the two warps of a pair take a half of
//     every key tile each and pass the reference on from step to step;
//   * scores are multiplied by scale_q scale_k (K arrives with the softmax scale folded in, which its
//     per-head scale absorbs), the output by scale_v, in fp32.
constexpr int kFa8Stages = 4;
constexpr uint32_t kFa8ColS = 0, kFa8ColO = 256;
constexpr int kFa8KTileBytes = 128 * 64;           // 128 keys x 64 channel bytes
constexpr int kFa8VTileBytes = 64 * 128;           // 64 channels x 128 key bytes
constexpr int kFa8VStageBytes = kFa8VTileBytes + 16 * 128;  // + the ones rows
constexpr uint32_t kFa8ColQ = 416;                 // Q_0, Q_1: 16 columns of 4 bytes each
constexpr float kFa8Headroom = 8.0f;               // the row maximum maps to 2^8 of E4M3's 448
// What the two warps of a pair hand each other: the reference of their 32 rows after every step, and the
// barriers that say so.
struct Fa8Barriers {
  uint64_t q_ready;
  uint64_t k_full[kFa8Stages], k_empty[kFa8Stages];
  uint64_t v_full[kFa8Stages], v_empty[kFa8Stages];
  uint64_t s_full[2][2], p_ready[2][2], pv_done[2], o_done[2];
  uint64_t teardown[2];
  uint32_t tmem_base;
  uint32_t abort_flag;
};
struct Fa8Refs {
  float m_ref[2][2][128];       // [column of steps][tile][row]
  uint64_t ready[2][2][4];      // [column of steps][tile][quarter]
};
constexpr int kFa8SmemBytes = kFa8Stages * (kFa8KTileBytes + kFa8VStageBytes) + (int)sizeof(Fa8Refs) + 512 + 1024;

// 32 scores -> 32 E4M3 probabilities 2^(s * scale - m), all from the special-function unit.  A polynomial good enough
// to stand beside it (poly_exp2_pair<true>) saves nothing here: core at 21,984 rows 2.13 ms as it is, 2.12
// with one pair of 16 on the FMA pipes, 2.17 with two, 2.18 with three.
__device__ __forceinline__ void exp2_chunk_e4m3(const uint32_t (&s)[32], float2 scale2, float2 neg_m2, uint32_t (&packed)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float2 p[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int pair = 2 * i + k;
      const float2 x = __ffma2_rn(make_float2(__uint_as_float(s[2 * pair]), __uint_as_float(s[2 * pair + 1])), scale2, neg_m2);
      p[k].x = fast_exp2(x.x);
      p[k].y = fast_exp2(x.y);
    }
    packed[i] = pack_e4m3x4(p[0].x, p[0].y, p[1].x, p[1].y);
  }
}

template <bool kFirst, bool kLast>
__global__ void __launch_bounds__(kFaThreads, 1)
flash_attention_fp8_kernel(const __grid_constant__ CUtensorMap tmap_k8, const __grid_constant__ CUtensorMap tmap_v8t,
                           const uint8_t* __restrict__ q8, const float* __restrict__ amax, __nv_bfloat16* __restrict__ o,
                           float* __restrict__ o_state, float* __restrict__ ml_state, int seq_len, int dim, int tile_begin,
                           int tile_end, FaJobs split, uint32_t* status, Stamp stamp) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* smem_k = smem;
  uint8_t* smem_v = smem_k + kFa8Stages * kFa8KTileBytes;
  Fa8Refs* refs = reinterpret_cast<Fa8Refs*>(smem_v + kFa8Stages * kFa8VStageBytes);
  Fa8Barriers* bars = reinterpret_cast<Fa8Barriers*>(refs + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const FaJob job = fa_job(split, blockIdx.x);
  const FaTiles kv = fa_tiles(split, blockIdx.x, tile_begin, tile_end);
  tile_begin = kv.begin;
  tile_end = kv.end;
  const int q0 = job.q_block * 256;
  const int head = job.head;
  const int n_kv = tile_end - tile_begin;
  constexpr bool first_chunk = kFirst;
  constexpr bool last_chunk = kLast;

  if (threadIdx.x == 0) {
    mbar_init(&bars->q_ready, kFaSoftmaxWarps);
    for (int s = 0; s < kFa8Stages; ++s) {
      mbar_init(&bars->k_full[s], 1);
      mbar_init(&bars->k_empty[s], 2);
      mbar_init(&bars->v_full[s], 1);
      mbar_init(&bars->v_empty[s], 2);
    }
    for (int t = 0; t < 2; ++t) {
      for (int h = 0; h < 2; ++h) {
        mbar_init(&bars->s_full[t][h], 1);
        mbar_init(&bars->p_ready[t][h], 8);
      }
      mbar_init(&bars->pv_done[t], 1);
      mbar_init(&bars->o_done[t], 1);
    }
    for (int i = 0; i < 16; ++i) mbar_init(&refs->ready[0][0][0] + i, 1);
    mbar_init(&bars->teardown[0], 1);
    mbar_init(&bars->teardown[1], 1);
    bars->abort_flag = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tmap_k8);
    tma_prefetch_desc(&tmap_v8t);
  }
  // the ones rows behind every V stage: 128 bytes of E4M3 1.0 (0x38), then 15 rows of zeros (a row
  // of equal bytes looks the same under the swizzle)
  for (int i = threadIdx.x; i < kFa8Stages * 16 * 128 / 16; i += kFaThreads) {
    const int stage = i / 128, piece = i % 128;  // 128 16-byte pieces per stage
    const uint32_t fill = piece < 8 ? 0x38383838u : 0u;
    reinterpret_cast<uint4*>(smem_v + stage * kFa8VStageBytes + kFa8VTileBytes)[piece] = make_uint4(fill, fill, fill, fill);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 16) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = bars->tmem_base;
  const WaitCtl ctl{&bars->abort_flag, status};
  const Span span(stamp);

  if (warp == 17) {
    // ------------------------------------------------------------------ TMA producer
    if (elect_one()) {
      uint32_t k_issued = 0, v_issued = 0;
      for (int j = 0; j < n_kv; ++j) {
        const int stage = j % kFa8Stages;
        const uint32_t phase = (uint32_t)(j / kFa8Stages) & 1u;
        if (!mbar_wait(&bars->k_empty[stage], phase ^ 1u, ctl)) break;
        mbar_expect_tx(&bars->k_full[stage], kFa8KTileBytes);
        tma_load_2d(smem_k + stage * kFa8KTileBytes, &tmap_k8, &bars->k_full[stage], head * 64, (tile_begin + j) * 128);
        ++k_issued;
        if (!mbar_wait(&bars->v_empty[stage], phase ^ 1u, ctl)) break;
        mbar_expect_tx(&bars->v_full[stage], kFa8VTileBytes);
        tma_load_2d(smem_v + stage * kFa8VStageBytes, &tmap_v8t, &bars->v_full[stage], (tile_begin + j) * 128, head * 64);
        ++v_issued;
      }
      drain_ring<kFa8Stages>(bars->k_full, k_issued, status);
      drain_ring<kFa8Stages>(bars->v_full, v_issued, status);
    }
  } else if (warp == 16 || warp == 18) {
    // ------------------------------------------------------------------ MMA issuer of tile t
    if (elect_one()) {
      const int t = warp == 16 ? 0 : 1;
      constexpr uint32_t idesc_qk = umma_idesc_e4m3(128, 64);
      constexpr uint32_t idesc_pv = umma_idesc_e4m3(128, kFaOCols);
      const uint32_t s_col = tmem_base + kFa8ColS + t * 128;
      const uint32_t o_col = tmem_base + kFa8ColO + t * kFaOCols;
      const uint32_t q_col = tmem_base + kFa8ColQ + t * 16;
      // S_h = Q x K[64h .. 64h+63]^T: 64 rows of 64 bytes = 4096 bytes per half, 32 channels per instruction
      auto issue_qk = [&](int h, int stage) {
        const uint64_t b_desc = smem_desc_sw64(smem_u32(smem_k + stage * kFa8KTileBytes + h * 4096), 16, 512);
#pragma unroll
        for (int k = 0; k < 2; ++k) umma_ts_f8(s_col + h * 64, q_col + k * 8, b_desc + 2 * k, idesc_qk, k != 0 ? 1u : 0u);
        umma_commit(&bars->s_full[t][h]);
      };
      bool ok = mbar_wait(&bars->q_ready, 0, ctl);
      if (ok) ok = mbar_wait(&bars->k_full[0], 0, ctl);
      if (ok) {
        tc_fence_after();
        issue_qk(0, 0);
        issue_qk(1, 0);
        umma_commit(&bars->k_empty[0]);
      }
      int stage = 0;
      uint32_t phase = 0;
      for (int j = 0; j < n_kv && ok; ++j) {
        int next_stage = stage + 1;
        uint32_t next_phase = phase;
        if (next_stage == kFa8Stages) { next_stage = 0; next_phase ^= 1u; }
        const bool last = j + 1 == n_kv;
        if (!mbar_wait(&bars->v_full[stage], phase, ctl)) { ok = false; break; }
        if (!last && !mbar_wait(&bars->k_full[next_stage], next_phase, ctl)) { ok = false; break; }
        for (int h = 0; h < 2; ++h) {
          if (!mbar_wait(&bars->p_ready[t][h], j & 1, ctl)) { ok = false; break; }
          tc_fence_after();
          // 64 keys of the transposed V tile: bytes [64h, 64h + 64) of every channel row, 32 keys per
          // instruction; 8 tensor-memory columns of P each (keys 0-31 in columns [0,8) of the half,
          // keys 32-63 in [32,40)); rows 64..79 of B are the ones rows behind the tile
          const uint64_t v_desc = smem_desc_sw128(smem_u32(smem_v + stage * kFa8VStageBytes + h * 64), 16, 1024);
#pragma unroll
          for (int k = 0; k < 2; ++k)
            umma_ts_f8(o_col, s_col + h * 64 + k * 32, v_desc + 2 * k, idesc_pv, (j | h | k) != 0 ? 1u : 0u);
          if (last) {
            umma_commit(&bars->pv_done[t]);
            if (h == 1) umma_commit(&bars->o_done[t]);
          } else {
            issue_qk(h, next_stage);
          }
        }
        if (!ok) break;
        umma_commit(&bars->v_empty[stage]);
        if (!last) umma_commit(&bars->k_empty[next_stage]);
        stage = next_stage;
        phase = next_phase;
      }
      if (!ok) {
        umma_commit(&bars->teardown[t]);
        const long long t0 = clock64();
        while (!mbar_try_wait(&bars->teardown[t], 0)) {
          if (clock64() - t0 > kTimeoutCycles) break;
        }
      }
    }
  } else if (warp < kFaSoftmaxWarps) {
    // ------------------------------------------------------------------ softmax warps
    const int t = warp >> 3;
    const int c = (warp >> 2) & 1;
    const uint32_t quarter = warp & 3u;
    const int row_in_tile = (int)quarter * 32 + lane;
    const uint32_t lane_base = (quarter * 32u) << 16;
    const int row_local = q0 + t * 128 + row_in_tile;
    const bool row_live = row_local < seq_len;
    const int row = row_local;
    const uint32_t s_addr = tmem_base + lane_base + kFa8ColS + t * 128;
    const uint32_t o_row = tmem_base + lane_base + kFa8ColO + t * kFaOCols, o_addr = o_row + c * 32;
    const uint32_t l_addr = tmem_base + lane_base + kFa8ColO + t * kFaOCols + 64;
    {
      // this thread's 32 channels (32 bytes) of its query row
      uint32_t qreg[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) qreg[i] = 0u;
      if (row_live) {
        const uint4* src = reinterpret_cast<const uint4*>(q8 + (size_t)row * dim + head * 64 + c * 32);
        const uint4 a = __ldg(src), b = __ldg(src + 1);
        qreg[0] = a.x; qreg[1] = a.y; qreg[2] = a.z; qreg[3] = a.w;
        qreg[4] = b.x; qreg[5] = b.y; qreg[6] = b.z; qreg[7] = b.w;
      }
      tmem_st8(tmem_base + lane_base + kFa8ColQ + t * 16 + c * 8, qreg);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->q_ready);
    }
    // dequantisation: score = (q8 . k8) scale_q scale_k / sqrt(64), output = (P v8) scale_v / sum P
    const float a_q = amax[head], a_k = amax[16 + head], a_v = amax[32 + head];
    const float scale_q = (a_q > 0.0f ? a_q : 1.0f) / 448.0f, scale_k = (a_k > 0.0f ? a_k : 1.0f) / 448.0f;
    const float scale_v = (a_v > 0.0f ? a_v : 1.0f) / 448.0f;
    const float scale_log2e = scale_q * scale_k;  // K was quantised with the softmax scale folded in
    const float2 scale2 = make_float2(scale_log2e, scale_log2e);
    float m_ref = -INFINITY;
    bool ok = true;
    // Warp c of a pair takes half c of every key tile whole (64 scores a thread) and they alternate: each
    // step starts from the reference the partner's step before it left, and leaves its own as soon as the
    // step's maximum is known - before its exponentials, so the partner does not wait for those.  Only
    // the last tile of a launch can reach past the sequence.
    auto step = [&](int j, bool may_mask) -> bool {
      if (!mbar_wait_warp(&bars->s_full[t][c], j & 1, ctl)) return false;
      tc_fence_after();
      const uint32_t base = s_addr + c * 64;
      const int valid = may_mask ? seq_len - ((tile_begin + j) * 2 + c) * 64 : 64;
      auto load = [&](int g, uint32_t (&s)[32]) {
        tmem_ld32(base + g * 32, s);
        tmem_ld_wait();
        if (may_mask && valid - g * 32 < 32) {
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (i >= valid - g * 32) s[i] = 0xff800000u;  // -inf
        }
      };
      // the first 32 scores are read once for the maximum and once more for the exponentials: 64 held
      // meanwhile would spill
      uint32_t s[32];
      load(0, s);
      float mx_scaled = max32(s);
      load(1, s);
      mx_scaled = fmaxf(mx_scaled, max32(s)) * scale_log2e;
      bool grow = true;
      if ((j | c) != 0) {
        if (!mbar_wait_warp(&refs->ready[c ^ 1][t][quarter], (uint32_t)(c == 1 ? j : j - 1) & 1u, ctl)) return false;
        m_ref = refs->m_ref[c ^ 1][t][row_in_tile];
        grow = mx_scaled > m_ref + kFa8Headroom + 0.75f;
      }
      const float m_old = m_ref;
      if (grow) m_ref = mx_scaled - kFa8Headroom;
      refs->m_ref[c][t][row_in_tile] = m_ref;
      __syncwarp();
      if (lane == 0) mbar_arrive(&refs->ready[c][t][quarter]);
      if ((j | c) != 0 && __any_sync(0xffffffffu, grow ? 1 : 0)) {
        // O_t may still be the target of the previous step's P V; what follows that tells when it has retired
        const int jp = c == 1 ? j : j - 1;
        const bool waited = jp + 1 < n_kv ? mbar_wait_warp(&bars->s_full[t][c ^ 1], (uint32_t)(jp + 1) & 1u, ctl)
                                          : mbar_wait_warp(&bars->pv_done[t], 0, ctl);
        if (!waited) return false;
        tc_fence_after();
        const float alpha = fast_exp2(m_old - m_ref);
#pragma unroll 1
        for (int g = 0; g < 5; ++g) {  // the row's 64 output channels, then its sum and 15 unused columns
          uint32_t acc[16];
          tmem_ld16(o_row + g * 16, acc);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[i] = __float_as_uint(__uint_as_float(acc[i]) * alpha);
          tmem_st16(o_row + g * 16, acc);
        }
      }
      const float2 neg_m2 = make_float2(-m_ref, -m_ref);
      uint32_t packed[8];  // 32 probabilities as E4M3 bytes, over the start of their scores' columns
      exp2_chunk_e4m3(s, scale2, neg_m2, packed);
      tmem_st8(base + 32, packed);
      load(0, s);
      exp2_chunk_e4m3(s, scale2, neg_m2, packed);
      tmem_st8(base, packed);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_count(&bars->p_ready[t][c], 2);
      return true;
    };
    for (int j = 0; j + 1 < n_kv && ok; ++j) ok = step(j, false);
    if (ok && n_kv > 0) ok = step(n_kv - 1, true);
    if (ok && c == 0 && n_kv > 0) {  // the last step was the partner's
      ok = mbar_wait_warp(&refs->ready[1][t][quarter], (uint32_t)(n_kv - 1) & 1u, ctl);
      if (ok) m_ref = refs->m_ref[1][t][row_in_tile];
    }
    if (ok && mbar_wait_warp(&bars->o_done[t], 0, ctl)) {
      tc_fence_after();
      uint32_t acc[32], sum[16];
      tmem_ld32(o_addr, acc);
      tmem_ld16(l_addr, sum);
      tmem_ld_wait();
      if (job.slot >= 0) {
        if (row_live) fa_store_part(split, job.slot, t * 128 + row_in_tile, c, acc, scale_v, m_ref, __uint_as_float(sum[0]));
      } else if (row_live) {
        float row_sum = __uint_as_float(sum[0]);
        float* ml_mine = ml_state + ((size_t)row * (dim / 64) + head) * 4 + 2 * c;
        if (!first_chunk) {
          const float m_old = ml_mine[0], l_old = ml_mine[1];
          float a_old = 1.0f, a_new = 1.0f;
          if (m_old != m_ref) {
            const float m_tot = fmaxf(m_old, m_ref);
            a_old = fast_exp2(m_old - m_tot);
            a_new = fast_exp2(m_ref - m_tot);
            m_ref = m_tot;
          }
          const uint4* src = reinterpret_cast<const uint4*>(o_state + (size_t)row * dim + head * 64 + c * 32);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint4 v = src[i];
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
              acc[4 * i + e] = __float_as_uint(fmaf(__uint_as_float(acc[4 * i + e]), a_new, __uint_as_float(w[e]) * a_old));
          }
          row_sum = fmaf(row_sum, a_new, l_old * a_old);
        }
        if (last_chunk) {
          const float inv = scale_v / row_sum;
          uint4* dst = reinterpret_cast<uint4*>(o + (size_t)row * dim + head * 64 + c * 32);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint4 w;
            w.x = pack_bf16(__uint_as_float(acc[q * 8 + 0]) * inv, __uint_as_float(acc[q * 8 + 1]) * inv);
            w.y = pack_bf16(__uint_as_float(acc[q * 8 + 2]) * inv, __uint_as_float(acc[q * 8 + 3]) * inv);
            w.z = pack_bf16(__uint_as_float(acc[q * 8 + 4]) * inv, __uint_as_float(acc[q * 8 + 5]) * inv);
            w.w = pack_bf16(__uint_as_float(acc[q * 8 + 6]) * inv, __uint_as_float(acc[q * 8 + 7]) * inv);
            dst[q] = w;
          }
        } else {
          uint4* dst = reinterpret_cast<uint4*>(o_state + (size_t)row * dim + head * 64 + c * 32);
#pragma unroll
          for (int i = 0; i < 8; ++i) dst[i] = make_uint4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
          ml_mine[0] = m_ref;
          ml_mine[1] = row_sum;
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 16) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// Rows of the split jobs: the parts brought to a common reference and added in the order of their keys.
constexpr int kCombineRows = 32;  // a block's rows; a thread has 8 channels of one
__global__ void __launch_bounds__(kCombineRows * 8)
combine_parts_kernel(FaJobs split, __nv_bfloat16* __restrict__ o, int seq_len, int dim, Stamp stamp) {
  const Span span(stamp);
  const int job = split.full + blockIdx.x, q_block = split.q_first + job % split.q_blocks, head = job / split.q_blocks;
  __shared__ uint4 tile[kCombineRows][9];  // (a column beside the eight, against bank conflicts)
  const int r = blockIdx.y * kCombineRows + (threadIdx.x & 31), ch = (threadIdx.x >> 5) * 8;  // a lane a row, as the parts lie
  const size_t slot0 = (size_t)blockIdx.x * split.parts;
  float m = -INFINITY;
#pragma unroll 4
  for (int p = 0; p < split.parts; ++p) m = fmaxf(m, split.ml[((slot0 + p) * 256 + r) * 2]);
  float acc[8], sum = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.0f;
#pragma unroll 4
  for (int p = 0; p < split.parts; ++p) {
    const float2 ml = *reinterpret_cast<const float2*>(split.ml + ((slot0 + p) * 256 + r) * 2);
    // (the E4M3 form's references are no whole numbers)
    const float d = ml.x - m, w = ml.x == m ? 1.0f : d == rintf(d) ? exp2_whole(d) : fast_exp2(d);
    sum = fmaf(ml.y, w, sum);
    const float4* src = reinterpret_cast<const float4*>(split.o) + ((slot0 + p) * 16 + ch / 4) * 256 + r;
    const float4 a = src[0], b = src[256];
    acc[0] = fmaf(a.x, w, acc[0]);
    acc[1] = fmaf(a.y, w, acc[1]);
    acc[2] = fmaf(a.z, w, acc[2]);
    acc[3] = fmaf(a.w, w, acc[3]);
    acc[4] = fmaf(b.x, w, acc[4]);
    acc[5] = fmaf(b.y, w, acc[5]);
    acc[6] = fmaf(b.z, w, acc[6]);
    acc[7] = fmaf(b.w, w, acc[7]);
  }
  const float inv = 1.0f / sum;
  tile[threadIdx.x & 31][threadIdx.x >> 5] =
      make_uint4(pack_bf16(acc[0] * inv, acc[1] * inv), pack_bf16(acc[2] * inv, acc[3] * inv), pack_bf16(acc[4] * inv, acc[5] * inv),
                 pack_bf16(acc[6] * inv, acc[7] * inv));
  __syncthreads();
  const int row = q_block * 256 + blockIdx.y * kCombineRows + (threadIdx.x >> 3);
  if (row < seq_len) *reinterpret_cast<uint4*>(o + (size_t)row * dim + head * 64 + (threadIdx.x & 7) * 8) = tile[threadIdx.x >> 3][threadIdx.x & 7];
}

// How the jobs that do not fill a wave of one CTA an SM are split: into so many parts that their waves end
// soonest.  A key tile of two query tiles takes about 1.05 us, a CTA 8 us besides, adding the parts up 8.
// (21,984 rows: 1376 jobs = 9 waves and 44 jobs, three parts each, 1.776 -> 1.718 ms; in the E4M3 form, when it
// took part of its exponentials from a polynomial, 2.14 -> 2.07; 31,751 rows, shifted, 4.36 -> 4.17 with its
// exponentials of that time.)  Sequences of several key chunks have hundreds of waves and are left alone.
static FaJobs split_plan(long long seq_len, long long rows, int n_seq, int heads, int num_sms, int block_rows) {
  const long long n_tiles = (seq_len + kFaTileKeys - 1) / kFaTileKeys, q_blocks = (rows + block_rows - 1) / block_rows;
  const long long count = q_blocks * heads * n_seq;
  FaJobs jobs{0, (int)q_blocks, heads, (int)count, (int)count, 1, nullptr, nullptr, nullptr};
  if (n_seq != 1 || seq_len <= kFaOneTileRows || n_tiles > kFaChunkTiles) return jobs;
  const long long rest = count % num_sms;
  if (rest == 0) return jobs;
  float best_us = 8.0f + 1.05f * (float)n_tiles;
  for (int parts = 2; parts <= 16 && n_tiles / parts >= 4; ++parts) {
    const float us = 8.0f + (float)((rest * parts + num_sms - 1) / num_sms) * (8.0f + 1.05f * (float)n_tiles / (float)parts);
    if (us < best_us) {
      best_us = us;
      jobs.parts = parts;
    }
  }
  if (jobs.parts > 1) {
    jobs.full = (int)(count - rest);
    jobs.count = jobs.full + (int)rest * jobs.parts;
  }
  return jobs;
}
static long long split_slots(const FaJobs& jobs) { return jobs.count - jobs.full; }
// The jobs of a launch over query rows [row0, row1), their parts in the context's state buffers; a context without
// room for them (none, another sequence length, more parts than the whole sequence has) splits nothing.
static FaJobs jobs_for(const litevggt_ctx* ctx, long long seq_len, long long row0, long long row1, int n_seq, int block_rows) {
  const int heads = ctx->sz.heads, sms = ctx->num_sms;
  FaJobs jobs = split_plan(seq_len, row1 - row0, n_seq, heads, sms, block_rows);
  if (ctx->ws.attn_o_state == nullptr || seq_len != ctx->sz.n_merged ||
      split_slots(jobs) > split_slots(split_plan(seq_len, seq_len, n_seq, heads, sms, block_rows))) {
    jobs.count = jobs.full = jobs.q_blocks * heads * n_seq;
    jobs.parts = 1;
  }
  jobs.q_first = (int)(row0 / block_rows);
  jobs.o = ctx->ws.attn_o_state;
  jobs.ml = ctx->ws.attn_ml_state;
  return jobs;
}
static cudaError_t launch_combine(const litevggt_ctx* ctx, const FaJobs& split, __nv_bfloat16* o, long long seq_len, cudaStream_t s,
                                  int* launches) {
  ++*launches;
  // (its blocks wait until the attention's CTAs leave: 608 threads of 96 registers, in either form of operands, leave no room for 256
  // of 40.  Blocks that fitted beside them, as they did beside 80, would all sit on the first SMs, 7.9 us where they take 5.1)
  return launch(combine_parts_kernel, dim3((unsigned)(split_slots(split) / split.parts), 256 / kCombineRows),
                kCombineRows * 8, 0, s, split, o, (int)seq_len, ctx->sz.dim, next_stamp(ctx));
}

cudaError_t launch_flash_attention_fp8(litevggt_ctx* ctx, long long m, __nv_bfloat16* o, cudaStream_t s, int* launches) {
  if (m == 0) return cudaSuccess;
  const int dim = ctx->sz.dim;
  Workspace& ws = ctx->ws;
  if (dim != 1024 || ws.q8 == nullptr) return cudaErrorInvalidValue;
  const long long m_pad = round_up(m, 128);
  CUtensorMap tmap_k, tmap_v;
  if (!make_tmap_u8_2d(ctx->encode_tiled, &tmap_k, ws.k8, (uint64_t)dim, (uint64_t)m, (uint64_t)dim, 64, 128) ||
      !make_tmap_u8_2d(ctx->encode_tiled, &tmap_v, ws.v8t, (uint64_t)m_pad, (uint64_t)dim, (uint64_t)m_pad, 128, 64))
    return cudaErrorInvalidValue;
  using Kernel = void (*)(const CUtensorMap, const CUtensorMap, const uint8_t*, const float*, __nv_bfloat16*, float*,
                          float*, int, int, int, int, FaJobs, uint32_t*, Stamp);
  const Kernel kernels[2][2] = {{flash_attention_fp8_kernel<false, false>, flash_attention_fp8_kernel<false, true>},
                                {flash_attention_fp8_kernel<true, false>, flash_attention_fp8_kernel<true, true>}};
  static std::atomic<unsigned long long> smem_set[2][2];
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b) {
      cudaError_t e = set_max_dynamic_smem_once(reinterpret_cast<const void*>(kernels[a][b]), kFa8SmemBytes, smem_set[a][b]);
      if (e != cudaSuccess) return e;
    }
  const FaJobs split = jobs_for(ctx, m, 0, m, 1, 256);
  const dim3 grid((unsigned)split.count);
  const int n_tiles = (int)((m + kFaTileKeys - 1) / kFaTileKeys);
  const int n_chunks = (n_tiles + kFaChunkTiles - 1) / kFaChunkTiles;
  const int per_chunk = (n_tiles + n_chunks - 1) / n_chunks;
  if (n_chunks > 1 && (ws.attn_o_state == nullptr || ws.attn_ml_state == nullptr)) return cudaErrorInvalidValue;
  for (int begin = 0; begin < n_tiles; begin += per_chunk) {
    const int end = begin + per_chunk < n_tiles ? begin + per_chunk : n_tiles;
    cudaError_t e = launch(kernels[begin == 0][end == n_tiles], grid, kFaThreads, kFa8SmemBytes, s, tmap_k, tmap_v, ws.q8,
                           ws.qkv_amax, o, ws.attn_o_state, ws.attn_ml_state, (int)m, dim, begin, end, split,
                           ws.status, next_stamp(ctx));
    if (e != cudaSuccess) return e;
    ++*launches;
  }
  return split.parts > 1 ? launch_combine(ctx, split, o, m, s, launches) : cudaSuccess;
}

// `first_counter`: of the job counters that the projection has zeroed, the first that is free
static cudaError_t launch_rows(litevggt_ctx* ctx, const __nv_bfloat16* qkv, long long seq_len, long long row0, long long row1, int n_seq,
                               int first_counter, __nv_bfloat16* o, cudaStream_t s, int* launches) {
  if (seq_len == 0 || row0 == row1 || n_seq == 0) return cudaSuccess;
  const int dim = ctx->sz.dim;
  if (dim != 1024 || ctx->ws.attn_kmax == nullptr) return cudaErrorInvalidValue;
  const long long rows = seq_len * n_seq;
  // (a head's row is 128 bytes; the next head's, brought along, is gone again before its turn: 130,125 rows read 2.39 GB a layer,
  // 2.13 where only the queries come alone, 1.91 where keys and values do too, in the same time)
  CUtensorMap tmap;
  if (!make_tmap_bf16_2d(ctx->encode_tiled, &tmap, qkv, (uint64_t)3 * dim, (uint64_t)rows, (uint64_t)3 * dim, 64, kFaTileKeys, true))
    return cudaErrorInvalidValue;
  using Kernel = void (*)(const CUtensorMap, __nv_bfloat16*, float*, float*, const float*, float, int,
                          int, int, int, FaJobs, uint32_t*, Stamp);
  // [query tiles of a CTA - 1][first chunk][last chunk]
  const Kernel kernels[2][2][2] = {
      {{flash_attention_kernel<1, false, false>, flash_attention_kernel<1, false, true>},
       {flash_attention_kernel<1, true, false>, flash_attention_kernel<1, true, true>}},
      {{flash_attention_kernel<2, false, false>, flash_attention_kernel<2, false, true>},
       {flash_attention_kernel<2, true, false>, flash_attention_kernel<2, true, true>}}};
  const int smem_bytes[2] = {FaShape<1>::kSmemBytes, FaShape<2>::kSmemBytes};
  static std::atomic<unsigned long long> smem_set[2][2][2];
  const int tiles = seq_len <= kFaOneTileRows ? 1 : 2;
  // balanced chunks of at most kFaChunkTiles key tiles; more than one needs the state buffers (which
  // are sized for the single long sequence of the global layer)
  const int n_tiles = (int)((seq_len + kFaTileKeys - 1) / kFaTileKeys);
  const int n_chunks = (n_tiles + kFaChunkTiles - 1) / kFaChunkTiles;
  const int per_chunk = (n_tiles + n_chunks - 1) / n_chunks;
  if (n_chunks > 1 && (n_seq != 1 || ctx->ws.attn_o_state == nullptr || ctx->ws.attn_ml_state == nullptr))
    return cudaErrorInvalidValue;
  FaJobs split = jobs_for(ctx, seq_len, row0, row1, n_seq, 128 * tiles);
  if (tiles == 2 && (ctx->ws.attn_taken == nullptr || first_counter + n_chunks > kAttnCounters)) return cudaErrorInvalidValue;
  split.taken = ctx->ws.attn_taken + first_counter;
  const dim3 grid = tiles == 2 ? dim3((unsigned)(split.count < ctx->num_sms ? split.count : ctx->num_sms))
                               : dim3((unsigned)split.q_blocks, (unsigned)ctx->sz.heads, (unsigned)n_seq);
  const int threads = tiles == 2 ? FaShape<2>::kThreads : FaShape<1>::kThreads;
  // CTAs of one tile that set themselves up under the projection's last blocks would sit two to an SM on the first SMs
  // to become free (four small frames: 9.9 us against 6.2).  Where there is an SM for each, they ask for one
  // of their own; where there is not, they wait.
  const bool early = tiles == 2 || (long long)grid.x * grid.y * grid.z <= ctx->num_sms;
  const int smem = tiles == 1 && early ? kFaAloneBytes : smem_bytes[tiles - 1];
  for (int begin = 0; begin < n_tiles; begin += per_chunk) {
    const int end = begin + per_chunk < n_tiles ? begin + per_chunk : n_tiles;
    const int a = tiles - 1, b = begin == 0, c = end == n_tiles;
    cudaError_t e = set_max_dynamic_smem_once(reinterpret_cast<const void*>(kernels[a][b][c]), a == 0 ? kFaAloneBytes : smem_bytes[a],
                                              smem_set[a][b][c]);
    if (e != cudaSuccess) return e;
    e = launch_clusters(1, early, kernels[a][b][c], grid, threads, smem, s, tmap, o, ctx->ws.attn_o_state, ctx->ws.attn_ml_state,
               ctx->ws.attn_kmax, key_bits(seq_len), (int)seq_len, dim, begin, end, split, ctx->ws.status, next_stamp(ctx));
    if (e != cudaSuccess) return e;
    ++*launches;
    ++split.taken;
  }
  return split.parts > 1 ? launch_combine(ctx, split, o, seq_len, s, launches) : cudaSuccess;
}

cudaError_t launch_flash_attention(litevggt_ctx* ctx, const __nv_bfloat16* qkv, long long seq_len, int n_seq,
                                   __nv_bfloat16* o, cudaStream_t s, int* launches) {
  return launch_rows(ctx, qkv, seq_len, 0, seq_len, n_seq, 0, o, s, launches);
}

cudaError_t launch_flash_attention_rows(litevggt_ctx* ctx, const __nv_bfloat16* qkv, long long m, long long row0, long long row1,
                                        __nv_bfloat16* o, cudaStream_t s, int* launches) {
  const int sms = ctx->num_sms, heads = ctx->sz.heads;
  if (row0 < 0 || row0 % 256 != 0 || row1 != attention_slab_end(m, row0, sms, heads)) return cudaErrorInvalidValue;
  return launch_rows(ctx, qkv, m, row0, row1, 1, attention_slab_index(row0, sms, heads), o, s, launches);
}

// What passes between launches: for several key chunks rows of fp32 partial output and of {reference, row
// sum} x 2 per head (one copy per thread of a row), for a split last wave the parts' rows; zero where
// neither happens.
size_t attention_state_bytes(long long m, int dim, int heads, int num_sms, size_t* ml_offset) {
  const long long n_tiles = (m + kFaTileKeys - 1) / kFaTileKeys;
  size_t o_bytes = 0, ml_bytes = 0;
  if (n_tiles > kFaChunkTiles) {
    o_bytes = (size_t)round_up(m * dim * 4, 256);
    ml_bytes = (size_t)round_up(m * heads * 16, 256);
  } else {
    const long long slots = split_slots(split_plan(m, m, 1, heads, num_sms, 256));
    o_bytes = (size_t)slots * 256 * 64 * 4;
    ml_bytes = (size_t)slots * 256 * 2 * 4;
  }
  *ml_offset = o_bytes;
  return o_bytes + ml_bytes;
}

}  // namespace lv

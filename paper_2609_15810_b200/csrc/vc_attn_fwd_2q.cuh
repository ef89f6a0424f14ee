// The default 8-bit attention kernel for sm_100a (Eq. 1, Eq. 6, Eq. 7): warp-specialized, two 128-row
// query tiles per CTA.  One translation unit per head dimension includes this file.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "vc_attn_shared.cuh"
#include "vc_internal.h"
#include "vc_launch.h"
#include "vc_sm100.cuh"

namespace vc {
namespace {

using namespace sm100;
using namespace attn;

// ---------------------------------------------------------------------------------------
// Two-query-tile kernel (default).  A CTA owns TWO 128-row query tiles of one (batch, head)
// and streams each K^_j / R^_j tile through both, so every key/value byte fetched from L2
// feeds 256 query rows.  Two decisions keep the softmax stage - the bottleneck on this GPU -
// as short as the method allows:
//   * The probability codes have tensor-memory columns of their own (32 per tile) and are the A operand
//     of the value product there, so a score tile is free as soon as its 128 x 128 values are in
//     registers.  At d = 128 one score buffer serves both query tiles in turn (all that tensor memory
//     has room for); at d = 64 each tile has its own, but for kSfu.  (An MMA with both operands in shared memory reads
//     128 bytes a clock, all a shared-memory port gives.  With the codes there as well, 32 KB written and
//     32 KB read per pair of tiles, every copy and store slowed the products down; the port was busy for 78 percent of
//     the launch at d = 128 and 69 at d = 64, now 53 and 39.  B2 H16 N16384 d64 1956 -> 1870 us, B1 H12 N32760 d128
//     without value smoothing 3677 -> 3604, B1 H40 12.49 -> 12.33 ms under the power cap, B1 H6 N1955 d64 29.8 -> 28.9 us.)
//   * The row sums of the decoded codes (Eq. 6: r_ij, and the normalizer l) come from the
//     tensor core: the value operand carries 16 extra rows of ones, so columns d..d+15 of the
//     accumulator hold l, rescaled by alpha together with the rest.  The softmax threads do
//     nothing but the row maximum and five instructions per four codes.
//
// What bounds it: per key tile and pair of query tiles the kernel takes about 2030 cycles at d = 128
// (1680 at d = 64).  The tensor pipe needs 1216 of them (704 at d = 64); two softmax warps per
// scheduler need about 1000 when nothing else runs on it and the correction warps and the hand-offs
// of the shared score buffer (1500 cycles per pair when they are all that is timed) take the rest.
// Above a few milliseconds at a stretch the power cap of the board bounds it as well.
// B1 H40 N32760 d128 13.3 -> 12.5 ms, B1 H12 without value smoothing 3.9 -> 3.1 (3.5 under the power cap), B2 H16 N16384 d64 2.13 -> 1.73 by: waits that
// test before they suspend, no operand expansion in front, query tiles of the last wave one by one.
//
//   warp 0        producer: Q0, Q1 once; then per key tile K^_j, R^_j (TMA) and the tile's block
//                 mean (written as a [d x 8] TF32 operand, see MeanRows) through a 4-stage ring
//   warp 1        score issuer (one elected lane), per key tile j and query tile t:
//                   S    = Q^_t K^_j^T         4 x kind::f8f6f4, once the previous scores are read
//   warp 3        accumulator issuer, per key tile j and query tile t:
//                   A_t += P^_t(j) [R^_j | 1]  4 x kind::f8f6f4, N = d + 16, codes from tensor memory
//                   A_t += rho_{j-1} mu~_{j-1} 1 x kind::tf32: the rank-one mean term of Eq. 6, one
//                                              tile late, because r_{j-1} is read back from A_t first
//   warps 4-7     softmax warpgroup of tile 0, one thread per query row (128 scores in
//   warps 8-11    registers); likewise tile 1: running max, alpha, ExpCast-FP8 codes (Eq. 7: no
//                 exponential, no conversion), code tile to tensor memory (4 keys a column)
//   warps 12-15   correction warpgroup of tile 0 (16-19: tile 1), one thread per row: reads l
//                 back, r_{j-1} = l_{j-1} - alpha_{j-1} l_{j-2}, rescales A_t by alpha_j when a
//                 row maximum moved, hands (r_hi, r_lo) alpha_j to the mean MMA, writes the output
//
// Tensor memory: S (128 columns; 2 x 128 at d = 64) | A_0 (d + 16) | A_1 (d + 16) | P_0 (32) | P_1 (32) at column 416.
// P formats of the two-query-tile kernel
constexpr int kPfExpCast = 0, kPfExp = 1, kPfExpPoly = 2, kPfExpMix = 3;

// 2^x for x <= 8 without the special-function unit: x = n + f with n the nearest integer
// (1.5 * 2^23 trick) and |f| <= 1/2, 2^f by a degree-4 polynomial (relative error 3.7e-6, a
// 1/17000 of an E4M3 step), 2^n by an add into the exponent field.  Inputs below -24 give the
// value at -24, which rounds to code 0 like the exact result.
__device__ __forceinline__ float exp2_poly(float x) {
  x = fmaxf(x, -24.0f);
  const float t = x + 12582912.0f;
  const float f = x - (t - 12582912.0f);
  float p = fmaf(0.009676037356257439f, f, 0.05592203512787819f);
  p = fmaf(p, f, 0.2402210682630539f);
  p = fmaf(p, f, 0.6931210160255432f);
  p = fmaf(p, f, 1.0000001192092896f);
  return __uint_as_float(__float_as_uint(p) + (__float_as_uint(t) << 23));
}

// One query tile or pair of tiles (TWO) of head bh, first tile q0.
//
// TWO = false: one query tile, for the CTAs of a last wave that pairs would leave half empty (see
// split_tiles).  The second tile's score columns, code tile and barriers become second buffers of the
// first tile: scores of key tile j + 1 are computed while tile j's are read, codes of tile j are
// written while the product of tile j - 1 runs.
//
// SMOOTH = false: value smoothing is off, every block mean is zero and the mean term falls away (no mean
// operand, no TF32 product, no per-tile read of l).  A launch argument instead of a template
// parameter costs 1 % of the kernel with smoothing on.
template <int D, int PF, bool INT8, bool SMOOTH, bool TWO>
__device__ __forceinline__ void attn_2q_body(const CUtensorMap& tm_q, const CUtensorMap& tm_k, const CUtensorMap& tm_v,
                                             const AttnArgs& a, const int q0, const int bh) {
  constexpr int kTmemCols = 512;
  // exponentials of the special-function unit: a softmax warp then waits for that unit, which the warp of the other
  // query tile wants too, and the two run better out of step and with results that leave a few at a time
  constexpr bool kSfu = PF == kPfExp || PF == kPfExpMix;
  // d = 64 leaves room in tensor memory for a score buffer per query tile (B2 H16 N16384 d64: 1.89 -> 1.83 ms,
  // without smoothing 1.85 -> 1.76); at d = 128 both tiles share one, and with kSfu as well, because the shared
  // buffer is what keeps the two tiles out of step (B1 H16 N16384 d64, exponentials of E4M3 scores 1593 -> 1461 us, of
  // INT8 scores 1793 -> 1611, three of four by the unit 1523 -> 1494; all by polynomial 3004 -> 3033, so that one keeps two)
  constexpr bool kTwoS = D == 64 && !kSfu;
  constexpr uint32_t O_COL = kTwoS ? 256 : 128, O_STRIDE = D + 16, L_COL = D, S1_COL = kTwoS ? 128 : O_COL + O_STRIDE, P_COL = 416;   // A_t at O_COL + t * O_STRIDE; l in its column d
  // Register re-partition (setmaxnreg): the CTA owns 640 x 96 registers; a warpgroup that asks for
  // more than the others released would block forever, so the budget is checked at compile time.
  constexpr int kRegCtl = 48, kRegSoftmax = 160, kRegCorr = 56;
  static_assert(kRegCtl + 2 * kRegSoftmax + 2 * kRegCorr <= 5 * 96, "register budget exceeds the CTA's allocation");
  constexpr uint32_t kQBytes = 128 * D, kKBytes = 128 * D, kVBytes = D * 128, kOnesBytes = 16 * 128, kMuBytes = D * 32;
  constexpr uint32_t kStageBytes = kKBytes + kVBytes + kOnesBytes + ((kMuBytes + 1023) / 1024) * 1024;
  constexpr uint32_t kAmBytes = 128 * 32;
  extern __shared__ __align__(1024) unsigned char smem[];     // (the swizzled tiles want 1024-byte alignment)
  unsigned char* sQ = smem;                                    // [2][128 x D]
  unsigned char* sAm = smem + 2 * kQBytes;                       // [2][128 x 8 fp32] row-sum pairs
  unsigned char* sStage = sAm + 2 * kAmBytes;                  // [kStages2]{K, V | ones, Mu}
  FaSmem* sh = reinterpret_cast<FaSmem*>(sStage + kStages2 * kStageBytes);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nb = a.nb;
  // buffer (and barrier) of scores, codes and products of key tile j, and the parity of its phase
  auto buf = [](int t, int j) { return TWO ? t : j & 1; };
  auto par = [](int j) { return TWO ? j & 1 : (j >> 1) & 1; };
  // slot of the hand-off of alpha (see FaSmem) and the parity of its phase, and the same for codes and correction
  // (with block means two slots do there: B1 H8 N2048 d128, INT8 scores, 40.2 us instead of 40.6 with four)
  auto slot = [](int t, int j) { return TWO ? 2 * t + (j & 1) : j & 3; };
  auto slot_par = [](int j) { return TWO ? (j >> 1) & 1 : (j >> 2) & 1; };
  auto pc_slot = [](int t, int j) { return TWO || SMOOTH ? 2 * t + (j & 1) : j & 3; };
  auto pc_par = [](int j) { return TWO || SMOOTH ? (j >> 1) & 1 : (j >> 2) & 1; };

  const int early = min(kStages2, nb);      // key tiles whose copies are issued before anything else happens
  if (tid == 0) {
    init_barriers(sh, TWO);
    pdl_wait();                             // the bundle is complete from here on
    mbar_expect_tx(&sh->q_full, (TWO ? 2 : 1) * kQBytes);
    tma_load_3d(sQ, &tm_q, &sh->q_full, 0, q0 * 128, bh);
    if (TWO) tma_load_3d(sQ + kQBytes, &tm_q, &sh->q_full, 0, (q0 + 1) * 128, bh);   // past the end: zero fill
    for (int j = 0; j < early; ++j) {
      mbar_expect_tx_only(&sh->kv_full[j], kKBytes + kVBytes);
      tma_load_3d(sStage + j * kStageBytes, &tm_k, &sh->kv_full[j], 0, j * 128, bh);
      tma_load_3d(sStage + j * kStageBytes + kKBytes, &tm_v, &sh->kv_full[j], j * 128, 0, bh);
    }
  }
  for (int i = tid; i < 2 * (int)kAmBytes / 16; i += 640) reinterpret_cast<uint4*>(sAm)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < kStages2 * (int)kMuBytes / 16; i += 640)
    reinterpret_cast<uint4*>(sStage + (i / (kMuBytes / 16)) * kStageBytes + kKBytes + kVBytes + kOnesBytes)[i % (kMuBytes / 16)] = make_uint4(0, 0, 0, 0);
  // 16 rows of E4M3 1.0 behind every value tile (the rows are uniform, so the swizzle is moot)
  for (int i = tid; i < kStages2 * (int)kOnesBytes / 16; i += 640)
    reinterpret_cast<uint4*>(sStage + (i / (kOnesBytes / 16)) * kStageBytes + kKBytes + kVBytes)[i % (kOnesBytes / 16)] = make_uint4(0x38383838u, 0x38383838u, 0x38383838u, 0x38383838u);
  pdl_wait();
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy stores -> tensor-core reads
  if (warp == 2) { tmem_alloc<kTmemCols>(&sh->tmem_base); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_allow();                              // (behind the allocation: the next kernel may want tensor memory too)
  const uint32_t tmem = sh->tmem_base;
  const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);

  if (warp < 4) {
    reg_dec<kRegCtl>();
    if (warp == 0) {
      // ------------------------------------------------------------------ TMA producer
      // (the whole warp runs the loop: one elected lane issues the copies, all write the block means)
      int j = 0;
      for (; j < nb; ++j) {
        const int st = j % kStages2, it = j / kStages2;
        unsigned char* base = sStage + st * kStageBytes;
        MeanRows<D> mu;
        if (SMOOTH) mu.fetch(a.v_means + ((size_t)bh * nb + j) * D, lane);
        if (!warp_wait2(&sh->kv_empty[st], (it & 1) ^ 1, sh, a.wait, 11)) break;
        if (j >= early && elect_one()) {
          mbar_expect_tx_only(&sh->kv_full[st], kKBytes + kVBytes);
          tma_load_3d(base, &tm_k, &sh->kv_full[st], 0, j * 128, bh);
          tma_load_3d(base + kKBytes, &tm_v, &sh->kv_full[st], j * 128, 0, bh);
        }
        if (SMOOTH) {
          mu.store(base + kKBytes + kVBytes + kOnesBytes, lane);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the stores -> tensor-core reads
        }
        __syncwarp();
        if (elect_one()) mbar_arrive(&sh->kv_full[st]);
        __syncwarp();
      }
      drain_loads(sh, j);                                 // (returns at once on a normal run)
    } else if (warp == 1) {
      // ------------------------------------------------------------------ score issuer
      // Issues S_t = Q^_t K^_jT for both query tiles into the ONE score buffer, in the fixed order
      // S_0(0), S_1(0), S_0(1), S_1(1), ...: each may overwrite the buffer as soon as the previous
      // one has been read into registers.  (The whole warp runs the loop so that descriptors stay
      // in uniform registers; one elected lane issues.  A separate warp issues the A_t updates, so
      // that neither kind of MMA ever waits behind a barrier that only the other kind needs.)
      const uint32_t idesc_qk = INT8 ? idesc_s8(128, 128) : idesc_e4m3(128, 128);
      const uint64_t dq0 = smem_desc_kmajor(smem_u32(sQ), D), dq1 = smem_desc_kmajor(smem_u32(sQ + kQBytes), D);
      bool ok = warp_wait2(&sh->q_full, 0, sh, a.wait, 20);
      for (int j = 0; ok && j < nb; ++j) {
        const int st = j % kStages2, it = j / kStages2;
        if (!(ok = warp_wait2(&sh->kv_full[st], it & 1, sh, a.wait, 21))) break;
        const uint64_t dk = smem_desc_kmajor(smem_u32(sStage + st * kStageBytes), D);
#pragma unroll
        for (int t = 0; t < (TWO ? 2 : 1); ++t) {
          // S_0(j) waits for the read of S_1(j-1), S_1(j) for the read of S_0(j); with one tile S(j) for
          // the read of S(j-2), the buffer's previous tenant
          if (TWO && kTwoS) {
            if (j > 0 && !(ok = warp_wait2(&sh->s_free[t], (j - 1) & 1, sh, a.wait, 22))) break;
          } else if (TWO ? (t == 0 ? j > 0 : true) : j > 1) {
            if (!(ok = warp_wait2(&sh->s_free[TWO ? 1 - t : j & 1], TWO ? (t == 0 ? j - 1 : j) & 1 : par(j) ^ 1, sh, a.wait, 22))) break;
          }
          if (elect_one()) {
            tc_fence_after();
            const uint64_t dq = t == 0 ? dq0 : dq1;
            const uint32_t s_col = tmem + (TWO ? (kTwoS ? t * S1_COL : 0) : (j & 1) * S1_COL);
#pragma unroll
            for (int k = 0; k < D / 32; ++k) {
              if constexpr (INT8) mma_s8_ss(s_col, dq + 2 * k, dk + 2 * k, idesc_qk, k > 0);
              else mma_f8_ss(s_col, dq + 2 * k, dk + 2 * k, idesc_qk, k > 0);
            }
            mma_commit(&sh->s_full[buf(t, j)]);
          }
          __syncwarp();
        }
      }
      drain_mmas(sh, 0);
    } else if (warp == 3) {
      // ------------------------------------------------------------------ accumulator issuer
      // A_t += P^_t(j) [R^_j | 1] once the codes are written, A_t is rescaled by alpha_j and the
      // row-sum pair of tile j-1 is in place; then the mean term of tile j-1.
      const uint32_t idesc_pv = idesc_e4m3(128, D + 16), idesc_mu = idesc_tf32(128, D);
      const uint64_t dam[2] = {smem_desc_kmajor(smem_u32(sAm), 32), smem_desc_kmajor(smem_u32(sAm + kAmBytes), 32)};
      bool ok = true;
      for (int j = 0; ok && j < nb; ++j) {
        const int st = j % kStages2, it = j / kStages2;
        const int stp = (j + kStages2 - 1) % kStages2;    // stage of tile j-1
        if (!(ok = warp_wait2(&sh->kv_full[st], it & 1, sh, a.wait, 25))) break;
        const uint64_t dv = smem_desc_kmajor(smem_u32(sStage + st * kStageBytes + kKBytes), 128);
        const uint64_t dm = smem_desc_kmajor(smem_u32(sStage + stp * kStageBytes + kKBytes + kVBytes + kOnesBytes), 32);
#pragma unroll
        for (int t = 0; t < (TWO ? 2 : 1); ++t) {
          if (!(ok = warp_wait2(&sh->pc_full[pc_slot(t, j)], pc_par(j), sh, a.wait, 23))) break;
          if (elect_one()) {
            tc_fence_after();
            const uint32_t o_col = tmem + O_COL + O_STRIDE * t;
#pragma unroll
            for (int k = 0; k < 4; ++k) mma_f8_ts(o_col, tmem + P_COL + 32 * buf(t, j) + 8 * k, dv + 2 * k, idesc_pv, (j > 0) | (k > 0));
            if (j > 0 && SMOOTH) mma_tf32_ss(o_col, dam[t], dm, idesc_mu, 1);
            mma_commit(&sh->o_done[buf(t, j)]);
            if (j > 0) mma_commit(&sh->kv_empty[stp]);    // this tile is done with stage j-1
          }
          __syncwarp();
        }
      }
      const uint64_t dml = smem_desc_kmajor(smem_u32(sStage + ((nb - 1) % kStages2) * kStageBytes + kKBytes + kVBytes + kOnesBytes), 32);
#pragma unroll
      for (int t = 0; t < (TWO ? 2 : 1); ++t) {           // mean term of the last tile
        if (!SMOOTH || !ok || !(ok = warp_wait2(&sh->fin_full[t], 0, sh, a.wait, 27))) break;
        if (elect_one()) {
          tc_fence_after();
          mma_tf32_ss(tmem + O_COL + O_STRIDE * t, dam[t], dml, idesc_mu, 1);
          mma_commit(&sh->o_final[t]);
        }
        __syncwarp();
      }
      drain_mmas(sh, 1);
    }
  } else if (warp < (TWO ? 12 : 8)) {
    // -------------------------------------------------------------------- softmax warpgroups
    reg_inc<kRegSoftmax>();
    const int t = TWO ? (warp - 4) >> 2 : 0;               // query tile of this warpgroup
    const int row = (warp & 3) * 32 + lane;
    const int qblk = q0 + t;
    const float sq = qblk < nb ? a.q_scale[(size_t)bh * nb + qblk] : 1.0f;
    const uint32_t alpha_at = smem_u32(&sh->alpha[0][row]);
    float m_run = -INFINITY;
    float sk_next = __ldg(&a.k_scale[(size_t)bh * nb]);   // fetched one tile ahead: an L2 round trip
    for (int j = 0; j < nb; ++j) {
      const float cs = (sq * sk_next) * a.sl;             // code units -> log2 domain
      if (j + 1 < nb) sk_next = __ldg(&a.k_scale[(size_t)bh * nb + j + 1]);
      if (!warp_wait2(&sh->s_full[buf(t, j)], par(j), sh, a.wait, 30)) break;
      tc_fence_after();
      uint32_t s0[32], s1[32], s2[32], s3[32];
      const uint32_t s_col = lane_base + (TWO ? (kTwoS ? t * S1_COL : 0) : (j & 1) * S1_COL);
      if (j == nb - 1 && (a.N & 127)) {                   // ragged last tile: padded keys score -inf
#pragma unroll 1
        for (int c = a.N & 127; c < 128; ++c) tmem_st1(s_col + c, INT8 ? 0xff800000u - 0x4B400000u : 0xff800000u);
        tmem_wait_st();
      }
      tmem_ld32(s_col, s0); tmem_ld32(s_col + 32, s1); tmem_ld32(s_col + 64, s2); tmem_ld32(s_col + 96, s3);
      tmem_wait_ld();
      tc_fence_before();
      mbar_arrive(&sh->s_free[buf(t, j)]);                 // the score buffer may be overwritten
      if constexpr (INT8) {
        // INT32 scores -> FP32, exactly: |s| <= 127 * 127 * 128 < 2^22, so the bits of 1.5 * 2^23 + s
        // are an integer add away, and subtracting the constant is exact.  (The two extra
        // instructions per score are what the E4M3 score product saves on this GPU.)
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          s0[i] = __float_as_uint(__uint_as_float(s0[i] + 0x4B400000u) - 12582912.0f);
          s1[i] = __float_as_uint(__uint_as_float(s1[i] + 0x4B400000u) - 12582912.0f);
          s2[i] = __float_as_uint(__uint_as_float(s2[i] + 0x4B400000u) - 12582912.0f);
          s3[i] = __float_as_uint(__uint_as_float(s3[i] + 0x4B400000u) - 12582912.0f);
        }
      }
      // (never taken: the end of a basic block here keeps the compiler from moving the maxima in front of
      // the release of the score buffer, which costs 4 to 14 percent of the kernel)
      if (a.n_pad < 0) break;
      float mx[8];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        mx[c] = max3(__uint_as_float(s0[16 * c]), __uint_as_float(s0[16 * c + 1]), __uint_as_float(s0[16 * c + 2]));
        mx[2 + c] = max3(__uint_as_float(s1[16 * c]), __uint_as_float(s1[16 * c + 1]), __uint_as_float(s1[16 * c + 2]));
        mx[4 + c] = max3(__uint_as_float(s2[16 * c]), __uint_as_float(s2[16 * c + 1]), __uint_as_float(s2[16 * c + 2]));
        mx[6 + c] = max3(__uint_as_float(s3[16 * c]), __uint_as_float(s3[16 * c + 1]), __uint_as_float(s3[16 * c + 2]));
#pragma unroll
        for (int i = 3; i < 15; i += 2) {
          mx[c] = max3(mx[c], __uint_as_float(s0[16 * c + i]), __uint_as_float(s0[16 * c + i + 1]));
          mx[2 + c] = max3(mx[2 + c], __uint_as_float(s1[16 * c + i]), __uint_as_float(s1[16 * c + i + 1]));
          mx[4 + c] = max3(mx[4 + c], __uint_as_float(s2[16 * c + i]), __uint_as_float(s2[16 * c + i + 1]));
          mx[6 + c] = max3(mx[6 + c], __uint_as_float(s3[16 * c + i]), __uint_as_float(s3[16 * c + i + 1]));
        }
        mx[c] = fmaxf(mx[c], __uint_as_float(s0[16 * c + 15]));
        mx[2 + c] = fmaxf(mx[2 + c], __uint_as_float(s1[16 * c + 15]));
        mx[4 + c] = fmaxf(mx[4 + c], __uint_as_float(s2[16 * c + 15]));
        mx[6 + c] = fmaxf(mx[6 + c], __uint_as_float(s3[16 * c + 15]));
      }
      const float mxa = max3(max3(mx[0], mx[1], mx[2]), max3(mx[3], mx[4], mx[5]), fmaxf(mx[6], mx[7]));
      const float m_new = fmaxf(m_run, mxa * cs);         // m' = max(m, rowmax S_ij)
      sts32(alpha_at + 512 * slot(t, j), ex2_approx(m_run - m_new));      // alpha; 0 on the first tile
      mbar_arrive(&sh->a_full[slot(t, j)]);
      m_run = m_new;
      // the previous code tile must have been consumed before it is overwritten
      if (TWO ? j > 0 && !warp_wait2(&sh->o_done[t], (j - 1) & 1, sh, a.wait, 31) : j > 1 && !warp_wait2(&sh->o_done[j & 1], par(j) ^ 1, sh, a.wait, 31)) break;

      const float fa = cs * 0.0625f, fb = (a.code_off - 8.0f * m_new) * 0.0078125f, nm = 8.0f - m_new;
      const uint64_t fa2 = pack_f32x2(fa, fa), fb2 = pack_f32x2(fb, fb);
      auto code4 = [&](const uint32_t (&sv)[32], int w) -> uint32_t {
        if constexpr (PF == kPfExpCast) {
          // Eq. 7: t = (8 u + 120 + beta) / 128, code = round-to-nearest-even(128 t) clipped at 0
          // (two packed FP32 instructions and a saturating pack per two scores)
          return expcast_codes4(sv[4 * w], sv[4 * w + 1], sv[4 * w + 2], sv[4 * w + 3], fa2, fb2);
        } else {
          // exponentiate, then cast (Fig. 4a upper box): on the special-function unit, on the
          // FMA pipe by a polynomial, or three and one per word
          const float x0 = fmaf(__uint_as_float(sv[4 * w]), cs, nm), x1 = fmaf(__uint_as_float(sv[4 * w + 1]), cs, nm);
          const float x2 = fmaf(__uint_as_float(sv[4 * w + 2]), cs, nm), x3 = fmaf(__uint_as_float(sv[4 * w + 3]), cs, nm);
          float p0, p1, p2, p3;
          if constexpr (PF == kPfExp) {
            p0 = ex2_approx(x0); p1 = ex2_approx(x1); p2 = ex2_approx(x2); p3 = ex2_approx(x3);
          } else if constexpr (PF == kPfExpPoly) {
            p0 = exp2_poly(x0); p1 = exp2_poly(x1); p2 = exp2_poly(x2); p3 = exp2_poly(x3);
          } else {
            p0 = ex2_approx(x0); p1 = ex2_approx(x1); p2 = ex2_approx(x2); p3 = exp2_poly(x3);
          }
          const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(p0, p1), __NV_SATFINITE, __NV_E4M3);
          const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(p2, p3), __NV_SATFINITE, __NV_E4M3);
          return lo | (hi << 16);
        }
      };
      const uint32_t p_col = lane_base + P_COL + 32 * buf(t, j);
      auto store32 = [&](const uint32_t (&sv)[32], int q) {                 // keys 32 q .. + 31
        if constexpr (kSfu) {
          // Four columns a store: with eight, 32 exponentials have to be done before any code leaves (B1 H16 N16384
          // d128, E4M3 / INT8 scores 1639 / 1801 us with eight, 1489 / 1683 with four, 1526 / 1718 with two; codes through
          // shared memory 1582 / 1773).  Without the unit eight are as good or better.
#pragma unroll
          for (int w = 0; w < 8; w += 4) tmem_st4(p_col + 8 * q + w, code4(sv, w), code4(sv, w + 1), code4(sv, w + 2), code4(sv, w + 3));
        } else {
          uint32_t c[8];
#pragma unroll
          for (int w = 0; w < 8; ++w) c[w] = code4(sv, w);
          tmem_st8(p_col + 8 * q, c);
        }
      };
      tc_fence_after();
      store32(s0, 0); store32(s1, 1); store32(s2, 2); store32(s3, 3);
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&sh->pc_full[pc_slot(t, j)]);
    }
  } else if (TWO ? warp >= 12 : warp >= 12 && warp < 16) {
    // -------------------------------------------------------------------- correction warpgroups
    reg_dec<kRegCorr>();
    const int t = TWO ? (warp - 12) >> 2 : 0;
    const int row = (warp & 3) * 32 + lane;
    const int qblk = q0 + t;
    const uint32_t o_base = lane_base + O_COL + O_STRIDE * t;
    // my row of the row-sum operand: 32-byte rows, the two 16-byte chunks swap when (row / 4) is odd
    const uint32_t am_row = smem_u32(sAm + t * kAmBytes + row * 32 + 16 * ((row >> 2) & 1));
    const uint32_t alpha_at = smem_u32(&sh->alpha[0][row]), vs_at = smem_u32(sh->v_scale[t]);
    // s_V of my channel, for everyone in the epilogue: read from global memory there, its eight dependent round trips
    // made the epilogue 2.8 us (B1 H2 N1024 d128 25.4 -> 24.0 us, B1 H6 N1955 d64 28.9 -> 28.1, B1 H12 N32760 d128 without
    // smoothing 3.60 -> 3.55 ms).  The barrier stands here, where every warp of the group comes by, and not where a wait
    // may have given up.
    if (row < D) sts32(vs_at + 4 * row, __ldg(&a.v_scale[(size_t)bh * D + row]));
    asm volatile("bar.sync %0, 128;" ::"r"(1 + t) : "memory");
    float l_resc = 0.f;       // l as it stands in column d after the latest rescale, before the tile's own sum
    float l_now = 0.f;
    bool ok = true;
    auto put_pair = [&](float rho) {                      // (rho_hi, rho_lo, 0, 0) for the mean MMA
      const uint32_t hi = (__float_as_uint(rho) + 0x1000u) & 0xffffe000u;   // nearest TF32
      sts128(am_row, hi, __float_as_uint(rho - __uint_as_float(hi)), 0u, 0u);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    };
    for (int j = 0; j < nb; ++j) {
      if (!(ok = warp_wait2(&sh->a_full[slot(t, j)], slot_par(j), sh, a.wait, 40))) break;
      const float alpha = lds32(alpha_at + 512 * slot(t, j));
      const bool moved = __any_sync(0xffffffffu, alpha != 1.0f);   // a row maximum of the warp moved
      // (without block means nothing needs l tile by tile: a warp whose maxima stand still passes on)
      if (j > 0 && (SMOOTH || moved)) {
        if (!(ok = warp_wait2(&sh->o_done[buf(t, j - 1)], par(j - 1), sh, a.wait, 41))) break;
        tc_fence_after();
        l_now = __uint_as_float(tmem_ld1(o_base + L_COL));   // l after tile j-1
        tmem_wait_ld();
        const float r_prev = l_now - l_resc;                 // r_{j-1} = P~ 1 over the decoded codes
        if (moved) {                                         // A <- alpha A (l included)
          uint32_t r[16];
#pragma unroll 1
          for (int c = 0; c < D / 16; ++c) {
            tmem_ld16(o_base + 16 * c, r);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; i += 2) unpack_b32x2(mul2(pack_b32x2(r[i], r[i + 1]), pack_f32x2(alpha, alpha)), r[i], r[i + 1]);
            tmem_st16(o_base + 16 * c, r);
          }
          // of the 16 row-sum columns only column d is ever read, and its value is at hand
          tmem_st1(o_base + L_COL, __float_as_uint(l_now * alpha));
          tmem_wait_st();
          tc_fence_before();
        }
        l_resc = l_now * alpha;
        if (SMOOTH) put_pair(r_prev * alpha);              // added after the rescale, so referenced to m_j
      }
      // Without block means a warp may come here without having waited for the product in front of the last one
      // on the last one's barrier, and the wait below would take that phase for the last.  The wait for
      // it stands in front of the last arrival: behind it both phases may be over before this warp looks.
      const int before = j - (TWO ? 1 : 2);
      if (!SMOOTH && j == nb - 1 && before >= 0 && !(ok = warp_wait2(&sh->o_done[buf(t, before)], par(before), sh, a.wait, 44))) break;
      mbar_arrive(&sh->pc_full[pc_slot(t, j)]);
    }
    // ---- last tile's mean term, then the epilogue: O = s_V * A / l
    if (ok && (ok = warp_wait2(&sh->o_done[buf(t, nb - 1)], par(nb - 1), sh, a.wait, 42))) {
      tc_fence_after();
      l_now = __uint_as_float(tmem_ld1(o_base + L_COL));
      tmem_wait_ld();
      if (SMOOTH) {
        put_pair(l_now - l_resc);
        mbar_arrive(&sh->fin_full[t]);
      }
    }
    if (ok && (!SMOOTH || warp_wait2(&sh->o_final[t], 0, sh, a.wait, 43))) {
      tc_fence_after();
      static_assert(kStageBytes >= 128 * 2 * D, "a query tile's output fits a stage");
      using Out = OutTile<D>;
      const int row0 = qblk * 128 + (warp & 3) * 32;       // the warp's first row
      const uint32_t tile = smem_u32(sStage + ((nb + t) % kStages2) * kStageBytes) + (warp & 3) * 32 * Out::ROW;
      const float inv_l = 1.0f / l_now;
#pragma unroll 1
      for (int c = 0; c < D / 16; ++c) {
        uint32_t r[16], out[8];
        tmem_ld16(o_base + 16 * c, r);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 s4 = lds128(vs_at + 64 * c + 16 * i);
          const __nv_bfloat162 h0 = __floats2bfloat162_rn(__uint_as_float(r[4 * i]) * inv_l * s4.x, __uint_as_float(r[4 * i + 1]) * inv_l * s4.y);
          const __nv_bfloat162 h1 = __floats2bfloat162_rn(__uint_as_float(r[4 * i + 2]) * inv_l * s4.z, __uint_as_float(r[4 * i + 3]) * inv_l * s4.w);
          out[2 * i] = *reinterpret_cast<const uint32_t*>(&h0);
          out[2 * i + 1] = *reinterpret_cast<const uint32_t*>(&h1);
        }
        sts128(Out::chunk(tile, lane, 2 * c), out[0], out[1], out[2], out[3]);
        sts128(Out::chunk(tile, lane, 2 * c + 1), out[4], out[5], out[6], out[7]);
      }
      Out::store(tile, reinterpret_cast<unsigned char*>(a.o + ((size_t)bh * a.N + row0) * D), 2 * D, a.N - row0, lane);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) tmem_dealloc<kTmemCols>(tmem);
}


// CTAs [0, n_pair) take pairs of query tiles, the rest one tile each; a head's odd last tile is alone
// either way.
template <int D, int PF, bool INT8, bool SMOOTH, bool ONE>
__global__ void __launch_bounds__(640, 1)
attn_fwd_2q_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                   const __grid_constant__ CUtensorMap tm_v, const AttnArgs a) {
  const TileOf w = tile_of(a.tiles, a.nb);
  if (w.q0 >= a.nb) return;                 // the missing second tile of a head's last pair
  if constexpr (ONE) {
    if (!w.two) {
      attn_2q_body<D, PF, INT8, SMOOTH, false>(tm_q, tm_k, tm_v, a, w.q0, w.bh);
      return;
    }
  }
  attn_2q_body<D, PF, INT8, SMOOTH, true>(tm_q, tm_k, tm_v, a, w.q0, w.bh);
}

template <int D>
cudaError_t run_2q(const Problem& pr, const QuantLayout& ql, const WorkLayout& wl, const uint8_t* quant, void* o, uint8_t* work,
                   cudaStream_t s) {
  alignas(64) CUtensorMap tq, tk, tv;
  AttnArgs a{};
  if (!fill_args8<D>(pr, ql, wl, quant, o, work, &a, &tq, &tk, &tv)) return cudaErrorUnknown;
  constexpr size_t stage = 2 * 128 * D + 2048 + ((D * 32 + 1023) / 1024) * 1024;
  constexpr size_t smem = 2 * 128 * D + 2 * 128 * 32 + kStages2 * stage + sizeof(FaSmem);
  static_assert(smem <= 227 * 1024, "shared memory of the kernel exceeds the SM");
  const bool int8 = pr.flags & VC_FLAG_INT8_QK, smooth = pr.flags & VC_FLAG_V_SMOOTH;
  const int pf = pr.p_format == VC_P_EXPCAST_E4M3 ? kPfExpCast
                 : pr.p_format == VC_P_EXP_E4M3   ? kPfExp
                 : pr.p_format == VC_P_EXP_POLY_E4M3 ? kPfExpPoly : kPfExpMix;
  if (int8 && pf > kPfExp) return cudaErrorNotSupported;
  unsigned grid;
  a.tiles = split_tiles(pr, pf == kPfExpCast, &grid);
#define VC_LAUNCH_2Q(...)                                                                                      \
  ((e = allow_smem<attn_fwd_2q_kernel<D, __VA_ARGS__>>()) == cudaSuccess                                       \
       ? (e = launch_overlapped(attn_fwd_2q_kernel<D, __VA_ARGS__>, dim3(grid), 640, smem, s, tq, tk, tv, a)) \
       : e)
  cudaError_t e = cudaSuccess;
  if (pf == kPfExpCast) {
    if (smooth) int8 ? VC_LAUNCH_2Q(kPfExpCast, true, true, true) : VC_LAUNCH_2Q(kPfExpCast, false, true, true);
    else int8 ? VC_LAUNCH_2Q(kPfExpCast, true, false, true) : VC_LAUNCH_2Q(kPfExpCast, false, false, true);
  }
  // (the other formats exist for comparison: always pairs, and means of zero are added)
  else if (pf == kPfExp) int8 ? VC_LAUNCH_2Q(kPfExp, true, true, false) : VC_LAUNCH_2Q(kPfExp, false, true, false);
  else if (pf == kPfExpPoly) VC_LAUNCH_2Q(kPfExpPoly, false, true, false);
  else VC_LAUNCH_2Q(kPfExpMix, false, true, false);
#undef VC_LAUNCH_2Q
  if (e != cudaSuccess) return e;
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace
}  // namespace vc

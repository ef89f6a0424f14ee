// 4-bit attention forward of VC-Attention on block-scaled FP4 tensor-core instructions
// (App. A "Scope of ExpCast-FP8", App. B: NVFP4 Q, K, R and P).
//
// Every operand of both products is NVFP4 as vc_prep wrote it - E2M1 elements, two per byte,
// under an unsigned E4M3 factor per 16 elements along the contraction axis - and both products
// run as tcgen05.mma kind::mxf4nvf4 (K = 64 per instruction), which multiplies each 16-element
// partial sum by the two factors.  The factors live in tensor memory; tcgen05.cp brings them
// there from shared memory in 512-byte chunks (128 operand rows x 4 groups).  The producer warp
// reads a tile's factors from the bundle's row-major arrays and writes them in chunk order.
//
// The pipeline is the one of the 8-bit kernel (two query tiles per CTA, one shared score
// buffer, probability codes through tensor memory, the row sums l from 16 rows of ones behind
// the value tile, the block-mean term as a TF32 MMA one tile late).  What differs is the
// softmax stage: P is quantized to NVFP4 per row and 16 keys.  The group maxima are a
// by-product of the running-max pass; per group the E4M3 factor of max p / 6 is formed once,
// its log2 is folded into the exponent offset, and an element costs one FMA, one ex2 and half a conversion:
// code = E2M1(2^(s cs + log2 2688 - m' - log2 f_g)).  Some of the groups take a polynomial in place of the ex2 (see
// vc_nvfp4_codes.cuh), because the special-function unit is what the stage waits for.  (A polynomial that is an
// exponential, with its range reduction, was slower: ten instructions an element instead of three and a half.)
//
// HYB = true is the hybrid 4-bit arrangement: the score product stays NVFP4, but P is the
// ExpCast-FP8 code of Eq. 7 (five instructions per four scores, as in the 8-bit kernel) and the value product
// runs as kind::mxf8f6f4: E4M3 P^ times E2M1 R^ under power-of-two factors per 32 tokens.  The
// value tile arrives through a 4-bit tensor map that spreads it into the 16-byte containers
// that instruction kind reads; P^ carries the constant factor 1.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "vc_attn_shared.cuh"
#include "vc_internal.h"
#include "vc_launch.h"
#include "vc_nvfp4_codes.cuh"
#include "vc_sm100.cuh"

namespace vc {
namespace {

using namespace sm100;
using namespace attn;

// Factors in MMA chunk order: chunk byte 16 (r % 32) + 4 (r / 32) + k is the factor of operand row r,
// group 4 kb + k.  A lane takes rows lane, lane + 32, lane + 64, lane + 96 of the 128: their four
// words are 16 consecutive bytes of the chunk, one store.  (A launch that rewrote the arrays into
// chunks for bulk copies cost 7 us and 2 x 9 MB at B1 H12 N32760 d128.)
template <int W> struct FactorRows {   // W words (of four factors) per row
  uint32_t w[4][W];
  __device__ __forceinline__ void fetch_row(int i, const uint8_t* src) {
    if constexpr (W == 2) {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(src));
      w[i][0] = v.x; w[i][1] = v.y;
    } else {
      w[i][0] = __ldg(reinterpret_cast<const uint32_t*>(src));
    }
  }
  // 128 rows of consecutive bytes (Q^ and K^: rows are tokens, groups run along channels)
  __device__ __forceinline__ void fetch_tokens(const uint8_t* tile, int lane) {
#pragma unroll
    for (int i = 0; i < 4; ++i) fetch_row(i, tile + (size_t)(lane + 32 * i) * (4 * W));
  }
  // rows are channels, groups run along tokens; the 16 rows behind the channels are the rows of ones
  template <int D> __device__ __forceinline__ void fetch_channels(const uint8_t* first, size_t pitch, uint32_t one, int lane) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (32 * i < D) fetch_row(i, first + (size_t)(lane + 32 * i) * pitch);
      else {
#pragma unroll
        for (int k = 0; k < W; ++k) w[i][k] = 32 * i == D && lane < 16 ? one : 0u;
      }
    }
  }
  __device__ __forceinline__ void store(unsigned char* chunks, int lane) const {
#pragma unroll
    for (int k = 0; k < W; ++k) *reinterpret_cast<uint4*>(chunks + 512 * k + 16 * lane) = make_uint4(w[0][k], w[1][k], w[2][k], w[3][k]);
  }
};

struct Attn4Args {
  const float *q_g, *k_g;          // NVFP4 outer scales per (b, h)
  const uint8_t *q_micro, *k_micro, *v_micro;
  const __nv_bfloat16* v_means;
  __nv_bfloat16* o;
  uint32_t* status;
  int N, n_pad, nb;
  Tiles tiles;
  float sl;                        // softmax_scale * log2(e)
  float code_off;                  // 120 + beta  (Eq. 7; hybrid arrangement only)
  WaitArgs wait;
};

// One query tile or pair of tiles (TWO) of head bh, first tile q0.
//   warp 0        TMA producer: Q^ tiles and their factors once; per key tile K^_j, R^_j, the
//                 tile's factor chunks and block mean through a 4-stage ring
//   warp 1        score issuer:        S = Q^_t K^_j^T            D/64 x kind::mxf4nvf4
//   warp 3        accumulator issuer:  A_t += P^_t(j) [R^_j | 1]  2 x kind::mxf4nvf4, N = d + 16
//                                      A_t += rho_{j-1} mu_{j-1}  1 x kind::tf32
//   warps 4-11    softmax warpgroups (tile 0, tile 1), one thread per query row
//   warps 12-19   correction warpgroups, one thread per query row
// Tensor memory: S (128 columns) | A_0 (d + 16) | A_1 (d + 16) | scale factors (56 columns; HYB 32) | P_0 | P_1 (16 each; HYB 32).
// The codes are the A operand of the value product there.  Through shared memory, where the copies and both operands
// of the score product meet, B1 H40 N32760 d128 took 11.69 ms instead of 11.20 (hybrid), B1 H24 N118800 83.3
// instead of 80.1, and B1 H12 N32760 4.49 instead of 4.45 (NVFP4).
template <int D, bool HYB, bool SMOOTH, bool POLY, bool TWO>
__device__ __forceinline__ void attn4_2q_body(const CUtensorMap& tm_q, const CUtensorMap& tm_k, const CUtensorMap& tm_v,
                                              const Attn4Args& a, const int q0, const int bh) {
  constexpr int kTmemCols = 512;
  constexpr int KB = D / 64;                        // K = 64 steps of the score product
  constexpr int kRowB = D / 2;                      // bytes per Q^/K^ row
  // d = 64 leaves room for a score buffer per query tile.  (B2 H16 N16384: hybrid 1.89 -> 1.88 ms; the
  // NVFP4 probabilities, which keep a softmax warp busy twice as long, lose by it: 3.44 -> 3.64.)
  constexpr bool kTwoS = D == 64 && HYB;
  constexpr uint32_t O_COL = kTwoS ? 256 : 128, O_STRIDE = D + 16, L_COL = D, S1_COL = kTwoS ? 128 : O_COL + O_STRIDE;
  constexpr uint32_t SF_COL = 416;
  // (HYB: P^ takes the factor 1 for every row, and so do the rows of ones, value rows 128..143: one chunk serves both)
  constexpr uint32_t SFQ_COL = SF_COL, SFK_COL = SF_COL + 16, SFV_COL = SF_COL + (HYB ? 24 : 40), SFP_COL = SF_COL + (HYB ? 28 : 24);
  constexpr uint32_t P_COL = SF_COL + (HYB ? 32 : 56), kPCols = HYB ? 32 : 16;
  static_assert(P_COL + 2 * kPCols <= kTmemCols, "tensor memory of the 4-bit kernel");
  // (the NVFP4 softmax wants the larger share: B1 H12 N32760 d128 4.44 -> 4.39 ms)
  constexpr int kRegCtl = 48, kRegSoftmax = HYB ? 160 : 168, kRegCorr = HYB ? 56 : 48;
  static_assert(kRegCtl + 2 * kRegSoftmax + 2 * kRegCorr <= 5 * 96, "register budget exceeds the CTA's allocation");
  constexpr int NVC = HYB ? 1 : 2;                  // value factor chunks per key tile
  constexpr uint32_t kVRow = HYB ? 128 : 64;        // bytes of a value row in shared memory
  constexpr uint32_t kQBytes = 128 * kRowB, kKBytes = 128 * kRowB, kVBytes = D * kVRow, kOnesBytes = 16 * kVRow;
  constexpr uint32_t kVTx = D * 64;                 // bytes the value copy reports (the packed ones)
  constexpr uint32_t kMuBytes = D * 32, kMuPad = ((kMuBytes + 1023) / 1024) * 1024;
  constexpr uint32_t kSfBytes = (KB + NVC) * 512, kSfPad = ((kSfBytes + 1023) / 1024) * 1024;
  constexpr uint32_t kStageBytes = kKBytes + kVBytes + kOnesBytes + kMuPad + kSfPad;
  constexpr uint32_t kSfpBytes = 1024, kAmBytes = 128 * 32;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* sQ = smem;                                    // [2][128 x D/2]
  unsigned char* sAm = sQ + 2 * kQBytes;                       // [2][128 x 8 fp32] row-sum pairs
  unsigned char* sSfq = sAm + 2 * kAmBytes;                    // [2][KB][512] Q^ factors
  unsigned char* sSfp = sSfq + 2 * 1024;                       // [2][2][512]  P^ factors (HYB: unused)
  unsigned char* sSfOnes = sSfp + 2 * kSfpBytes;               // [512] factors of value rows 128..143, then the table of logarithms
  float* sLg2 = reinterpret_cast<float*>(sSfOnes + 512);       // [128] log2 of the E4M3 values
  unsigned char* sStage = sSfOnes + 1024;                      // [kStages2]{K, V | ones, Mu, factors}
  FaSmem* sh = reinterpret_cast<FaSmem*>(sStage + kStages2 * kStageBytes);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nb = a.nb;
  // (one tile: double buffers, as in the 8-bit kernel)
  // buffer (and barrier) of scores, codes and products of key tile j, and the parity of its phase
  auto buf = [](int t, int j) { return TWO ? t : j & 1; };
  auto par = [](int j) { return TWO ? j & 1 : (j >> 1) & 1; };
  // slot of the hand-offs of alpha and of codes and correction (see FaSmem), and the parity of its phase
  auto slot = [](int t, int j) { return TWO ? 2 * t + (j & 1) : j & 3; };
  auto slot_par = [](int j) { return TWO ? (j >> 1) & 1 : (j >> 2) & 1; };

  const int early = min(kStages2, nb);      // key tiles whose copies are issued before anything else happens
  if (tid == 0) {
    init_barriers(sh, TWO);
    pdl_wait();                             // the bundle is complete from here on
    mbar_expect_tx_only(&sh->q_full, (TWO ? 2 : 1) * kQBytes);
    tma_load_3d(sQ, &tm_q, &sh->q_full, 0, q0 * 128, bh);
    if (TWO) tma_load_3d(sQ + kQBytes, &tm_q, &sh->q_full, 0, (q0 + 1) * 128, bh);   // past the end: zero fill
    for (int j = 0; j < early; ++j) {
      mbar_expect_tx_only(&sh->kv_full[j], kKBytes + kVTx);
      tma_load_3d(sStage + j * kStageBytes, &tm_k, &sh->kv_full[j], 0, j * 128, bh);
      tma_load_3d(sStage + j * kStageBytes + kKBytes, &tm_v, &sh->kv_full[j], HYB ? j * 128 : j * 64, 0, bh);   // elements resp. bytes
    }
  }
  for (int i = tid; i < 2 * (int)kAmBytes / 16; i += 640) reinterpret_cast<uint4*>(sAm)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < kStages2 * (int)kMuBytes / 16; i += 640)
    reinterpret_cast<uint4*>(sStage + (i / (kMuBytes / 16)) * kStageBytes + kKBytes + kVBytes + kOnesBytes)[i % (kMuBytes / 16)] = make_uint4(0, 0, 0, 0);
  // 16 rows of E2M1 1.0 (two per byte) behind every value tile; their factor chunk: 1.0 for
  // rows 0..15 of the second 128-row half, group bytes 0..3
  // (HYB: the same bytes, of which the product reads the low 8 of every 16; factor code 127 = 2^0,
  // and a chunk of that code for every row of P^)
  for (int i = tid; i < kStages2 * (int)kOnesBytes / 16; i += 640)
    reinterpret_cast<uint4*>(sStage + (i / (kOnesBytes / 16)) * kStageBytes + kKBytes + kVBytes)[i % (kOnesBytes / 16)] = make_uint4(0x22222222u, 0x22222222u, 0x22222222u, 0x22222222u);
  for (int i = tid; i < 128; i += 640)
    reinterpret_cast<uint32_t*>(sSfOnes)[i] = HYB ? 0x7f7f7f7fu : ((i & 3) == 0 && i < 64) ? 0x38383838u : 0u;
  if constexpr (!HYB)                                          // (no lane takes code 127, the NaN)
    for (int i = tid; i < 128; i += 640) sLg2[i] = nvfp4::log2_entry(i);
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
      // (the whole warp runs the loop: one elected lane issues the copies, all write factors and means)
      FactorRows<KB> fq;
#pragma unroll 1
      for (int t = 0; t < (TWO ? 2 : 1); ++t) {            // (past the end: zero codes, any factors)
        fq.fetch_tokens(a.q_micro + ((size_t)bh * a.n_pad + min(q0 + t, nb - 1) * 128) * (D / 16), lane);
        fq.store(sSfq + t * 1024, lane);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");          // the stores -> tensor-core reads
      __syncwarp();
      if (elect_one()) mbar_arrive(&sh->q_full);
      int j = 0;
      for (; j < nb; ++j) {
        const int st = j % kStages2, it = j / kStages2;
        unsigned char* base = sStage + st * kStageBytes;
        unsigned char* extra = base + kKBytes + kVBytes + kOnesBytes;       // block mean, then the factor chunks
        FactorRows<KB> fk;
        FactorRows<NVC> fv;
        MeanRows<D> mu;
        fk.fetch_tokens(a.k_micro + ((size_t)bh * a.n_pad + j * 128) * (D / 16), lane);
        if (HYB) fv.template fetch_channels<D>(a.v_micro + (size_t)bh * D * (a.n_pad / 32) + j * 4, a.n_pad / 32, 0x7f7f7f7fu, lane);
        else fv.template fetch_channels<D>(a.v_micro + (size_t)bh * D * (a.n_pad / 16) + j * 8, a.n_pad / 16, 0x38383838u, lane);
        if (SMOOTH) mu.fetch(a.v_means + ((size_t)bh * nb + j) * D, lane);
        if (!warp_wait2(&sh->kv_empty[st], (it & 1) ^ 1, sh, a.wait, 11)) break;
        if (j >= early && elect_one()) {
          mbar_expect_tx_only(&sh->kv_full[st], kKBytes + kVTx);
          tma_load_3d(base, &tm_k, &sh->kv_full[st], 0, j * 128, bh);
          tma_load_3d(base + kKBytes, &tm_v, &sh->kv_full[st], HYB ? j * 128 : j * 64, 0, bh);   // elements resp. bytes
        }
        fk.store(extra + kMuPad, lane);
        fv.store(extra + kMuPad + KB * 512, lane);
        if (SMOOTH) mu.store(extra, lane);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");        // the stores -> tensor-core reads
        __syncwarp();
        if (elect_one()) mbar_arrive(&sh->kv_full[st]);
        __syncwarp();
      }
      drain_loads(sh, j);                                 // (returns at once on a normal run)
    } else if (warp == 1) {
      // ------------------------------------------------------------------ score issuer
      const uint32_t idesc_qk = idesc_nvfp4(128, 128);
      const uint64_t dq0 = smem_desc_kmajor(smem_u32(sQ), kRowB), dq1 = smem_desc_kmajor(smem_u32(sQ + kQBytes), kRowB);
      bool ok = warp_wait2(&sh->q_full, 0, sh, a.wait, 20);
      if (ok && elect_one()) {
        for (int t = 0; t < (TWO ? 2 : 1); ++t)
          for (int kb = 0; kb < KB; ++kb)
            tmem_cp_sf(tmem + SFQ_COL + (t * KB + kb) * 4, smem_desc_sf_chunk(smem_u32(sSfq + t * 1024 + kb * 512)));
      }
      __syncwarp();
      for (int j = 0; ok && j < nb; ++j) {
        const int st = j % kStages2, it = j / kStages2;
        if (!(ok = warp_wait2(&sh->kv_full[st], it & 1, sh, a.wait, 21))) break;
        const unsigned char* base = sStage + st * kStageBytes;
        const uint64_t dk = smem_desc_kmajor(smem_u32(base), kRowB);
        const uint32_t sf_smem = smem_u32(base + kKBytes + kVBytes + kOnesBytes + kMuPad);
#pragma unroll
        for (int t = 0; t < (TWO ? 2 : 1); ++t) {
          if (TWO && kTwoS) {
            if (j > 0 && !(ok = warp_wait2(&sh->s_free[t], (j - 1) & 1, sh, a.wait, 22))) break;
          } else if (TWO ? (t == 0 ? j > 0 : true) : j > 1) {
            if (!(ok = warp_wait2(&sh->s_free[TWO ? 1 - t : j & 1], TWO ? (t == 0 ? j - 1 : j) & 1 : par(j) ^ 1, sh, a.wait, 22))) break;
          }
          if (elect_one()) {
            tc_fence_after();
            if (t == 0) {
#pragma unroll
              for (int kb = 0; kb < KB; ++kb) tmem_cp_sf(tmem + SFK_COL + kb * 4, smem_desc_sf_chunk(sf_smem + kb * 512));
            }
            const uint64_t dq = t == 0 ? dq0 : dq1;
#pragma unroll
            for (int kb = 0; kb < KB; ++kb)
              mma_nvfp4_ss(tmem + (TWO ? (kTwoS ? t * S1_COL : 0) : (j & 1) * S1_COL), dq + 2 * kb, dk + 2 * kb, idesc_qk, kb > 0, tmem + SFQ_COL + (t * KB + kb) * 4,
                           tmem + SFK_COL + kb * 4);
            mma_commit(&sh->s_full[buf(t, j)]);
          }
          __syncwarp();
        }
      }
      drain_mmas(sh, 0);
    } else if (warp == 3) {
      // ------------------------------------------------------------------ accumulator issuer
      const uint32_t idesc_pv = idesc_nvfp4(128, D + 16), idesc_mu = idesc_tf32(128, D);
      const uint64_t dam[2] = {smem_desc_kmajor(smem_u32(sAm), 32), smem_desc_kmajor(smem_u32(sAm + kAmBytes), 32)};
      if (elect_one()) {
        if (HYB) {                                         // P^, and at d = 128 the rows of ones
          tmem_cp_sf(tmem + SFP_COL, smem_desc_sf_chunk(smem_u32(sSfOnes)));
        } else if (D == 128) {                             // factors of the rows of ones (value rows 128..143)
          tmem_cp_sf(tmem + SFV_COL + 4, smem_desc_sf_chunk(smem_u32(sSfOnes)));
          tmem_cp_sf(tmem + SFV_COL + 12, smem_desc_sf_chunk(smem_u32(sSfOnes)));
        }
      }
      __syncwarp();
      bool ok = true;
      for (int j = 0; ok && j < nb; ++j) {
        const int st = j % kStages2, it = j / kStages2;
        const int stp = (j + kStages2 - 1) % kStages2;    // stage of tile j-1
        if (!(ok = warp_wait2(&sh->kv_full[st], it & 1, sh, a.wait, 25))) break;
        const unsigned char* base = sStage + st * kStageBytes;
        const uint64_t dv = smem_desc_kmajor(smem_u32(base + kKBytes), kVRow);
        const uint64_t dm = smem_desc_kmajor(smem_u32(sStage + stp * kStageBytes + kKBytes + kVBytes + kOnesBytes), 32);
        const uint32_t sfv_smem = smem_u32(base + kKBytes + kVBytes + kOnesBytes + kMuPad + KB * 512);
#pragma unroll
        for (int t = 0; t < (TWO ? 2 : 1); ++t) {
          if (!(ok = warp_wait2(&sh->pc_full[slot(t, j)], slot_par(j), sh, a.wait, 23))) break;
          if (elect_one()) {
            tc_fence_after();
            const uint32_t o_col = tmem + O_COL + O_STRIDE * t;
            const int b = buf(t, j);
            const uint32_t p_at = tmem + P_COL + kPCols * b;
            if constexpr (HYB) {
              if (t == 0) tmem_cp_sf(tmem + SFV_COL, smem_desc_sf_chunk(sfv_smem));
#pragma unroll
              for (int k = 0; k < 4; ++k)                  // 32 keys each; factor byte k of the value rows
                mma_mxf8_ts(o_col, p_at + 8 * k, dv + 2 * k, idesc_mxf8_e4m3_e2m1(128, D + 16, k), (j > 0) | (k > 0),
                            tmem + SFP_COL, tmem + SFV_COL);
            } else {
              if (t == 0) {
                tmem_cp_sf(tmem + SFV_COL, smem_desc_sf_chunk(sfv_smem));
                tmem_cp_sf(tmem + SFV_COL + 8, smem_desc_sf_chunk(sfv_smem + 512));
              }
              tmem_cp_sf(tmem + SFP_COL + b * 8, smem_desc_sf_chunk(smem_u32(sSfp + b * kSfpBytes)));
              tmem_cp_sf(tmem + SFP_COL + b * 8 + 4, smem_desc_sf_chunk(smem_u32(sSfp + b * kSfpBytes + 512)));
#pragma unroll
              for (int kb = 0; kb < 2; ++kb)
                mma_nvfp4_ts(o_col, p_at + 8 * kb, dv + 2 * kb, idesc_pv, (j > 0) | (kb > 0), tmem + SFP_COL + b * 8 + kb * 4,
                             tmem + SFV_COL + kb * 8);
            }
            if (j > 0 && SMOOTH) mma_tf32_ss(o_col, dam[t], dm, idesc_mu, 1);
            mma_commit(&sh->o_done[b]);
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
    const uint32_t sfp_row = smem_u32(sSfp + t * kSfpBytes + (row & 31) * 16 + (row >> 5) * 4);
    const float cs = (a.q_g[bh] * a.k_g[bh]) * a.sl;       // code units -> log2 domain
    const uint32_t lg2_at = smem_u32(sLg2);
    const uint32_t alpha_at = smem_u32(&sh->alpha[0][row]);
    float m_run = -INFINITY;
    for (int j = 0; j < nb; ++j) {
      if (!warp_wait2(&sh->s_full[buf(t, j)], par(j), sh, a.wait, 30)) break;
      tc_fence_after();
      uint32_t s0[32], s1[32], s2[32], s3[32];
      const uint32_t s_col = lane_base + (TWO ? (kTwoS ? t * S1_COL : 0) : (j & 1) * S1_COL);
      if (j == nb - 1 && (a.N & 127)) {                   // ragged last tile: padded keys score -inf
#pragma unroll 1
        for (int c = a.N & 127; c < 128; ++c) tmem_st1(s_col + c, 0xff800000u);
        tmem_wait_st();
      }
      tmem_ld32(s_col, s0); tmem_ld32(s_col + 32, s1); tmem_ld32(s_col + 64, s2); tmem_ld32(s_col + 96, s3);
      tmem_wait_ld();
      tc_fence_before();
      mbar_arrive(&sh->s_free[buf(t, j)]);                 // the score buffer may be overwritten
      // (never taken: the end of a basic block here keeps the compiler from moving the maxima in front of
      // the release of the score buffer, which costs 4 to 14 percent of the hybrid kernel; with NVFP4
      // probabilities the exponentials hide it, and the larger block is 2.4 percent faster)
      if (HYB && a.n_pad < 0) break;
      float mx[8];                                        // maxima of the eight 16-key groups
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
      if constexpr (HYB) {
        // ExpCast-FP8 (Eq. 7): t = (8 u + 120 + beta) / 128, code = round-to-nearest-even(128 t)
        // clipped at 0 (two packed FP32 instructions and a saturating pack per two scores)
        if (TWO ? j > 0 && !warp_wait2(&sh->o_done[t], (j - 1) & 1, sh, a.wait, 31) : j > 1 && !warp_wait2(&sh->o_done[j & 1], par(j) ^ 1, sh, a.wait, 31)) break;
        const float fa = cs * 0.0625f, fb = (a.code_off - 8.0f * m_new) * 0.0078125f;
        const uint64_t fa2 = pack_f32x2(fa, fa), fb2 = pack_f32x2(fb, fb);
        auto code4 = [&](const uint32_t (&sv)[32], int w) -> uint32_t {
          return expcast_codes4(sv[4 * w], sv[4 * w + 1], sv[4 * w + 2], sv[4 * w + 3], fa2, fb2);
        };
        const uint32_t p_col = lane_base + P_COL + kPCols * buf(t, j);
        auto store32 = [&](const uint32_t (&sv)[32], int q) {               // keys 32 q .. + 31, four a column
          uint32_t c[8];
#pragma unroll
          for (int w = 0; w < 8; ++w) c[w] = code4(sv, w);
          tmem_st8(p_col + 8 * q, c);
        };
        tc_fence_after();
        store32(s0, 0); store32(s1, 1); store32(s2, 2); store32(s3, 3);
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&sh->pc_full[slot(t, j)]);
        continue;
      }
      // NVFP4 (see nvfp4::Row; POLY: some groups' codes by the polynomial)
      const nvfp4::Row<D, POLY> nv(cs, m_new, lg2_at);
      uint32_t sfw[2] = {0u, 0u};
      float off[8];
      // Six factors in front of the wait, two behind it, where they overlap the first exponentials (four and
      // four at d = 64): B1 H12 N32760 d128 4.33 ms with six, 4.39 with four, 4.47 with none;
      // B2 H16 N16384 d64 2.83 with six, 2.75 with four, 2.79 with none
      constexpr int kAhead = D == 128 ? 6 : 4;
#pragma unroll
      for (int g = 0; g < kAhead; g += 2) nv.factors(g, mx, sfw, off);
      // the previous code tile must have been consumed before it is overwritten
      if (TWO ? j > 0 && !warp_wait2(&sh->o_done[t], (j - 1) & 1, sh, a.wait, 31) : j > 1 && !warp_wait2(&sh->o_done[j & 1], par(j) ^ 1, sh, a.wait, 31)) break;
#pragma unroll
      for (int g = kAhead; g < 8; g += 2) nv.factors(g, mx, sfw, off);
      const uint32_t p_col = lane_base + P_COL + kPCols * buf(t, j);
      auto store32 = [&](const uint32_t (&sv)[32], int q) {       // keys 32 q .. + 31, eight a column
        const uint2 lo = nv.codes16(sv, 0, 2 * q, off), hi = nv.codes16(sv, 1, 2 * q + 1, off);
        tmem_st4(p_col + 4 * q, lo.x, lo.y, hi.x, hi.y);
      };
      tc_fence_after();
      store32(s0, 0); store32(s1, 1); store32(s2, 2); store32(s3, 3);
      sts32(sfp_row + (TWO ? 0 : (j & 1) * kSfpBytes), __uint_as_float(sfw[0]));
      sts32(sfp_row + (TWO ? 0 : (j & 1) * kSfpBytes) + 512, __uint_as_float(sfw[1]));                               // the chunk of keys 64..127
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");          // the factors -> tensor-core reads
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&sh->pc_full[slot(t, j)]);
    }
  } else if (TWO ? warp >= 12 : warp >= 12 && warp < 16) {
    // -------------------------------------------------------------------- correction warpgroups
    reg_dec<kRegCorr>();
    const int t = TWO ? (warp - 12) >> 2 : 0;
    const int row = (warp & 3) * 32 + lane;
    const int qblk = q0 + t;
    const uint32_t o_base = lane_base + O_COL + O_STRIDE * t;
    const uint32_t am_row = smem_u32(sAm + t * kAmBytes + row * 32 + 16 * ((row >> 2) & 1));
    const uint32_t alpha_at = smem_u32(&sh->alpha[0][row]);
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
        const float r_prev = l_now - l_resc;                 // r_{j-1}: sum of the decoded codes
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
        if (SMOOTH) put_pair(r_prev * alpha);
      }
      // Without block means a warp may come here without having waited for the product in front of the last one
      // on the last one's barrier, and the wait below would take that phase for the last.  The wait for
      // it stands in front of the last arrival: behind it both phases may be over before this warp looks.
      const int before = j - (TWO ? 1 : 2);
      if (!SMOOTH && j == nb - 1 && before >= 0 && !(ok = warp_wait2(&sh->o_done[buf(t, before)], par(before), sh, a.wait, 44))) break;
      mbar_arrive(&sh->pc_full[slot(t, j)]);
    }
    // ---- last tile's mean term, then the epilogue: O = A / l (means are unscaled at 4 bits, App. B)
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
      constexpr int W = kStageBytes >= 128 * 2 * D ? D : D / 2;          // output columns of a query tile that fit a stage
      static_assert(kStageBytes >= 128 * 2 * W, "half a query tile's output fits a stage");
      using Out = OutTile<W>;
      const int row0 = qblk * 128 + (warp & 3) * 32;       // the warp's first row
      const uint32_t tile = smem_u32(sStage + ((nb + t) % kStages2) * kStageBytes) + (warp & 3) * 32 * Out::ROW;
      const float inv_l = 1.0f / l_now;
#pragma unroll 1
      for (int h = 0; h < D; h += W) {
#pragma unroll 1
        for (int c = 0; c < W / 16; ++c) {
          uint32_t r[16], out[8];
          tmem_ld16(o_base + h + 16 * c, r);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(r[2 * i]) * inv_l, __uint_as_float(r[2 * i + 1]) * inv_l);
            out[i] = *reinterpret_cast<uint32_t*>(&h2);
          }
          sts128(Out::chunk(tile, lane, 2 * c), out[0], out[1], out[2], out[3]);
          sts128(Out::chunk(tile, lane, 2 * c + 1), out[4], out[5], out[6], out[7]);
        }
        Out::store(tile, reinterpret_cast<unsigned char*>(a.o + ((size_t)bh * a.N + row0) * D + h), 2 * D, a.N - row0, lane);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) tmem_dealloc<kTmemCols>(tmem);
}

// CTAs with a pair of query tiles, and behind them CTAs with one (see split_tiles).
template <int D, bool HYB, bool SMOOTH, bool POLY>
__global__ void __launch_bounds__(640, 1)
attn4_fwd_2q_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                    const __grid_constant__ CUtensorMap tm_v, const Attn4Args a) {
  const TileOf w = tile_of(a.tiles, a.nb);
  if (w.q0 >= a.nb) return;                 // the missing second tile of a head's last pair
  if (w.two) attn4_2q_body<D, HYB, SMOOTH, POLY, true>(tm_q, tm_k, tm_v, a, w.q0, w.bh);
  else attn4_2q_body<D, HYB, SMOOTH, POLY, false>(tm_q, tm_k, tm_v, a, w.q0, w.bh);
}

template <int D, bool HYB>
cudaError_t run4(const Problem& pr, const QuantLayout& ql, const WorkLayout& wl, const uint8_t* quant,
                 void* o, uint8_t* work, cudaStream_t s) {
  constexpr int KB = D / 64, NVC = HYB ? 1 : 2;
  constexpr size_t kVRow = HYB ? 128 : 64;
  alignas(64) CUtensorMap tq, tk, tv;
  if (!make_map(&tq, quant + ql.q_codes, D / 2, pr.n_pad, pr.BH, D / 2, 128) ||
      !make_map(&tk, quant + ql.k_codes, D / 2, pr.n_pad, pr.BH, D / 2, 128) ||
      !(HYB ? make_map_u4(&tv, quant + ql.v_codes, (uint64_t)pr.n_pad, D, pr.BH, D)
            : make_map(&tv, quant + ql.v_codes, (uint64_t)pr.n_pad / 2, D, pr.BH, 64, D)))
    return cudaErrorUnknown;
  Attn4Args a{};
  a.q_g = (const float*)(quant + ql.q_scale);
  a.k_g = (const float*)(quant + ql.k_scale);
  a.q_micro = quant + ql.q_micro; a.k_micro = quant + ql.k_micro; a.v_micro = quant + ql.v_micro;
  a.v_means = (const __nv_bfloat16*)(quant + ql.v_means);
  a.o = (__nv_bfloat16*)o;
  a.status = (uint32_t*)(work + wl.status);
  a.N = pr.N; a.n_pad = pr.n_pad; a.nb = pr.nb;
  a.sl = pr.softmax_scale * 1.4426950408889634f;
  a.code_off = 120.0f + pr.beta;
  a.wait = {a.status, attn_wait_limit(), attn_wait_nonblocking()};
  constexpr size_t stage = 128 * (D / 2) + (D + 16) * kVRow + ((D * 32 + 1023) / 1024) * 1024 + (((KB + NVC) * 512 + 1023) / 1024) * 1024;
  constexpr size_t smem = 1024 + 2 * 128 * (D / 2) + 2 * 128 * 32 + 2 * 1024 + 2 * 1024 + 1024 + kStages2 * stage + sizeof(FaSmem);
  static_assert(smem <= 227 * 1024, "shared memory of the 4-bit kernel exceeds the SM");
  unsigned grid;
  a.tiles = split_tiles(pr, true, &grid);
  // NVFP4 codes by polynomial from six key tiles on: the loop's longer code has to be fetched and the first tiles, with nothing
  // to overlap, wait for it.  Whole calls, us, without / with: d64 N360 H80 40.3 / 42.3, N576 H48 41.1 / 42.3, N768 H40 36.5 / 35.9,
  // N1024 H37 41.8 / 40.9; d128 N360 H80 54.6 / 55.2, N576 H48 52.9 / 53.5, N768 H40 46.0 / 45.7, N1024 H37 53.1 / 52.7.
  const bool poly = !HYB && pr.nb >= 6;
  cudaError_t e = cudaSuccess;
#define VC_LAUNCH_4(...)                                                                                        \
  ((e = allow_smem<attn4_fwd_2q_kernel<D, HYB, __VA_ARGS__>>()) == cudaSuccess                                  \
       ? (e = launch_overlapped(attn4_fwd_2q_kernel<D, HYB, __VA_ARGS__>, dim3(grid), 640, smem, s, tq, tk, tv, a)) \
       : e)
  if (pr.flags & VC_FLAG_V_SMOOTH) poly ? VC_LAUNCH_4(true, !HYB) : VC_LAUNCH_4(true, false);
  else poly ? VC_LAUNCH_4(false, !HYB) : VC_LAUNCH_4(false, false);
#undef VC_LAUNCH_4
  if (e != cudaSuccess) return e;
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_attn_fwd4(const Problem& pr, const QuantLayout& ql, const WorkLayout& wl,
                             const uint8_t* quant, void* o, uint8_t* work, cudaStream_t stream) {
  if (hybrid4(pr))
    return pr.d == 128 ? run4<128, true>(pr, ql, wl, quant, o, work, stream) : run4<64, true>(pr, ql, wl, quant, o, work, stream);
  return pr.d == 128 ? run4<128, false>(pr, ql, wl, quant, o, work, stream) : run4<64, false>(pr, ql, wl, quant, o, work, stream);
}

}  // namespace vc

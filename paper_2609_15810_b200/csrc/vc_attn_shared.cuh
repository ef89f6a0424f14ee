// Pieces shared by the 8-bit and 4-bit attention kernels: the barrier block of the
// two-query-tile pipeline, bounded waits, the block-mean operand layout, TMA descriptors.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "vc_internal.h"
#include "vc_sm100.cuh"

namespace vc {
namespace attn {

using namespace sm100;

constexpr uint32_t kErrTimeout = kStatusTimeout;

// Where a wait that gives up says so, the polls after which it does, and (test hook) whether these may sleep.
struct WaitArgs {
  uint32_t* status;
  uint32_t limit, nonblocking;
};

// Which query tiles a CTA owns.  CTAs [0, n_pair) take a pair, two CTAs share each pair behind them.
//
// One CTA fits an SM, so the last wave of pairs costs a pair's time however few SMs it uses; a tile alone
// takes 0.77 to 0.85 of that.  When the last wave's pairs are no more than half the SMs, their tiles go
// to CTAs of their own.  (With more pairs than that some SM would have two tiles anyway.)  One head of
// 16384 tokens, 64 pairs or 128 tiles: fp8 160 -> 137 us, d64 142 -> 107, hybrid 165 -> 137, NVFP4
// 268 -> 207; B2 H16 N4096 INT8 scores (3.46 waves) 254 -> 231 us.
struct Tiles {
  int n_pair, qpairs;        // CTAs with a pair of tiles; pairs per head (the last one may lack its second tile)
};

// Arguments of the 8-bit attention kernels.
struct AttnArgs {
  const float *q_scale, *k_scale, *v_scale;
  const __nv_bfloat16* v_means;
  __nv_bfloat16* o;
  uint32_t* status;
  int N, n_pad, nb, p_format;
  Tiles tiles;
  float sl;        // softmax_scale * log2(e)
  float code_off;  // 120 + beta  (Eq. 7)
  WaitArgs wait;
};

constexpr int kStages2 = 4;
constexpr uint32_t kWaitLimit2 = 1u << 18;   // default polls of a wait, x up to 4 us per try: about one second
constexpr uint32_t kDrainLimit = 1u << 22;   // polls of the exit waits for a CTA's own copies and MMAs

inline uint32_t attn_wait_limit() {
  const uint32_t lim = wait_limit_override();
  return lim ? lim : kWaitLimit2;
}
// with the test override a poll never sleeps, so that a tiny limit really is a short wait
inline uint32_t attn_wait_nonblocking() { return wait_limit_override() ? 1u : 0u; }

struct FaSmem {
  uint64_t q_full, kv_full[kStages2], kv_empty[kStages2];
  uint64_t s_full[2], s_free[2], o_done[2], fin_full[2], o_final[2];
  // Hand-offs of alpha (a_full, 128 softmax threads) and of codes and correction (pc_full, 128 softmax and 128
  // correction threads).  Both can run ahead of their consumer and a parity wait aliases after two phases,
  // so they take slots in turn: two per query tile, four when there is one tile.  Why that is enough:
  //   pair of tiles   softmax is at key tile j + 2 only when product j is complete, so every arrival for j is in
  //                   before anyone can make one for j + 2.
  //   one tile        softmax is at j + 2 when product j - 1 is complete, and without block means a correction
  //                   warp whose maxima stand still follows it at once, while another still rescales for j.
  //                   Softmax at j + 4 has seen product j + 1, hence every arrival for j + 1 and for j.
  // (With block means every correction warp waits for product j - 1 at j, and two slots would do.)
  uint64_t a_full[4], pc_full[4];
  uint64_t drain[2];      // exit: "every MMA this issuer warp issued has completed"
  float alpha[4][128];
  alignas(16) float v_scale[2][128];  // s_V, one copy per correction warpgroup
  uint32_t tmem_base;
  volatile int abort;
};

// One thread, in front of the CTA's first barrier.  A stage is given back by the products of every tile.
__device__ __forceinline__ void init_barriers(FaSmem* sh, bool two) {
  mbar_init(&sh->q_full, 1);
  for (int i = 0; i < kStages2; ++i) { mbar_init(&sh->kv_full[i], 1); mbar_init(&sh->kv_empty[i], two ? 2 : 1); }
  for (int i = 0; i < 2; ++i) {
    mbar_init(&sh->s_full[i], 1); mbar_init(&sh->s_free[i], 128); mbar_init(&sh->o_done[i], 1);
    mbar_init(&sh->fin_full[i], 128); mbar_init(&sh->o_final[i], 1);
    for (int b = 0; b < 2; ++b) { mbar_init(&sh->a_full[2 * i + b], 128); mbar_init(&sh->pc_full[2 * i + b], 256); }
  }
  mbar_init(&sh->drain[0], 1); mbar_init(&sh->drain[1], 1);
  sh->abort = 0;
  mbar_fence_init();
}

struct TileOf {
  int bh, q0;
  bool two;
};
__device__ __forceinline__ TileOf tile_of(const Tiles& t, int nb) {
  const int idx = blockIdx.x, behind = idx - t.n_pair;
  const int pair = behind < 0 ? idx : t.n_pair + (behind >> 1);
  TileOf w;
  w.bh = pair / t.qpairs;
  w.q0 = 2 * (pair - w.bh * t.qpairs) + (behind < 0 ? 0 : behind & 1);
  w.two = behind < 0 && w.q0 + 1 < nb;
  return w;
}
inline Tiles split_tiles(const Problem& pr, bool singles, unsigned* grid) {
  Tiles t{};
  t.qpairs = (pr.nb + 1) / 2;
  const int pairs = t.qpairs * pr.BH, sms = sm_count(), last = pairs % sms;
  t.n_pair = singles && 2 * last <= sms ? pairs - last : pairs;
  *grid = (unsigned)(t.n_pair + 2 * (pairs - t.n_pair));
  return t;
}

// Bounded wait of a whole warp.  A key tile's critical chain holds a dozen of these and many find
// their phase complete, so a wait starts with a bare non-blocking test and a vote (about 30 cycles);
// behind it the loop that sleeps in hardware wakes up through one vote as well, and its limits are
// kernel arguments, not loads.  (With the limits read from shared memory in front of the first test
// and the vote behind the loop a completed wait took 170 cycles.  8-bit kernel at B1 H12 N32760 d128:
// 3.52 -> 3.34 ms, at B2 H16 N16384 d64: 2.21 -> 1.94 ms; hybrid 3.40 -> 3.26, NVFP4 5.66 -> 5.28 ms.)
__device__ __forceinline__ bool warp_wait2(uint64_t* bar, uint32_t parity, FaSmem* sh, const WaitArgs& w, uint32_t code) {
  if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return true;
  if (!w.nonblocking) {
#pragma unroll 1
    for (uint32_t i = 0; i < w.limit; ++i) {
      if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
      if ((i & 63u) == 63u && __any_sync(0xffffffffu, sh->abort)) return false;
    }
  } else {
#pragma unroll 1
    for (uint32_t i = 0; i < w.limit; ++i) {
      if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return true;
      if ((i & 63u) == 63u && __any_sync(0xffffffffu, sh->abort)) return false;
    }
  }
  sh->abort = 1;
  atomicExch(w.status, kErrTimeout | code);
  return false;
}

// Exit protocol of the pipelined kernels.  A CTA may leave early (a wait gave up and set `abort`),
// and even then nothing it started may outlive it: shared memory and tensor memory go back to
// the SM when the CTA exits, so a bulk copy still landing or an MMA still reading would touch
// memory that belongs to somebody else by then.
//   producer warp   waits (bounded, generous) for every copy it issued and nobody consumed
//   issuer warps    commit to their own barrier and wait for it: all their MMAs have completed
// tcgen05.ld / tcgen05.st of the other warps are complete at their wait::ld / wait::st.  Only
// then does the CTA reach the barrier in front of the tensor-memory release.
__device__ __forceinline__ void drain_loads(FaSmem* sh, int issued) {
  mbar_wait(&sh->q_full, 0, kDrainLimit);
  for (int jj = issued > kStages2 ? issued - kStages2 : 0; jj < issued; ++jj)
    mbar_wait(&sh->kv_full[jj % kStages2], (jj / kStages2) & 1, kDrainLimit);
}
__device__ __forceinline__ void drain_mmas(FaSmem* sh, int which) {
  if (elect_one()) mma_commit(&sh->drain[which]);
  __syncwarp();
  mbar_wait(&sh->drain[which], 0, kDrainLimit);
}

// Block means as the B operand of the per-tile mean-restoration MMA: a [d][8] fp32 tile with entry
// [c][0] = [c][1] = mu~[c] (for r_hi and r_lo) and zeros elsewhere, in 32-byte rows whose two 16-byte
// chunks swap when (row / 4) is odd.  The producer warp writes the two live words of every row into
// the key tile's stage, next to the copies it issues; the zeros are written once per CTA.  (As a
// tensor in global memory, expanded by a launch of its own and fetched by TMA, the same operand was
// 32 bytes per mean: 42 MB written and 4 of the 37 KB a key tile moves into shared memory at B1 H40
// N32760 d128.)
template <int D>
struct MeanRows {
  uint16_t v[D / 32];
  // bf16 bits of the means of channels lane, lane + 32, ...
  __device__ __forceinline__ void fetch(const __nv_bfloat16* means, int lane) {
#pragma unroll
    for (int i = 0; i < D / 32; ++i) v[i] = __ldg(reinterpret_cast<const unsigned short*>(means) + lane + 32 * i);
  }
  __device__ __forceinline__ void store(unsigned char* tile, int lane) const {
#pragma unroll
    for (int i = 0; i < D / 32; ++i) {
      const int row = lane + 32 * i;
      *reinterpret_cast<uint2*>(tile + row * 32 + 16 * ((row >> 2) & 1)) = make_uint2((uint32_t)v[i] << 16, (uint32_t)v[i] << 16);
    }
  }
};

// Output rows leave through shared memory.  A thread of the epilogue holds one row, and storing it from there puts the
// lanes of a warp on 32 lines at a time.  So a warp writes its 32 rows, W columns at a time, into a tile of its own
// (16-byte chunk c at position c ^ swizzle: no bank conflicts) and stores it in whole lines: B2 H16 N4096 d128 INT8 scores
// 267.3 -> 263.1 us, B1 H16 N4096 FP8 126.8 -> 124.9.  (The epilogue by the softmax warps, 64 columns at a time, is 0.2 us
// shorter, but what it keeps alive across their loop costs more: the same calls 267 and 131 us.)
// The tile lies in stage (nb + t) % kStages2 of the ring: it held key tile nb - 4 + t, and what may still be read when tile t's
// last product is complete are the last key tile and the block mean of the one before it.
template <int W> struct OutTile {
  static constexpr int CPR = W / 8, ROW = 2 * W;           // chunks and bytes per row
  static __device__ __forceinline__ int swizzle(int row) { return CPR >= 8 ? row & 7 : (row >> 1) & (CPR - 1); }
  static __device__ __forceinline__ uint32_t chunk(uint32_t tile, int row, int c) { return tile + row * ROW + ((c ^ swizzle(row)) << 4); }
  // rows [0, rows) of the warp's 32 -> dst, `pitch` bytes apart
  static __device__ __forceinline__ void store(uint32_t tile, unsigned char* dst, int pitch, int rows, int lane) {
    __syncwarp();
#pragma unroll 4
    for (int k = 0; k < CPR; ++k) {
      const int row = (k * 32 + lane) / CPR, c = lane % CPR;
      if (row < rows) {
        const float4 v = lds128(chunk(tile, row, c));
        *reinterpret_cast<float4*>(dst + (size_t)row * pitch + 16 * c) = v;
      }
    }
    __syncwarp();
  }
};

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;   // resolved once; the driver entry point never changes
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// 3-D byte tensor [dim2][dim1][dim0], box {box0, box1, 1}, swizzle chosen by the box width.
inline bool make_map(CUtensorMap* m, const void* base, uint64_t dim0, uint64_t dim1, uint64_t dim2, uint32_t box0, uint32_t box1) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {dim0, dim1, dim2};
  const cuuint64_t strides[2] = {dim0, dim0 * dim1};
  const cuuint32_t box[3] = {box0, box1, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUtensorMapSwizzle sw = box0 == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (box0 == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}


// 3-D tensor of packed 4-bit elements [dim2][dim1][dim0 elements]; a box of 128 elements x box1
// rows lands in shared memory as 128-byte rows of 16-byte containers (16 elements in the low 8
// bytes, 128-byte swizzle): the layout kind::mxf8f6f4 reads 4-bit operands in.  The copy reports
// the packed bytes (64 per row) to its mbarrier.  `base` must be 32-byte aligned, dim0 a
// multiple of 128.
inline bool make_map_u4(CUtensorMap* m, const void* base, uint64_t dim0, uint64_t dim1, uint64_t dim2, uint32_t box1) {
  EncodeTiledFn fn = encode_fn();
  if (!fn || ((uintptr_t)base & 31) || (dim0 & 127)) return false;
  const cuuint64_t dims[3] = {dim0, dim1, dim2};
  const cuuint64_t strides[2] = {dim0 / 2, dim0 / 2 * dim1};
  const cuuint32_t box[3] = {128, box1, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_16U4_ALIGN16B, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Arguments and operand maps of the 8-bit kernels.
template <int D>
inline bool fill_args8(const Problem& pr, const QuantLayout& ql, const WorkLayout& wl, const uint8_t* quant, void* o, uint8_t* work,
                       AttnArgs* a, CUtensorMap* tq, CUtensorMap* tk, CUtensorMap* tv) {
  if (!make_map(tq, quant + ql.q_codes, D, pr.n_pad, pr.BH, D, 128) ||
      !make_map(tk, quant + ql.k_codes, D, pr.n_pad, pr.BH, D, 128) ||
      !make_map(tv, quant + ql.v_codes, pr.n_pad, D, pr.BH, 128, D))
    return false;
  a->q_scale = (const float*)(quant + ql.q_scale);
  a->k_scale = (const float*)(quant + ql.k_scale);
  a->v_scale = (const float*)(quant + ql.v_scale);
  a->v_means = (const __nv_bfloat16*)(quant + ql.v_means);
  a->o = (__nv_bfloat16*)o;
  a->status = (uint32_t*)(work + wl.status);
  a->N = pr.N; a->n_pad = pr.n_pad; a->nb = pr.nb; a->p_format = pr.p_format;
  a->sl = pr.softmax_scale * 1.4426950408889634f;
  a->code_off = 120.0f + pr.beta;
  a->wait = {a->status, attn_wait_limit(), attn_wait_nonblocking()};
  return true;
}

}  // namespace attn
}  // namespace vc

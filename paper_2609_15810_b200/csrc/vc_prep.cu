// Fused preprocessing pass of VC-Attention for sm_100a (Sec. 3.4 "Fused preprocessing",
// App. B): every operand is read as bf16 with 16-byte vector loads and leaves as low-bit
// codes plus scales; no rotated / permuted / centered high-precision tensor reaches HBM.
//
//   Q : RoPE -> Hadamard (in registers, a row in two threads) -> per-128-row scale -> codes
//   K : RoPE -> column sums (stats launch) ... gather by pi -> RoPE at the source position
//       -> subtract channel mean -> Hadamard -> scale -> codes
//   V : gather by pi -> block mean (Eq. 4) and residual amax (stats launch) ...
//       gather -> residual -> codes written channel-major, block means beside them
//
// The two global reductions (K channel mean over all tokens, per-channel amax of the V
// residual over all tokens) force statistics launches before the quantizing launches; heads
// can be processed in groups so that the second read of K and V may hit L2.  All passes are
// persistent kernels that prefetch the next row blocks with cp.async while they transform
// the current one.
#include <algorithm>
#include <climits>

#include "vc_launch.h"
#include "vc_prep_common.cuh"

namespace vc {
namespace {

// ---------------------------------------------------------------------------------------
// RoPE tables: per axis a, entry [pos][i] = (cos, sin)(pos * theta^(-2 i / d_a)), evaluated
// in double and rounded once to fp32.
// The same launch clears the words that must start at zero (the status word, the maxima) and, when
// the caller supplies the statistics, turns them into the K mean and the value scales of the bundle.
struct SetUp {
  unsigned int *status, *zero;
  int n_zero;                       // words behind `zero`
  int n_ext;                        // B H d with supplied statistics, else 0
  const float *ext_k_mean, *ext_v_amax;   // ext_k_mean: null = a mean of zero (K smoothing off)
  float *k_mean, *v_scale;
};
__device__ __forceinline__ float value_scale(float amax) { return amax > 0.f ? amax / 448.0f : 1.0f; }
__device__ __forceinline__ float outer_scale(float amax) { return amax > 0.f ? amax / 2688.0f : 1.0f; }     // NVFP4, per head

// Frequency of pair i of an axis with `pairs` channel pairs, and the entry of a position: (cos, sin) and, in `folded`, the
// rotation folded into the first Hadamard level, u = x0 (c + s) + x1 (c - s), v = x0 (c - s) - x1 (c + s), each
// coefficient rounded once.
__device__ __forceinline__ double rope_freq(double theta, int i, int pairs) { return pow(theta, -2.0 * (double)i / (double)(2 * pairs)); }
__device__ __forceinline__ void rope_entry_of(int pos, double freq, float2* plain, float2* folded) {
  double c, sn;
  sincos((double)pos * freq, &sn, &c);
  *plain = make_float2((float)c, (float)sn);
  *folded = make_float2((float)(c + sn), (float)(c - sn));
}

__global__ void rope_table_kernel(float2* tab, RopeDesc rd, double theta, const SetUp u) {
  // (The wait stands in front of the arithmetic: entries computed beside the end of the attention before them make calls
  // of 2000 to 4000 tokens 1 to 3 percent slower.)
  pdl_wait();
  pdl_allow();
  const int e = blockIdx.x * blockDim.x + threadIdx.x, all = gridDim.x * blockDim.x;
  if (e == 0) *u.status = 0u;
  for (int i = e; i < u.n_zero; i += all) u.zero[i] = 0u;
  for (int i = e; i < u.n_ext; i += all) {
    u.k_mean[i] = u.ext_k_mean ? u.ext_k_mean[i] : 0.f;
    u.v_scale[i] = value_scale(u.ext_v_amax[i]);
  }
  if (e >= rd.entries) return;
  const int a = e >= rd.off[2] ? 2 : (e >= rd.off[1] ? 1 : 0), r = e - rd.off[a], pos = r / rd.pairs[a], i = r - pos * rd.pairs[a];
  float2 plain, folded;
  rope_entry_of(pos, rope_freq(theta, i, rd.pairs[a]), &plain, &folded);
  tab[e] = plain;
  tab[rd.entries + e] = folded;
}

// ---------------------------------------------------------------------------------------
// Persistent, pipelined passes.  Every pass is a loop over work items (tensor, head, block of
// 128 rows); a CTA takes items blockIdx.x, blockIdx.x + gridDim.x, ...  The 16-byte chunks of
// the NEXT items are already on their way into a ring of shared-memory stages (cp.async, no
// registers held for bytes in flight) while the current item is transformed, so the load
// latency of a block hides behind the arithmetic of the blocks before it.  In the K column sums
// a thread fetches exactly the chunks it will read itself and in the Q/K pass a warp fetches
// exactly the rows it will transform, so those passes need no CTA-wide barrier for the data;
// V is staged as a tile because its codes leave channel-major.
// (One bulk-async copy per gathered row was tried instead of cp.async: 128 small copies per
// block kept the copy engine, not HBM, busy.)
constexpr int kThreads = 256;      // threads of the column-sum and V passes
constexpr int kRowThreads = 128;   // rows of a Q/K item (threads of the pass = rows x threads per row)
constexpr int kTpr = 2;            // threads per Q/K row

template <int D> struct Geo {
  static constexpr int pitch = 2 * D + 16;          // row pitch of the thread-per-row layout
  static constexpr int stage_bytes = kBlock * pitch;
};

// Items are numbered block-fastest, then head, then tensor.  The CTA with number `rank` of a pass visits
// items rank + k * stride: the position is divided out once and then advanced by the grid stride with carries
// (the divisions are not free at 64 elements per thread and item).
struct Cursor {
  int blk, hh, z;            // block, head within the launch's group, tensor
};
struct CursorStep {
  int dblk, dhh;             // stride = dhh * nb + dblk
};
__device__ __forceinline__ Cursor cursor_at(int item, int nb, int nh) {
  Cursor c;
  c.blk = item % nb;
  const int r = item / nb;
  c.hh = r % nh;
  c.z = r / nh;
  return c;
}
__device__ __forceinline__ CursorStep cursor_step(int stride, int nb) {
  CursorStep s;
  s.dhh = stride / nb;
  s.dblk = stride - s.dhh * nb;
  return s;
}
__device__ __forceinline__ void advance(Cursor& c, const CursorStep& s, int nb, int nh) {
  c.blk += s.dblk;
  c.hh += s.dhh;
  if (c.blk >= nb) { c.blk -= nb; ++c.hh; }
  while (c.hh >= nh) { c.hh -= nh; ++c.z; }      // at most once unless the launch is tiny
}
// Start of head bh in an input tensor, in bytes (bh = b * H + h, general strides).
__device__ __forceinline__ int64_t head_offset_bytes(const PrepArgs& a, int bh) {
  const int b = (int)div40((unsigned)bh, a.mul_H), h = bh - b * a.H;
  return 2 * (b * a.stride_b + h * a.stride_h);
}

// ---------------------------------------------------------------------------------------
// K column sums after RoPE (the channel mean of Sec. 3.4 is taken after the rotation).  A lane
// owns 8 consecutive channels of D/16 rows, so a column's partial sums meet by xor-shuffles.
// A RoPE table entry: from the copy in shared memory (address in the shared window) when there
// is one, else from global memory.
struct RopeTab {
  uint32_t saddr;            // 0: no copy in shared memory
  const float2* g;
};
__device__ __forceinline__ float2 rope_entry_s(uint32_t saddr, int e) {
  float2 r;
  asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "r"(saddr + 8u * (uint32_t)e));
  return r;
}
__device__ __forceinline__ float2 rope_entry(const RopeTab& t, int e) {
  return t.saddr ? rope_entry_s(t.saddr, e) : __ldg(t.g + e);
}

struct PairSlots {          // the 4 channel pairs a lane owns: axis and table slot of each
  int axis[4], idx[4], stride[4];
};
__device__ __forceinline__ PairSlots pair_slots(const RopeDesc& rd, int first_pair) {
  PairSlots ps;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int p = first_pair + j;
    const int ax = p >= rd.pair_start[2] ? 2 : (p >= rd.pair_start[1] ? 1 : 0);
    ps.axis[j] = ax;
    ps.idx[j] = rd.off[ax] + (p - rd.pair_start[ax]);
    ps.stride[j] = rd.pairs[ax];
  }
  return ps;
}

template <int D>
__device__ __forceinline__ void k_colsum_item(const PrepArgs& a, const unsigned char* mine /*this thread's chunk of its first row*/,
                                              int step /*bytes to its next row's*/, float* red, const RopeTab& tab, const PairSlots& ps,
                                              float* out /*[D]*/, int blk) {
  constexpr int LPR = D / 8;         // lanes per row
  constexpr int RPL = LPR / 2;       // rows per lane (a warp covers 16 rows)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lr = lane % LPR, hb = lane / LPR;
  const bool do_rope = a.flags & VC_FLAG_ROPE;
  // grid position of the lane's first row; the following rows advance x with carry
  int tt, ty, tx;
  grid_pos(a.rd, blk * kBlock + 16 * warp + RPL * hb, tt, ty, tx);
  float s[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) s[c] = 0.f;
  const int t0 = blk * kBlock + 16 * warp + RPL * hb;
  const int n_rows = min(RPL, a.N - t0);           // rows of a lane ascend: the rest is padding
  if (do_rope && tab.saddr) {
    // The rotation is accumulated directly (four FMAs per channel pair and row).  The lane's four
    // table addresses follow its rows: x advances by one per row, so the entries of the pairs on
    // the x axis move by one table row and the others stay; a row that wraps x recomputes them.
    // The coefficients of the pairs on the t and y axes are the same for all of a lane's rows
    // unless x wraps, so they stay in registers; only lanes whose pairs lie on the x axis reload
    // per row (a predicated load: the other lanes take no shared-memory bandwidth).
    uint32_t ad[4], inc[4];
    float cc[4], ss[4];
    auto locate = [&]() {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int pos = ps.axis[j] == 0 ? tt : (ps.axis[j] == 1 ? ty : tx);
        ad[j] = tab.saddr + 8u * (uint32_t)(ps.idx[j] + pos * ps.stride[j]);
        asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(cc[j]), "=f"(ss[j]) : "r"(ad[j]));
      }
    };
#pragma unroll
    for (int j = 0; j < 4; ++j) inc[j] = ps.axis[j] == 2 ? 8u * (uint32_t)ps.stride[j] : 0u;
    locate();
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      if (i >= n_rows) break;
      const uint4 raw = *reinterpret_cast<const uint4*>(mine + i * step);
      const unsigned int w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float x0 = __uint_as_float(w[j] << 16), x1 = __uint_as_float(w[j] & 0xffff0000u);
        s[2 * j] = fmaf(-x1, ss[j], fmaf(x0, cc[j], s[2 * j]));
        s[2 * j + 1] = fmaf(x1, cc[j], fmaf(x0, ss[j], s[2 * j + 1]));
      }
      if (i + 1 < RPL) {
        if (++tx == a.rd.grid_w) {
          tx = 0;
          if (++ty == a.rd.grid_h) { ty = 0; ++tt; }
          locate();
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (inc[j]) {
              ad[j] += inc[j];
              asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(cc[j]), "=f"(ss[j]) : "r"(ad[j]));
            }
          }
        }
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      if (i >= n_rows) break;
      const uint4 raw = *reinterpret_cast<const uint4*>(mine + i * step);
      const unsigned int w[4] = {raw.x, raw.y, raw.z, raw.w};
      float x[8];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        x[2 * j] = __uint_as_float(w[j] << 16);
        x[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
      }
      if (do_rope) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int pos = ps.axis[j] == 0 ? tt : (ps.axis[j] == 1 ? ty : tx);
          const float2 cs = rope_entry(tab, ps.idx[j] + pos * ps.stride[j]);
          const float x0 = x[2 * j], x1 = x[2 * j + 1];
          x[2 * j] = x0 * cs.x - x1 * cs.y;
          x[2 * j + 1] = x0 * cs.y + x1 * cs.x;
        }
        if (++tx == a.rd.grid_w) { tx = 0; if (++ty == a.rd.grid_h) { ty = 0; ++tt; } }
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) s[c] += x[c];
    }
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) {
#pragma unroll
    for (int m = LPR; m < 32; m <<= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], m);
  }
  __syncthreads();                           // the previous item's reads of `red` are done
  if (hb == 0) {
#pragma unroll
    for (int c = 0; c < 8; ++c) red[warp * D + 8 * lr + c] = s[c];
  }
  __syncthreads();
  if (tid < D) {
    float t = 0.f;
#pragma unroll
    for (int w8 = 0; w8 < 8; ++w8) t += red[w8 * D + tid];
    out[tid] = t;
  }
}

// ---------------------------------------------------------------------------------------
// Q / K, one row per thread.  All D channels of a row sit in the registers of one thread, so
// the Hadamard rotation is D/2 * log2 D register butterflies with no shuffle, RoPE pairs and
// NVFP4 groups are thread-local, and a row's codes leave as 16-byte stores.
enum { kStageAmax = 1, kStageQuant8 = 2, kStageQuant4 = 3, kStageQuant8I = 4 };   // 8I: INT8 codes (VC_FLAG_INT8_QK)

template <int D> struct RopeSplit;          // pair boundaries of the default channel split
template <> struct RopeSplit<128> { static constexpr int p1 = 22, p2 = 43; };   // 44 / 42 / 42
template <> struct RopeSplit<64> { static constexpr int p1 = 12, p2 = 22; };    // 24 / 20 / 20

// Reads the thread's row out of the stage, releases the stage, then transforms the row.
// `red` is [2][8] floats and `kmean_s` [D] floats of compute-warp scratch.
// Q and K run through one copy of the row body (TENSOR is a run-time argument): the unrolled body
// is tens of KB of code, and two copies of it thrash the instruction cache.
//
// Two threads per row (kTpr): the lanes 0..15 of a warp hold channels [0, D/2) of 16 rows and the
// lanes 16..31 channels [D/2, D) of the same rows; the last Hadamard level crosses the two halves with
// one shuffle per value.  RoPE pairs and NVFP4 groups stay thread-local.  (Measured against it: one
// thread per row needs twice the registers, so half the warps per SM; four threads per row add a second
// shuffle level to the shared-memory pipe, B1 H40 N32760 0.70 instead of 0.60 ms.)
__device__ __forceinline__ int qk_row_of(int tid) { return 16 * (tid >> 5) + (tid & 15); }
__device__ __forceinline__ int qk_part_of(int tid) { return (tid >> 4) & 1; }

template <int D> __device__ __forceinline__ constexpr int rope_axis_of(int p) {
  return p < RopeSplit<D>::p1 ? 0 : (p < RopeSplit<D>::p2 ? 1 : 2);
}

template <int D, int STAGE, typename AmaxAt, typename Outer>
__device__ __forceinline__ void qk_row_item(const PrepArgs& a, const int TENSOR /*0 = Q, 1 = K*/, const unsigned char* stage,
                                            unsigned char* out_tile, float* red, float* kmean_s, const RopeTab& tab, int bh,
                                            int blk, int iter, bool new_head, int src_row, AmaxAt amax_at, Outer outer) {
  constexpr int C = D / kTpr;                      // channels per thread
  constexpr int NT = kRowThreads * kTpr;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row = qk_row_of(tid), part = qk_part_of(tid);
  const bool do_rope = a.flags & VC_FLAG_ROPE;
  const bool do_had = a.flags & VC_FLAG_HADAMARD;
  const bool center = TENSOR == 1 && (a.flags & VC_FLAG_K_SMOOTH);
  const bool valid = src_row >= 0;               // src_row: the input row behind this thread's row
  const int src = valid ? src_row : 0;           // (RoPE acts at the source position)
  // (a row without a source reads what the stage holds and is zeroed below)
  uint4 raw[C / 8];
#pragma unroll
  for (int i = 0; i < C / 8; ++i) raw[i] = *reinterpret_cast<const uint4*>(stage + row * Geo<D>::pitch + part * (2 * C) + 16 * i);
  if (center && new_head) {
    __syncthreads();                               // everyone is done with the previous head's mean
    for (int c = tid; c < D; c += NT) kmean_s[c] = a.k_mean[(size_t)bh * D + c];
    __syncthreads();
  }

  float x[C];
#pragma unroll
  for (int i = 0; i < C / 8; ++i) {
    const unsigned int w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[8 * i + 2 * j] = __uint_as_float(w[j] << 16);
      x[8 * i + 2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
    }
  }
  if (!valid) {
#pragma unroll
    for (int c = 0; c < C; ++c) x[c] = 0.f;
  }
  if (do_rope && valid) {
    int tt, ty, tx;
    grid_pos(a.rd, src, tt, ty, tx);
    // entry of pair p of axis ax: off[ax] + pos[ax] * pairs[ax] + (p - pair_start[ax])
    const int e[3] = {a.rd.off[0] + tt * a.rd.pairs[0] - a.rd.pair_start[0],
                      a.rd.off[1] + ty * a.rd.pairs[1] - a.rd.pair_start[1],
                      a.rd.off[2] + tx * a.rd.pairs[2] - a.rd.pair_start[2]};
    const int p0 = part * (C / 2);               // first pair of this thread
    if (a.rope_default && tab.saddr) {
      // compile-time pair boundaries: the axis of local pair i is known for either part, so the
      // table base of each (axis in part 0, axis in part 1) combination is selected once per row
      int base[3][3];
#pragma unroll
      for (int a0 = 0; a0 < 3; ++a0)
#pragma unroll
        for (int a1 = 0; a1 < 3; ++a1) base[a0][a1] = (part ? e[a1] : e[a0]) + p0;
#pragma unroll
      for (int i = 0; i < C / 2; ++i) {
        const float2 cs = rope_entry_s(tab.saddr, base[rope_axis_of<D>(i)][rope_axis_of<D>(C / 2 + i)] + i);
        const float x0 = x[2 * i], x1 = x[2 * i + 1];
        x[2 * i] = x0 * cs.x - x1 * cs.y;
        x[2 * i + 1] = x0 * cs.y + x1 * cs.x;
      }
    } else {
#pragma unroll
      for (int i = 0; i < C / 2; ++i) {
        const int p = p0 + i;
        const int eb = p < a.rd.pair_start[1] ? e[0] : (p < a.rd.pair_start[2] ? e[1] : e[2]);
        const float2 cs = rope_entry(tab, eb + p);
        const float x0 = x[2 * i], x1 = x[2 * i + 1];
        x[2 * i] = x0 * cs.x - x1 * cs.y;
        x[2 * i + 1] = x0 * cs.y + x1 * cs.x;
      }
    }
  }
  if (center && valid) {
    const float4* km = reinterpret_cast<const float4*>(kmean_s + part * C);
#pragma unroll
    for (int c4 = 0; c4 < C / 4; ++c4) {
      const float4 m = km[c4];
      x[4 * c4] -= m.x; x[4 * c4 + 1] -= m.y; x[4 * c4 + 2] -= m.z; x[4 * c4 + 3] -= m.w;
    }
  }
  if (do_had) {
#pragma unroll
    for (int sft = 1; sft < C; sft <<= 1) {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if (!(c & sft)) {
          const float u = x[c], v = x[c | sft];
          x[c] = u + v;
          x[c | sft] = u - v;
        }
      }
    }
    // the level that pairs channel c with c + D/2: the lower half takes mine + theirs, the upper
    // half theirs - mine (one fused multiply-add with +-1, exact)
    const float sgn = part ? -1.0f : 1.0f;
#pragma unroll
    for (int c = 0; c < C; ++c) x[c] = fmaf(x[c], sgn, __shfl_xor_sync(0xffffffffu, x[c], 16));
  }
  const float rs = do_had ? (D == 128 ? 0.08838834764831845f : 0.125f) : 1.0f;   // 1/sqrt(D)

  float amax = 0.f;
  if constexpr (STAGE != kStageQuant4) {
    float m0 = 0.f, m1 = 0.f;
#pragma unroll
    for (int c = 0; c < C; c += 4) {
      m0 = max3(m0, fabsf(x[c]), fabsf(x[c + 1]));
      m1 = max3(m1, fabsf(x[c + 2]), fabsf(x[c + 3]));
    }
    amax = warp_max(fmaxf(m0, m1) * rs);        // max and the (positive) scale commute exactly
    float* rbuf = red + 8 * (iter & 1);         // alternate buffers: one barrier per item suffices
    if (lane == 0) rbuf[warp] = amax;
    __syncthreads();
    amax = fmaxf(fmaxf(rbuf[0], rbuf[1]), fmaxf(rbuf[2], rbuf[3]));
    amax = fmaxf(amax, fmaxf(fmaxf(rbuf[4], rbuf[5]), fmaxf(rbuf[6], rbuf[7])));
  }
  if constexpr (STAGE == kStageAmax) {
    if (tid == 0) atomicMax(amax_at(), __float_as_uint(amax));
    return;
  }
  const size_t row_g = (size_t)bh * a.n_pad + (size_t)blk * kBlock + row;

  if constexpr (STAGE == kStageQuant8 || STAGE == kStageQuant8I) {
    // E4M3 codes (top value 448), or INT8 codes (top value 127; the INT8 Q K^T of Fig. 3)
    constexpr bool int8 = STAGE == kStageQuant8I;
    const float top = int8 ? 127.0f : 448.0f;
    const float inv = amax > 0.f ? top / amax : 0.f;
    if (tid == 0) (TENSOR == 0 ? a.q_scale : a.k_scale)[(size_t)bh * a.nb + blk] = amax > 0.f ? amax / top : 1.0f;
    // codes go to the swizzled output tile; the CTA copies it out with coalesced stores
    constexpr int CPR = D / 16;
    uint4* dst = reinterpret_cast<uint4*>(out_tile + row * D);
    const int sw = (row / (8 / CPR)) & (CPR - 1);
#pragma unroll
    for (int i = 0; i < C / 16; ++i) {
      unsigned int w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 16 * i + 4 * j;
        if constexpr (int8) {
          // |y| <= 127: adding 1.5 * 2^23 rounds y to the nearest even integer into the low mantissa
          // bits, two's complement for negative values; the low bytes are the codes
          const unsigned int r0 = __float_as_uint(((x[c] * rs) * inv) + 12582912.0f), r1 = __float_as_uint(((x[c + 1] * rs) * inv) + 12582912.0f);
          const unsigned int r2 = __float_as_uint(((x[c + 2] * rs) * inv) + 12582912.0f), r3 = __float_as_uint(((x[c + 3] * rs) * inv) + 12582912.0f);
          w[j] = __byte_perm(__byte_perm(r0, r1, 0x0040), __byte_perm(r2, r3, 0x0040), 0x5410);
        } else {
          const unsigned int lo = __nv_cvt_float2_to_fp8x2(make_float2((x[c] * rs) * inv, (x[c + 1] * rs) * inv), __NV_SATFINITE, __NV_E4M3);
          const unsigned int hi = __nv_cvt_float2_to_fp8x2(make_float2((x[c + 2] * rs) * inv, (x[c + 3] * rs) * inv), __NV_SATFINITE, __NV_E4M3);
          w[j] = lo | (hi << 16);
        }
      }
      dst[(part * (C / 16) + i) ^ sw] = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }

  if constexpr (STAGE == kStageQuant4) {
    // NVFP4: outer scale g per (b, h), microscale per token per 16 channels
    const float g = outer();
    const float inv6 = 1.0f / (6.0f * g);
    constexpr int MB = C / 16;                   // microscale bytes of this thread
    unsigned int codes[C / 8], micro[(MB + 3) / 4];
#pragma unroll
    for (int i = 0; i < (MB + 3) / 4; ++i) micro[i] = 0;
#pragma unroll
    for (int gq = 0; gq < C / 16; ++gq) {
      float m = 0.f;
#pragma unroll
      for (int c = 0; c < 16; ++c) { x[16 * gq + c] *= rs; m = fmaxf(m, fabsf(x[16 * gq + c])); }
      const unsigned int sb = __nv_cvt_float_to_fp8(m * inv6, __NV_SATFINITE, __NV_E4M3);
      const float sdec = e4m3_to_float(sb);
      const float rcp = sdec > 0.f ? 1.0f / (g * sdec) : 0.f;
      micro[gq / 4] |= sb << (8 * (gq & 3));
#pragma unroll
      for (int wi = 0; wi < 2; ++wi) {
        unsigned int word = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int c = 16 * gq + 8 * wi + 2 * j;
          const unsigned int two = __nv_cvt_float2_to_fp4x2(make_float2(x[c] * rcp, x[c + 1] * rcp), __NV_E2M1, cudaRoundNearest);
          word |= (two & 0xffu) << (8 * j);
        }
        codes[2 * gq + wi] = sdec > 0.f ? word : 0u;
      }
    }
    constexpr int CPR = D / 32;
    uint4* dst = reinterpret_cast<uint4*>(out_tile + row * (D / 2));
    const int sw = (row / (8 / CPR)) & (CPR - 1);
#pragma unroll
    for (int i = 0; i < C / 32; ++i) dst[(part * (C / 32) + i) ^ sw] = make_uint4(codes[4 * i], codes[4 * i + 1], codes[4 * i + 2], codes[4 * i + 3]);
    uint8_t* mrow = (TENSOR == 0 ? a.q_micro : a.k_micro) + row_g * (D / 16) + part * MB;
    if constexpr (MB % 4 == 0) {
#pragma unroll
      for (int i = 0; i < MB / 4; ++i) reinterpret_cast<unsigned int*>(mrow)[i] = micro[i];
    } else {
      static_assert(MB == 2, "microscale bytes per thread");
      *reinterpret_cast<unsigned short*>(mrow) = (unsigned short)micro[0];
    }
  }
}

// ---------------------------------------------------------------------------------------
// The same row transform with fewer instructions, for the standard configuration (RoPE with the
// default channel split and the table in shared memory, Hadamard on; K smoothing either way):
//  * rotation, centering and the first Hadamard level are one step per channel pair: with
//    (A, B) = (c + s, c - s) from the folded table and (m+, m-) = (m0 + m1, m0 - m1) of the mean,
//    u = x0 A + x1 B - m+  and  v = x0 B - x1 A - m-  are the level-1 outputs (4 FMAs per pair);
//  * a pair lives in one 64-bit register and the other levels, the cross-lane level and the scale
//    multiply are packed two-lane FP32 instructions (add / sub / fma / mul .f32x2: the same FP32
//    operation per lane, one instruction issued for two);
//  * at 8 bits 1 / sqrt(D) and the quantization scale are one factor.
// The 4-bit head-maximum and NVFP4 stages run on the same transform.
// `kmean_pm` holds (m+, m-) per pair, zeros while Q rows or unsmoothed K rows are processed.  `amax_at()`: where the head
// maximum is collected; `outer()`: the head's NVFP4 outer scale.  (Functions, and not values: a pointer that lives through the item
// costs the general row body spills, B1 H24 N118800 d128 without RoPE 1429 -> 1500 us.)
template <int D, int STAGE, typename AmaxAt, typename Outer>
__device__ __forceinline__ void qk_row_item_fast(const PrepArgs& a, const int TENSOR, const unsigned char* stage,
                                                 unsigned char* out_tile, float* red, float* kmean_pm, uint32_t tab_saddr,
                                                 int bh, int blk, int iter, bool new_head, int src_row, AmaxAt amax_at, Outer outer) {
  constexpr int C = D / kTpr, P = C / 2;           // channels and pairs per thread
  constexpr int NT = kRowThreads * kTpr;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row = qk_row_of(tid), part = qk_part_of(tid);
  const bool valid = src_row >= 0;
  const int src = valid ? src_row : 0;
  uint4 raw[C / 8];
#pragma unroll
  for (int i = 0; i < C / 8; ++i) raw[i] = *reinterpret_cast<const uint4*>(stage + row * Geo<D>::pitch + part * (2 * C) + 16 * i);
  if (TENSOR == 1 && (a.flags & VC_FLAG_K_SMOOTH) && new_head) {
    __syncthreads();                               // everyone is done with the previous head's mean
    for (int pr = tid; pr < D / 2; pr += NT) {
      const float2 m = *reinterpret_cast<const float2*>(a.k_mean + (size_t)bh * D + 2 * pr);
      *reinterpret_cast<float2*>(kmean_pm + 2 * pr) = make_float2(m.x + m.y, m.x - m.y);
    }
    __syncthreads();
  }
  int tt, ty, tx;
  grid_pos(a.rd, src, tt, ty, tx);
  const int e[3] = {a.rd.off[0] + tt * a.rd.pairs[0] - a.rd.pair_start[0],
                    a.rd.off[1] + ty * a.rd.pairs[1] - a.rd.pair_start[1],
                    a.rd.off[2] + tx * a.rd.pairs[2] - a.rd.pair_start[2]};
  const int p0 = part * P;
  // byte address of pair i's entry = base of its axis + 8 i (the axis of local pair i is known at
  // compile time for either part: one base per combination, selected once per row)
  // (written as a selection per pair; identical selections fold into one value per combination)
  auto base_of = [&](int i) -> uint32_t {          // i is a compile-time constant after unrolling
    const int ee = part ? e[rope_axis_of<D>(P + i)] : e[rope_axis_of<D>(i)];
    return tab_saddr + 8u * (uint32_t)(ee + p0);
  };
  const float4* km = reinterpret_cast<const float4*>(kmean_pm + part * C);

  uint64_t X[P];
#pragma unroll
  for (int i = 0; i < P; i += 2) {
    const float4 m = km[i / 2];                    // (m+, m-) of pairs i and i + 1
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int ii = i + k;
      const unsigned int w = ii % 4 == 0 ? raw[ii / 4].x : (ii % 4 == 1 ? raw[ii / 4].y : (ii % 4 == 2 ? raw[ii / 4].z : raw[ii / 4].w));
      const float x0 = __uint_as_float(w << 16), x1 = __uint_as_float(w & 0xffff0000u);
      float A, B;
      asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(A), "=f"(B)
          : "r"(base_of(ii) + 8u * ii));
      const float mp = k == 0 ? m.x : m.z, mm = k == 0 ? m.y : m.w;
      const float u = fmaf(x0, A, fmaf(x1, B, -mp));
      const float v = fmaf(x0, B, fmaf(-x1, A, -mm));
      X[ii] = pack_f32x2(u, v);
    }
  }
  if (!valid) {                                    // a padding row: zeros (codes 0, no part in the maximum)
#pragma unroll
    for (int i = 0; i < P; ++i) X[i] = 0ull;
  }
  // Hadamard levels 2 .. C/2 on whole pairs
#pragma unroll
  for (int h = 1; h < P; h <<= 1) {
#pragma unroll
    for (int i = 0; i < P; ++i) {
      if (!(i & h)) {
        const uint64_t U = X[i], V = X[i | h];
        X[i] = add2(U, V);
        X[i | h] = sub2(U, V);
      }
    }
  }
  // the level that pairs channel c with c + D/2: the lower half takes mine + theirs, the upper half theirs - mine
  const float sg = part ? -1.0f : 1.0f;
  const uint64_t SG = pack_f32x2(sg, sg);
#pragma unroll
  for (int i = 0; i < P; ++i) {
    float lo, hi;
    unpack2(X[i], lo, hi);
    const float olo = __shfl_xor_sync(0xffffffffu, lo, 16), ohi = __shfl_xor_sync(0xffffffffu, hi, 16);
    X[i] = fma2(X[i], SG, pack_f32x2(olo, ohi));
  }
  constexpr float rs = D == 128 ? 0.08838834764831845f : 0.125f;   // 1/sqrt(D)

  float amax = 0.f;
  if constexpr (STAGE != kStageQuant4) {
    float m0 = 0.f, m1 = 0.f;
#pragma unroll
    for (int i = 0; i < P; i += 2) {
      float a0, a1, b0, b1;
      unpack2(X[i], a0, a1);
      unpack2(X[i + 1], b0, b1);
      m0 = max3(m0, fabsf(a0), fabsf(a1));
      m1 = max3(m1, fabsf(b0), fabsf(b1));
    }
    amax = warp_max(fmaxf(m0, m1) * rs);           // max and the (positive) scale commute exactly
    float* rbuf = red + 8 * (iter & 1);            // alternate buffers: one barrier per item suffices
    if (lane == 0) rbuf[warp] = amax;
    __syncthreads();
    amax = fmaxf(fmaxf(rbuf[0], rbuf[1]), fmaxf(rbuf[2], rbuf[3]));
    amax = fmaxf(amax, fmaxf(fmaxf(rbuf[4], rbuf[5]), fmaxf(rbuf[6], rbuf[7])));
  }
  if constexpr (STAGE == kStageAmax) {
    if (tid == 0) atomicMax(amax_at(), __float_as_uint(amax));
    return;
  }
  if constexpr (STAGE == kStageQuant4) {
    // NVFP4: outer scale g per (b, h), microscale per token per 16 channels (the arithmetic of the
    // general row body: y = x / sqrt(D), then y / (g * microscale), each rounded once)
    const float g = outer();
    const float inv6 = 1.0f / (6.0f * g);
    const uint64_t RS = pack_f32x2(rs, rs);
    constexpr int MB = C / 16;                     // microscale bytes of this thread
    unsigned int codes[C / 8], micro[(MB + 3) / 4];
#pragma unroll
    for (int i = 0; i < (MB + 3) / 4; ++i) micro[i] = 0;
#pragma unroll
    for (int gq = 0; gq < C / 16; ++gq) {
      float m0 = 0.f, m1 = 0.f;
#pragma unroll
      for (int i = 0; i < 8; i += 2) {
        float a0, a1, b0, b1;
        X[8 * gq + i] = mul2(X[8 * gq + i], RS);
        X[8 * gq + i + 1] = mul2(X[8 * gq + i + 1], RS);
        unpack2(X[8 * gq + i], a0, a1);
        unpack2(X[8 * gq + i + 1], b0, b1);
        m0 = max3(m0, fabsf(a0), fabsf(a1));
        m1 = max3(m1, fabsf(b0), fabsf(b1));
      }
      const float m = fmaxf(m0, m1);
      const unsigned int sb = __nv_cvt_float_to_fp8(m * inv6, __NV_SATFINITE, __NV_E4M3);
      const float sdec = e4m3_to_float(sb);
      const float rcp = sdec > 0.f ? 1.0f / (g * sdec) : 0.f;
      const uint64_t RC = pack_f32x2(rcp, rcp);
      micro[gq / 4] |= sb << (8 * (gq & 3));
#pragma unroll
      for (int wi = 0; wi < 2; ++wi) {
        unsigned int word = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float y0, y1;
          unpack2(mul2(X[8 * gq + 4 * wi + j], RC), y0, y1);
          const unsigned int two = __nv_cvt_float2_to_fp4x2(make_float2(y0, y1), __NV_E2M1, cudaRoundNearest);
          word |= (two & 0xffu) << (8 * j);
        }
        codes[2 * gq + wi] = sdec > 0.f ? word : 0u;
      }
    }
    constexpr int CPR4 = D / 32;
    uint4* dst4 = reinterpret_cast<uint4*>(out_tile + row * (D / 2));
    const int sw4 = (row / (8 / CPR4)) & (CPR4 - 1);
#pragma unroll
    for (int i = 0; i < C / 32; ++i) dst4[(part * (C / 32) + i) ^ sw4] = make_uint4(codes[4 * i], codes[4 * i + 1], codes[4 * i + 2], codes[4 * i + 3]);
    const size_t row_g = (size_t)bh * a.n_pad + (size_t)blk * kBlock + row;
    uint8_t* mrow = (TENSOR == 0 ? a.q_micro : a.k_micro) + row_g * (D / 16) + part * MB;
    if constexpr (MB % 4 == 0) {
#pragma unroll
      for (int i = 0; i < MB / 4; ++i) reinterpret_cast<unsigned int*>(mrow)[i] = micro[i];
    } else {
      static_assert(MB == 2, "microscale bytes per thread");
      *reinterpret_cast<unsigned short*>(mrow) = (unsigned short)micro[0];
    }
    return;
  }

  constexpr bool int8 = STAGE == kStageQuant8I;
  const float top = int8 ? 127.0f : 448.0f;
  const float f = amax > 0.f ? rs * (top / amax) : 0.f;   // 1/sqrt(D) and 1/scale in one factor
  if (tid == 0) (TENSOR == 0 ? a.q_scale : a.k_scale)[(size_t)bh * a.nb + blk] = amax > 0.f ? amax / top : 1.0f;
  const uint64_t F = pack_f32x2(f, f);
  constexpr int CPR = D / 16;
  uint4* dst = reinterpret_cast<uint4*>(out_tile + row * D);
  const int sw = (row / (8 / CPR)) & (CPR - 1);
#pragma unroll
  for (int i = 0; i < C / 16; ++i) {
    unsigned int w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int pi = 8 * i + 2 * j;                // pairs pi, pi + 1 = channels 16 i + 4 j .. + 3
      if constexpr (int8) {
        const uint64_t MG = pack_f32x2(12582912.0f, 12582912.0f);
        const uint64_t ra = fma2(X[pi], F, MG), rb = fma2(X[pi + 1], F, MG);
        w[j] = __byte_perm(__byte_perm((unsigned int)ra, (unsigned int)(ra >> 32), 0x0040),
                           __byte_perm((unsigned int)rb, (unsigned int)(rb >> 32), 0x0040), 0x5410);
      } else {
        float y0, y1, y2, y3;
        unpack2(mul2(X[pi], F), y0, y1);
        unpack2(mul2(X[pi + 1], F), y2, y3);
        const unsigned int lo = __nv_cvt_float2_to_fp8x2(make_float2(y0, y1), __NV_SATFINITE, __NV_E4M3);
        const unsigned int hi = __nv_cvt_float2_to_fp8x2(make_float2(y2, y3), __NV_SATFINITE, __NV_E4M3);
        w[j] = lo | (hi << 16);
      }
    }
    dst[(part * (C / 16) + i) ^ sw] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// ---------------------------------------------------------------------------------------
// V.  A thread owns one channel pair and 128 / (256 / (D/2)) consecutive tokens of the gathered
// block, so block means and the channel-major (token-contiguous) code rows need no transposition.
enum { kVStats = 0, kVQuant8 = 1, kVQuant4 = 2, kVQuant4M = 3 };   // 4M: E2M1 under power-of-two factors per 32 tokens

// Statistics of a value block (launch 1b): block mean per channel (Eq. 4) and the block's
// max |v - mu|, folded into the head's per-channel maximum.  One pass over the thread's tokens
// collects the sum, the maximum and the minimum (the last two on the packed bf16 pairs as they
// are: max/min.bf16x2), one exchange combines the token groups, and
//     max_i |v_i - mu| = max(max_i v_i - mu, mu - min_i v_i)
// bit for bit, because the FP32 subtraction is monotonic.
template <int D, bool FULL>
__device__ __forceinline__ void v_stats_item(const PrepArgs& a, const unsigned char* stage, float* red, int bh, int blk, unsigned int* amax_at /*[D]*/) {
  constexpr int CP = D / 2, TG = kThreads / CP, TPG = kBlock / TG;
  const int tid = threadIdx.x;
  const int cp = tid % CP, tg = tid / CP;
  const int n_valid = FULL ? kBlock : min(kBlock, a.N - blk * kBlock);
  const unsigned char* mine = stage + tg * TPG * (2 * D) + 4 * cp;
  float s0 = 0.f, s1 = 0.f;
  __nv_bfloat162 mx = __halves2bfloat162(__ushort_as_bfloat16(0xff80), __ushort_as_bfloat16(0xff80));   // -inf
  __nv_bfloat162 mn = __halves2bfloat162(__ushort_as_bfloat16(0x7f80), __ushort_as_bfloat16(0x7f80));   // +inf
#pragma unroll
  for (int i = 0; i < TPG; ++i) {
    if (FULL || tg * TPG + i < n_valid) {
      const unsigned int w = *reinterpret_cast<const unsigned int*>(mine + i * (2 * D));
      s0 += __uint_as_float(w << 16);
      s1 += __uint_as_float(w & 0xffff0000u);
      const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&w);
      mx = __hmax2(mx, v);
      mn = __hmin2(mn, v);
    }
  }
  // red: [TG][D] sums, then [TG][CP] packed maxima, then [TG][CP] packed minima
  unsigned int* red_mx = reinterpret_cast<unsigned int*>(red + TG * D);
  unsigned int* red_mn = red_mx + TG * CP;
  *reinterpret_cast<float2*>(red + tg * D + 2 * cp) = make_float2(s0, s1);
  red_mx[tg * CP + cp] = *reinterpret_cast<unsigned int*>(&mx);
  red_mn[tg * CP + cp] = *reinterpret_cast<unsigned int*>(&mn);
  __syncthreads();                           // (the barrier at the top of the next item covers these reads)
  if (tg == 0) {
    s0 = 0.f; s1 = 0.f;
#pragma unroll
    for (int g = 0; g < TG; ++g) {
      const float2 p = *reinterpret_cast<const float2*>(red + g * D + 2 * cp);
      s0 += p.x; s1 += p.y;
      if (g > 0) {
        mx = __hmax2(mx, *reinterpret_cast<const __nv_bfloat162*>(&red_mx[g * CP + cp]));
        mn = __hmin2(mn, *reinterpret_cast<const __nv_bfloat162*>(&red_mn[g * CP + cp]));
      }
    }
    const bool smooth = a.flags & VC_FLAG_V_SMOOTH;
    const float mu0 = smooth ? s0 / (float)n_valid : 0.f, mu1 = smooth ? s1 / (float)n_valid : 0.f;
    const size_t mu_at = ((size_t)bh * a.nb + blk) * D + 2 * cp;
    *reinterpret_cast<float2*>(a.v_mu + mu_at) = make_float2(mu0, mu1);
    const float2 hi = __bfloat1622float2(mx), lo = __bfloat1622float2(mn);
    const float m0 = fmaxf(hi.x - mu0, mu0 - lo.x), m1 = fmaxf(hi.y - mu1, mu1 - lo.y);
    atomicMax(&amax_at[2 * cp], __float_as_uint(m0));
    atomicMax(&amax_at[2 * cp + 1], __float_as_uint(m1));
  }
}

// FULL: all 128 rows of the block exist (every block but a head's ragged last one): no row tests.
template <int D, int STAGE, bool FULL>
__device__ __forceinline__ void v_item(const PrepArgs& a, const unsigned char* stage, float* red, int bh, int blk,
                                       float2 mu_in, float2 am_in) {
  constexpr int CP = D / 2;             // channel pairs
  constexpr int TG = kThreads / CP;     // token groups
  constexpr int TPG = kBlock / TG;      // tokens per thread
  const int tid = threadIdx.x;
  const int cp = tid % CP, tg = tid / CP;
  const int n_valid = FULL ? kBlock : min(kBlock, a.N - blk * kBlock);
  float v0[TPG], v1[TPG];
  const unsigned char* mine = stage + tg * TPG * (2 * D) + 4 * cp;
#pragma unroll
  for (int i = 0; i < TPG; ++i) {
    const unsigned int w = (FULL || tg * TPG + i < n_valid) ? *reinterpret_cast<const unsigned int*>(mine + i * (2 * D)) : 0u;
    v0[i] = __uint_as_float(w << 16);
    v1[i] = __uint_as_float(w & 0xffff0000u);
  }
  const bool smooth = a.flags & VC_FLAG_V_SMOOTH;
  const size_t mu_at = ((size_t)bh * a.nb + blk) * D + 2 * cp;
  float mu0 = 0.f, mu1 = 0.f;

  // At 4 bits the values have no tensor-level scale, so nothing of a block's codes depends on
  // other blocks: the block mean is formed here, in the quantizing pass, and the statistics
  // launch is not needed.
  constexpr bool kFusedMean = STAGE == kVQuant4 || STAGE == kVQuant4M;
  static_assert(STAGE != kVStats, "the statistics stage has its own item function");
  if constexpr (kFusedMean) {
    __syncthreads();                         // the previous item's reads of `red` are done
    if (smooth) {
      float s0 = 0.f, s1 = 0.f;
#pragma unroll
      for (int i = 0; i < TPG; ++i) { s0 += v0[i]; s1 += v1[i]; }
      red[tg * D + 2 * cp] = s0;
      red[tg * D + 2 * cp + 1] = s1;
      __syncthreads();
      s0 = 0.f; s1 = 0.f;
#pragma unroll
      for (int g = 0; g < TG; ++g) { s0 += red[g * D + 2 * cp]; s1 += red[g * D + 2 * cp + 1]; }
      mu0 = s0 / (float)n_valid;
      mu1 = s1 / (float)n_valid;
      if constexpr (kFusedMean) {
        // at 4 bits the mean is stored as bf16 and added back unscaled (App. B): subtract exactly
        // that number, so that Eq. 6 restores what Eq. 4 removed
        mu0 = __bfloat162float(__float2bfloat16_rn(mu0));
        mu1 = __bfloat162float(__float2bfloat16_rn(mu1));
      }
      __syncthreads();
    }
  }
  if constexpr (!kFusedMean) {
    mu0 = mu_in.x;
    mu1 = mu_in.y;
  }
  float r0[TPG], r1[TPG];
#pragma unroll
  for (int i = 0; i < TPG; ++i) {
    const bool valid = FULL || tg * TPG + i < n_valid;
    r0[i] = valid ? v0[i] - mu0 : 0.f;
    r1[i] = valid ? v1[i] - mu1 : 0.f;
  }
  const size_t tok0 = (size_t)blk * kBlock + tg * TPG;

  if constexpr (STAGE == kVQuant8) {
    const float am0 = am_in.x, am1 = am_in.y;
    const float inv0 = am0 > 0.f ? 448.0f / am0 : 0.f, inv1 = am1 > 0.f ? 448.0f / am1 : 0.f;
    unsigned int w0[TPG / 4], w1[TPG / 4];
#pragma unroll
    for (int j = 0; j < TPG / 4; ++j) {
      unsigned int lo = __nv_cvt_float2_to_fp8x2(make_float2(r0[4 * j] * inv0, r0[4 * j + 1] * inv0), __NV_SATFINITE, __NV_E4M3);
      unsigned int hi = __nv_cvt_float2_to_fp8x2(make_float2(r0[4 * j + 2] * inv0, r0[4 * j + 3] * inv0), __NV_SATFINITE, __NV_E4M3);
      w0[j] = lo | (hi << 16);
      lo = __nv_cvt_float2_to_fp8x2(make_float2(r1[4 * j] * inv1, r1[4 * j + 1] * inv1), __NV_SATFINITE, __NV_E4M3);
      hi = __nv_cvt_float2_to_fp8x2(make_float2(r1[4 * j + 2] * inv1, r1[4 * j + 3] * inv1), __NV_SATFINITE, __NV_E4M3);
      w1[j] = lo | (hi << 16);
    }
    uint4* d0 = reinterpret_cast<uint4*>(a.v_codes + ((size_t)bh * D + 2 * cp) * a.n_pad + tok0);
    uint4* d1 = reinterpret_cast<uint4*>(a.v_codes + ((size_t)bh * D + 2 * cp + 1) * a.n_pad + tok0);
#pragma unroll
    for (int j = 0; j < TPG / 16; ++j) {
      d0[j] = make_uint4(w0[4 * j], w0[4 * j + 1], w0[4 * j + 2], w0[4 * j + 3]);
      d1[j] = make_uint4(w1[4 * j], w1[4 * j + 1], w1[4 * j + 2], w1[4 * j + 3]);
    }
    if (tg == 0) {   // block means stored divided by the value scale (App. B)
      const float a0 = mu0 * (am0 > 0.f ? inv0 : 1.0f), a1 = mu1 * (am1 > 0.f ? inv1 : 1.0f);
      *reinterpret_cast<__nv_bfloat162*>(a.v_means + mu_at) = __floats2bfloat162_rn(a0, a1);
    }
  }

  if constexpr (STAGE == kVQuant4) {
    // NVFP4 along tokens: one microscale per channel per 16 consecutive permuted tokens
    const float sixth = 1.0f / 6.0f;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const float* r = half == 0 ? r0 : r1;
      const int c = 2 * cp + half;
      unsigned int packed[TPG / 8];
      unsigned int micro = 0;
#pragma unroll
      for (int gq = 0; gq < TPG / 16; ++gq) {
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) m = fmaxf(m, fabsf(r[16 * gq + i]));
        const unsigned int sb = __nv_cvt_float_to_fp8(m * sixth, __NV_SATFINITE, __NV_E4M3);
        const float sdec = e4m3_to_float(sb);
        const float rcp = sdec > 0.f ? 1.0f / sdec : 0.f;
        micro |= sb << (8 * gq);
#pragma unroll
        for (int wi = 0; wi < 2; ++wi) {
          unsigned int word = 0;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int i = 16 * gq + 8 * wi + 2 * j;
            const unsigned int two = __nv_cvt_float2_to_fp4x2(make_float2(r[i] * rcp, r[i + 1] * rcp), __NV_E2M1, cudaRoundNearest);
            word |= (two & 0xffu) << (8 * j);
          }
          packed[2 * gq + wi] = sdec > 0.f ? word : 0u;
        }
      }
      uint8_t* d = a.v_codes + ((size_t)bh * D + c) * (a.n_pad / 2) + tok0 / 2;
      uint8_t* md = a.v_micro + ((size_t)bh * D + c) * (a.n_pad / 16) + tok0 / 16;
      if constexpr (TPG == 32) {
        *reinterpret_cast<uint4*>(d) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        *reinterpret_cast<unsigned short*>(md) = (unsigned short)micro;
      } else {
        *reinterpret_cast<uint2*>(d) = make_uint2(packed[0], packed[1]);
        *md = (uint8_t)micro;
      }
    }
    if (tg == 0)
      *reinterpret_cast<__nv_bfloat162*>(a.v_means + mu_at) = __floats2bfloat162_rn(mu0, mu1);
  }

  if constexpr (STAGE == kVQuant4M) {
    // E2M1 under one power-of-two factor per channel per 32 consecutive permuted tokens (the
    // operand format of the FP8 x FP4 block-scaled product).  Factor 2^e with e the smallest
    // exponent that keeps the group maximum inside the E2M1 range: y = max / 6 (one division),
    // e = exponent(y), plus one unless y is a power of two.  Scaling by 2^-e is exact.
    float m0 = 0.f, m1 = 0.f;
#pragma unroll
    for (int i = 0; i < TPG; ++i) { m0 = fmaxf(m0, fabsf(r0[i])); m1 = fmaxf(m1, fabsf(r1[i])); }
    if constexpr (TPG == 16) {               // a group spans two threads (token groups 2g, 2g + 1)
      __syncthreads();                       // the previous item's reads of `red` are done
      red[tg * D + 2 * cp] = m0;
      red[tg * D + 2 * cp + 1] = m1;
      __syncthreads();
      m0 = fmaxf(m0, red[(tg ^ 1) * D + 2 * cp]);
      m1 = fmaxf(m1, red[(tg ^ 1) * D + 2 * cp + 1]);
    }
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const float* r = half == 0 ? r0 : r1;
      const float m = half == 0 ? m0 : m1;
      const int c = 2 * cp + half;
      const unsigned int yb = __float_as_uint(__fdiv_rn(m, 6.0f));
      int code = (int)((yb >> 23) & 0xffu) + ((yb & 0x7fffffu) ? 1 : 0);     // e + 127
      code = m > 0.f ? min(max(code, 0), 254) : 0;
      const float rs = __uint_as_float((unsigned int)(254 - code) << 23);     // 2^-e
      unsigned int packed[TPG / 8];
#pragma unroll
      for (int wi = 0; wi < TPG / 8; ++wi) {
        unsigned int word = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int i = 8 * wi + 2 * j;
          const unsigned int two = __nv_cvt_float2_to_fp4x2(make_float2(r[i] * rs, r[i + 1] * rs), __NV_E2M1, cudaRoundNearest);
          word |= (two & 0xffu) << (8 * j);
        }
        packed[wi] = m > 0.f ? word : 0u;
      }
      uint8_t* d = a.v_codes + ((size_t)bh * D + c) * (a.n_pad / 2) + tok0 / 2;
      uint8_t* md = a.v_micro + ((size_t)bh * D + c) * (a.n_pad / 32) + tok0 / 32;
      if constexpr (TPG == 32) {
        *reinterpret_cast<uint4*>(d) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        *md = (uint8_t)code;
      } else {
        *reinterpret_cast<uint2*>(d) = make_uint2(packed[0], packed[1]);
        if ((tg & 1) == 0) *md = (uint8_t)code;
      }
    }
    if (tg == 0)
      *reinterpret_cast<__nv_bfloat162*>(a.v_means + mu_at) = __floats2bfloat162_rn(mu0, mu1);
  }
}

// ---------------------------------------------------------------------------------------
// RoPE table -> shared memory (when it fits), once per CTA.
__device__ __forceinline__ RopeTab stage_rope_table(const PrepArgs& a, unsigned char* at, bool folded = false) {
  const float2* src = a.rope + (folded ? a.rd.entries : 0);
  RopeTab tab{0u, src};
  if ((a.flags & VC_FLAG_ROPE) && a.rope_in_smem) {
    float2* tab_s = reinterpret_cast<float2*>(at);
    for (int e = threadIdx.x; e < a.rd.entries; e += blockDim.x) tab_s[e] = __ldg(&src[e]);
    tab.saddr = smem_u32(at);
  }
  __syncthreads();
  return tab;
}

// Where a CTA stands in a pass: CTA `rank` of `stride`, n items.
struct Slot {
  int rank, stride, n_items;
};

// Column sums of RoPE(K) per block (the channel mean is taken after the rotation).
// Shared memory: [2 stages x 32 KB][red: 8 D floats][RoPE table].
template <int D>
__device__ __forceinline__ void kcolsum_pass(const PrepArgs& a, unsigned char* smem, const Slot sl, int nh) {
  constexpr int LPR = D / 8, RPL = LPR / 2, kStage = kThreads * RPL * 16;
  float* red = reinterpret_cast<float*>(smem + 2 * kStage);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lr = lane % LPR, hb = lane / LPR;
  const PairSlots ps = pair_slots(a.rd, 4 * lr);
  const CursorStep step = cursor_step(sl.stride, a.nb);
  auto issue = [&](int item, const Cursor& c, int st) {
    if (item < sl.n_items) {
      const char* base = reinterpret_cast<const char*>(a.k) + head_offset_bytes(a, a.bh0 + c.hh) + 16 * lr;
      const int t0 = c.blk * kBlock + 16 * warp + RPL * hb;
      unsigned char* dst = smem + st * kStage + tid * 16;
#pragma unroll
      for (int i = 0; i < RPL; ++i)
        if (t0 + i < a.N) cp_async16(dst + i * kThreads * 16, base + (int64_t)(t0 + i) * a.stride_n_bytes);
    }
    cp_async_commit();
  };
  Cursor cur = cursor_at(sl.rank, a.nb, nh), nxt = cur;
  advance(nxt, step, a.nb, nh);
  issue(sl.rank, cur, 0);
  pdl_wait();
  const RopeTab tab = stage_rope_table(a, smem + 2 * kStage + 8 * D * 4);
  int i = 0;
  for (int item = sl.rank; item < sl.n_items; item += sl.stride, ++i) {
    issue(item + sl.stride, nxt, (i + 1) & 1);
    cp_async_wait<1>();                       // this thread's chunks of item i have landed
    k_colsum_item<D>(a, smem + (i & 1) * kStage + tid * 16, kThreads * 16, red, tab, ps, a.k_part + ((size_t)(a.bh0 + cur.hh) * a.nb + cur.blk) * D, cur.blk);
    cur = nxt;
    advance(nxt, step, a.nb, nh);
  }
}

// V pass: STAGE = block means + residual amax, or quantization of the residual.
// Shared memory: [3 stages x (128 x 2 D)][red: 16 D floats][source rows: 2 x 128].
template <int D, int STAGE>
__device__ __forceinline__ void v_pass(const PrepArgs& a, unsigned char* smem, const Slot sl, int nh) {
  constexpr int LPR = D / 8, kStage = kBlock * 2 * D, NL = kBlock * LPR / kThreads;
  float* red = reinterpret_cast<float*>(smem + 3 * kStage);
  int* src_ring = reinterpret_cast<int*>(red + 16 * D);                // [2][128]
  const int tid = threadIdx.x;
  const CursorStep step = cursor_step(sl.stride, a.nb);
  // source row of row `tid` of an item (the gather by pi), -1 if there is none
  auto fetch = [&](int item, const Cursor& c) -> int {
    if (item >= sl.n_items || tid >= kBlock) return -1;
    const int t = c.blk * kBlock + tid;
    if (t >= a.N) return -1;
    return a.perm ? min(max(__ldg(a.perm + (size_t)(a.bh0 + c.hh) * a.N + t), 0), a.N - 1) : t;   // clamped: never a bad address
  };
  auto issue = [&](int item, const Cursor& c, int st, const int* src) {
    if (item < sl.n_items) {
      const char* base = reinterpret_cast<const char*>(a.v) + head_offset_bytes(a, a.bh0 + c.hh) + 16 * (tid % LPR);
      unsigned char* dst = smem + st * kStage + tid * 16;
#pragma unroll
      for (int k = 0; k < NL; ++k) {
        const int sr = src[tid / LPR + k * (kThreads / LPR)];
        if (sr >= 0) cp_async16(dst + k * kThreads * 16, base + (int64_t)sr * a.stride_n_bytes);
      }
    }
    cp_async_commit();
  };
  // per-item scalars of the quantizing stage, fetched one item ahead
  const int cp = tid % (D / 2);
  auto fetch_mu = [&](int item, const Cursor& c) -> float2 {
    if (STAGE == kVStats || STAGE == kVQuant4 || STAGE == kVQuant4M || item >= sl.n_items) return make_float2(0.f, 0.f);
    return *reinterpret_cast<const float2*>(a.v_mu + ((size_t)(a.bh0 + c.hh) * a.nb + c.blk) * D + 2 * cp);
  };
  // cursors of items i, i+1, i+2 and i+4 of this CTA
  const int g = sl.stride;
  Cursor c0 = cursor_at(sl.rank, a.nb, nh), c1 = c0;
  advance(c1, step, a.nb, nh);
  Cursor c2 = c1;
  advance(c2, step, a.nb, nh);
  Cursor c4 = c2;
  advance(c4, step, a.nb, nh);
  if (tid < kBlock) {
    src_ring[tid] = fetch(sl.rank, c0);
    src_ring[kBlock + tid] = fetch(sl.rank + g, c1);
  }
  __syncthreads();
  issue(sl.rank, c0, 0, src_ring);
  issue(sl.rank + g, c1, 1, src_ring + kBlock);
  __syncthreads();                            // the two slices have been read
  if (tid < kBlock) src_ring[tid] = fetch(sl.rank + 2 * g, c2);
  int nxt = fetch(sl.rank + 3 * g, c4);    // (c4 still stands at item 3 here)
  advance(c4, step, a.nb, nh);
  pdl_wait();                                 // (the inputs are in flight; the statistics may be read from here on)
  float2 mu = fetch_mu(sl.rank, c0), am = make_float2(0.f, 0.f);
  int i = 0, last_hh = -1;
  for (int item = sl.rank; item < sl.n_items; item += g, ++i) {
    cp_async_wait<1>();                       // my chunks of item i have landed ...
    __syncthreads();                          // ... and everyone's; all are done with item i-1
    if (tid < kBlock) src_ring[((i + 1) & 1) * kBlock + tid] = nxt;     // source rows of item i+3
    nxt = fetch(item + 4 * g, c4);
    issue(item + 2 * g, c2, (i + 2) % 3, src_ring + (i & 1) * kBlock);
    const float2 mu_next = fetch_mu(item + g, c1);
    if (STAGE == kVQuant8 && c0.hh != last_hh) {
      const size_t at = (size_t)(a.bh0 + c0.hh) * D + 2 * cp;
      am = make_float2(__uint_as_float(a.v_amax[at]), __uint_as_float(a.v_amax[at + 1]));
      last_hh = c0.hh;
    }
    const unsigned char* stage = smem + (i % 3) * kStage;
    const bool full = a.N - c0.blk * kBlock >= kBlock;
    if constexpr (STAGE == kVStats) {
      unsigned int* amax_at = a.v_amax + (size_t)(a.bh0 + c0.hh) * D;
      if (full) v_stats_item<D, true>(a, stage, red, a.bh0 + c0.hh, c0.blk, amax_at);
      else v_stats_item<D, false>(a, stage, red, a.bh0 + c0.hh, c0.blk, amax_at);
    } else {
      if (full) v_item<D, STAGE, true>(a, stage, red, a.bh0 + c0.hh, c0.blk, mu, am);
      else v_item<D, STAGE, false>(a, stage, red, a.bh0 + c0.hh, c0.blk, mu, am);
    }
    mu = mu_next;
    c0 = c1; c1 = c2;
    advance(c2, step, a.nb, nh);
    advance(c4, step, a.nb, nh);
  }
}

// Per-head finalization.  kMeans: K channel mean, V scale; a block of 8 D threads per head, the block partial sums are added in
// double, in eight interleaved slices that are then added in a fixed order.  kOuter (4 bits): the outer scale of Q, or on its
// own, behind the next launch, that of K.
enum { kMeans = 1, kOuter = 2 };
template <int D, int BITS, int WHAT>
__global__ void prep_finalize_kernel(const PrepArgs a) {
  __shared__ double part[8][D];
  const int bh = a.bh0 + blockIdx.x, c = threadIdx.x % D, slice = threadIdx.x / D;
  pdl_wait();
  pdl_allow();
  if ((WHAT & kOuter) && threadIdx.x == 0) {
    constexpr bool kOfK = !(WHAT & kMeans);
    (kOfK ? a.k_scale : a.q_scale)[bh] = outer_scale(__uint_as_float(a.qk_amax[kOfK * a.BH + bh]));
  }
  if (!(WHAT & kMeans)) return;
  if (a.flags & VC_FLAG_K_SMOOTH) {
    double s = 0.0;
#pragma unroll 8
    for (int j = slice; j < a.nb; j += 8) s += (double)a.k_part[((size_t)bh * a.nb + j) * D + c];
    part[slice][c] = s;
    __syncthreads();
  }
  if (slice == 0) {
    double s = 0.0;
    if (a.flags & VC_FLAG_K_SMOOTH)
      for (int k = 0; k < 8; ++k) s += part[k][c];
    a.k_mean[(size_t)bh * D + c] = (float)(s / (double)a.N);
    a.v_scale[(size_t)bh * D + c] = BITS == 8 ? value_scale(__uint_as_float(a.v_amax[(size_t)bh * D + c])) : 1.0f;
  }
}

// A warp's rows of the swizzled code tile, from row0 on -> rows `first` + row0 and on of `codes`: full-line stores.
template <int ROW_BYTES>
__device__ __forceinline__ void store_warp_rows(uint8_t* codes, size_t first, const unsigned char* out_tile, int row0, int lane) {
  constexpr int CPR = ROW_BYTES / 16, RW = 32 / kTpr;                // 16-byte chunks per code row, rows of a warp
  uint4* gdst = reinterpret_cast<uint4*>(codes + (first + row0) * ROW_BYTES) + lane;
#pragma unroll
  for (int k = 0; k < CPR * RW / 32; ++k) {
    const int idx = k * 32 + lane, row = row0 + idx / CPR, chunk = idx % CPR;
    const int sw = (row / (8 / CPR)) & (CPR - 1);
    gdst[k * 32] = *reinterpret_cast<const uint4*>(out_tile + row * ROW_BYTES + ((chunk ^ sw) << 4));
  }
}

// Q/K pass: STAGE = amax (4-bit head amax of tensor z0), or quantization of Q (z = 0) and K
// (z = 1).  A warp owns 32 / kTpr rows of the block from end to end: it copies them in (consecutive
// lanes on consecutive 16-byte chunks, the source rows taken from a small ring of permutation
// entries in shared memory), its threads read their rows from the padded tile, and the rows'
// codes leave through the warp's slice of a swizzled tile, again with full-line stores.  So the
// data needs warp-level synchronization only; the one CTA-wide barrier per item is the exchange
// of the block maximum.
// Shared memory: [2 stages x 128 x pitch][out tile 128 x D][src ring 3 x 128][scratch][RoPE table].
// FAST: the packed row transform (standard configuration), see qk_row_item_fast.  OUTER: the items form the NVFP4 outer scale
// from the head maximum themselves, one of a head's blocks stores it (else it is read).
template <int D, int STAGE, bool FAST, bool OUTER = false>
__device__ __forceinline__ void qk_pass(const PrepArgs& a, unsigned char* smem, const Slot sl, int nh, int z0) {
  constexpr int NT = kRowThreads * kTpr;
  constexpr int kRowBytes = STAGE == kStageQuant4 ? D / 2 : D;      // code bytes per row
  constexpr int RW = 32 / kTpr;                                      // rows of a warp
  constexpr int LPR = D / 8;                                         // lanes on one input row
  constexpr int RPI = 32 / LPR;                                      // input rows per warp instruction
  unsigned char* out_tile = smem + 2 * Geo<D>::stage_bytes;
  int* src_ring = reinterpret_cast<int*>(out_tile + kBlock * D);     // [3][128]
  float* red = reinterpret_cast<float*>(src_ring + 3 * kBlock);      // [2][8]
  float* kmean_s = red + 16;                                         // [D]
  const int tid = threadIdx.x, lane = tid & 31, row0 = (tid >> 5) * RW;
  if (FAST) {
    for (int c = tid; c < D; c += NT) kmean_s[c] = 0.f;    // (m+, m-) pairs: zeros until a smoothed K head arrives
  }
  const int my_row = qk_row_of(tid);
  const CursorStep step = cursor_step(sl.stride, a.nb);
  auto fetch = [&](int item, const Cursor& c) -> int {   // input row behind row `row0 + lane` of the item, -1 if none
    if (item >= sl.n_items || lane >= RW) return -1;
    const int t = c.blk * kBlock + row0 + lane;
    if (t >= a.N) return -1;
    // the head amax is a maximum over all rows: that stage reads the rows in place
    const bool gather = (c.z + z0) == 1 && a.perm != nullptr && STAGE != kStageAmax;
    return gather ? min(max(__ldg(&a.perm[(size_t)(a.bh0 + c.hh) * a.N + t]), 0), a.N - 1) : t;   // clamped: never a bad address
  };
  auto issue = [&](int item, const Cursor& c, int st, const int* src) {
    if (item < sl.n_items) {
      const char* base = reinterpret_cast<const char*>((c.z + z0) == 0 ? a.q : a.k) + head_offset_bytes(a, a.bh0 + c.hh) + 16 * (lane % LPR);
      unsigned char* dst = smem + st * Geo<D>::stage_bytes + 16 * (lane % LPR) + (row0 + lane / LPR) * Geo<D>::pitch;
#pragma unroll
      for (int k = 0; k < RW / RPI; ++k) {
        const int sr = src[row0 + lane / LPR + k * RPI];
        if (sr >= 0) cp_async16(dst + k * RPI * Geo<D>::pitch, base + (int64_t)sr * a.stride_n_bytes);
      }
    }
    cp_async_commit();
  };
  // cursors of items i, i+1 and i+3 of this CTA
  const int g = sl.stride;
  Cursor c0 = cursor_at(sl.rank, a.nb, nh), c1 = c0;
  advance(c1, step, a.nb, nh);
  Cursor c3 = c1;
  advance(c3, step, a.nb, nh);
  if (lane < RW) {
    src_ring[row0 + lane] = fetch(sl.rank, c0);
    src_ring[kBlock + row0 + lane] = fetch(sl.rank + g, c1);
  }
  int nxt = fetch(sl.rank + 2 * g, c3);    // (c3 still stands at item 2 here)
  advance(c3, step, a.nb, nh);
  __syncwarp();
  issue(sl.rank, c0, 0, src_ring);
  pdl_wait();                                 // (the first rows are in flight)
  const RopeTab tab = stage_rope_table(a, reinterpret_cast<unsigned char*>(kmean_s + D), FAST);
  int i = 0, last_hh = -1;
  for (int item = sl.rank; item < sl.n_items; item += g, ++i) {
    cp_async_wait<0>();                       // my chunks of item i have landed ...
    __syncwarp();                             // ... and the warp's; the warp is done with item i-1
    if (lane < RW) src_ring[((i + 2) % 3) * kBlock + row0 + lane] = nxt;
    nxt = fetch(item + 3 * g, c3);
    issue(item + g, c1, (i + 1) & 1, src_ring + ((i + 1) % 3) * kBlock);
    const unsigned char* stage = smem + (i & 1) * Geo<D>::stage_bytes;
    const int s0 = src_ring[(i % 3) * kBlock + my_row];
    const int tensor = c0.z + z0, bh = a.bh0 + c0.hh;
    auto amax_at = [&] { return a.qk_amax + tensor * a.BH + bh; };
    auto outer = [&] {
      if constexpr (!OUTER) return (tensor == 0 ? a.q_scale : a.k_scale)[bh];
      const float s = outer_scale(__uint_as_float(*amax_at()));
      if (tid == 0 && c0.blk == 0) (tensor == 0 ? a.q_scale : a.k_scale)[bh] = s;
      return s;
    };
    if constexpr (FAST)
      qk_row_item_fast<D, STAGE>(a, tensor, stage, out_tile, red, kmean_s, tab.saddr, bh, c0.blk, i, tensor == 1 && c0.hh != last_hh, s0, amax_at, outer);
    else
      qk_row_item<D, STAGE>(a, tensor, stage, out_tile, red, kmean_s, tab, bh, c0.blk, i, tensor == 1 && c0.hh != last_hh, s0, amax_at, outer);
    if (tensor == 1) last_hh = c0.hh;
    if constexpr (STAGE != kStageAmax) {
      __syncwarp();                           // the warp's rows of the code tile are complete
      store_warp_rows<kRowBytes>(tensor == 0 ? a.q_codes : a.k_codes, (size_t)bh * a.n_pad + (size_t)c0.blk * kBlock, out_tile, row0, lane);
    }
    c0 = c1;
    advance(c1, step, a.nb, nh);
    advance(c3, step, a.nb, nh);
  }
}

// ---------------------------------------------------------------------------------------
// Launches.  Passes that do not depend on one another share one: the statistics passes wait on their
// copies, the Q/K row transform on instruction issue and the shared-memory pipe, so CTAs of both kinds
// on an SM overlap where either kind alone leaves the other resource idle.  Each pass gets a share of
// the CTAs (2 per SM) in proportion to what it costs alone, or all take every pass in turn (see share_ctas).
//   8 bits  1: K column sums | V statistics | Q codes      2: K codes | V codes
//   4 bits  1: K column sums | Q head maximum | V codes    2: K head maximum | Q codes    3: K codes
// (On a wide grid the passes over rows leave the launches they share with the others, see run_phases.)
// with the per-head finalization in between.
enum { kPhase1 = 1, kPhase2 = 2, kPhase3 = 3 };

// Time of 128 rows of each pass relative to the Q/K quantizing pass, tuned with the passes side by side
// (B1 H40 N32760 573 -> 569 us, B1 H12 N32760 190 -> 186 against the ratios measured alone).
constexpr float kCostRows = 1.0f, kCostAmax = 0.9f, kCostSums = 0.6f, kCostVStats = 0.47f, kCostV8 = 0.66f, kCostV4 = 1.0f;

// Which CTAs take the items of which pass: ctas[k] CTAs share pass k's items, in shares one pass's CTAs behind
// the other's, in turns from CTA first[k] on (modulo the grid).
struct Share {
  int items[3], first[3], ctas[3];
  int grid;
  int z0;                    // first tensor of the Q/K quantizing pass (0 = Q, 1 = K)
};

// Pass PASS of a launch.  VARIANT: INT8 codes (8 bits), power-of-two value factors (4 bits, launch 1), outer scale formed from the
// head maximum by every item (4 bits, launches 2 and 3).
template <int D, int BITS, int PHASE, bool FAST, int VARIANT, int PASS>
__device__ __forceinline__ void one_pass(const PrepArgs& a, unsigned char* smem, const Slot sl, int nh, int z0) {
  constexpr int kQuant = BITS == 4 ? kStageQuant4 : (VARIANT ? kStageQuant8I : kStageQuant8);
  if constexpr (PHASE == kPhase1 && PASS == 0) qk_pass<D, BITS == 8 ? kQuant : kStageAmax, FAST>(a, smem, sl, nh, 0);
  else if constexpr (PHASE == kPhase1 && PASS == 1) kcolsum_pass<D>(a, smem, sl, nh);
  else if constexpr (PHASE == kPhase1) v_pass<D, BITS == 8 ? kVStats : (VARIANT ? kVQuant4M : kVQuant4)>(a, smem, sl, nh);
  else if constexpr (BITS == 8 && PASS == 0) qk_pass<D, kQuant, FAST>(a, smem, sl, nh, z0);
  else if constexpr (BITS == 8) v_pass<D, kVQuant8>(a, smem, sl, nh);
  else if constexpr (PHASE == kPhase2 && PASS == 0) qk_pass<D, kQuant, FAST, VARIANT != 0>(a, smem, sl, nh, 0);
  else if constexpr (PHASE == kPhase2) qk_pass<D, kStageAmax, FAST>(a, smem, sl, nh, 1);
  else qk_pass<D, kQuant, FAST, VARIANT != 0>(a, smem, sl, nh, 1);
}

// TURNS = false: a CTA belongs to one pass.  TURNS = true: every CTA takes its part of every pass, one pass after
// the other; the second half of the CTAs starts with the second pass, so that kinds still meet on an SM.
template <int D, int BITS, int PHASE, bool FAST, int VARIANT, bool TURNS>
__global__ void __launch_bounds__(kThreads, 2) prep_kernel(const PrepArgs a, const Share s, int nh) {
  extern __shared__ __align__(128) unsigned char smem[];
  // (No early pdl_allow: attention CTAs that start one by one as this kernel's leave do not run through a
  // head's key tiles together, and the hybrid attention takes 3.5 percent longer at B1 H40 N32760, 3.6 at
  // B1 H12 N32760.  Nor where the attention is one wave: 1 to 2 percent at 2000 to 4000 tokens.  The next kernel
  // starts when the last CTA has ended.)
  constexpr int kPasses = PHASE == kPhase3 ? 1 : (PHASE == kPhase1 ? 3 : 2);
  const int b = blockIdx.x;
  if constexpr (!TURNS) {
    const int n0 = s.ctas[0], n1 = s.ctas[1];
    if (kPasses == 1 || b < n0) one_pass<D, BITS, PHASE, FAST, VARIANT, 0>(a, smem, Slot{b, n0, s.items[0]}, nh, s.z0);
    else if (kPasses == 2 || b < n0 + n1) one_pass<D, BITS, PHASE, FAST, VARIANT, 1>(a, smem, Slot{b - n0, n1, s.items[1]}, nh, s.z0);
    else one_pass<D, BITS, PHASE, FAST, VARIANT, 2>(a, smem, Slot{b - n0 - n1, s.ctas[2], s.items[2]}, nh, s.z0);
  } else {
    int k = 2 * b >= s.grid ? 1 : 0;
    bool again = false;
#pragma unroll 1
    for (int turn = 0; turn < kPasses; ++turn, k = k + 1 < kPasses ? k + 1 : 0) {
      const int items = k == 0 ? s.items[0] : (k == 1 ? s.items[1] : s.items[2]);
      const int first = k == 0 ? s.first[0] : (k == 1 ? s.first[1] : s.first[2]);
      const int ctas = k == 0 ? s.ctas[0] : (k == 1 ? s.ctas[1] : s.ctas[2]);
      const int rank = b >= first ? b - first : b - first + s.grid;
      if (rank >= ctas) continue;
      if (again) { cp_async_wait<0>(); __syncthreads(); }       // the stages are the next pass's
      again = true;
      const Slot sl{rank, ctas, items};
      if (k == 0) one_pass<D, BITS, PHASE, FAST, VARIANT, 0>(a, smem, sl, nh, s.z0);
      else if (kPasses == 2 || k == 1) one_pass<D, BITS, PHASE, FAST, VARIANT, 1>(a, smem, sl, nh, s.z0);
      else one_pass<D, BITS, PHASE, FAST, VARIANT, 2>(a, smem, sl, nh, s.z0);
    }
  }
}

// Shared memory that lets two CTAs of a launch stay on an SM.
constexpr size_t kHalfSm = 113 * 1024;

// Shares of a launch on `per_sm` CTAs per SM.  While they fit, every item has a CTA.  Up to turns_from items per
// CTA each pass gets CTAs in proportion to items x cost.  Beyond that every CTA takes its part of every pass: the
// costs hold for one head dimension, one set of passes and one locality of the gather, and a pass whose
// CTAs have too much keeps the launch waiting.  A CTA pays for it with one more filling of its pipeline
// per pass, some 3 us.  Measured at 8 bits, d128 (the costs' own case): B1 H24 N32760 in shares 333 us, in
// turns 339; H32 442 and 436; H40 550 and 540; H24 N118800 1246 and 1159 (a launch per pass: 1206).  Elsewhere
// turns win from 16 items per CTA on: d64 B1 H8 N32760 80 and 74 us, H12 N327680 1143 and 971 (a
// launch per pass: 1067); 4 bits d64 H40 N32760 524 and 459 (488); supplied statistics, d128, H24 N118800
// 1020 and 859 (863); without K smoothing H40 N32760 483 and 452 (474).
struct Work {
  int items;
  float cost;
};
inline Share share_ctas(const Work w0, const Work w1, const Work w2, int z0, int per_sm, int turns_from, bool* turns) {
  const Work w[3] = {w0, w1, w2};
  const int64_t most = (int64_t)per_sm * sm_count(), items = (int64_t)w0.items + w1.items + w2.items;
  Share s{};
  s.z0 = z0;
  for (int k = 0; k < 3; ++k) s.items[k] = s.ctas[k] = w[k].items;
  *turns = items > most * (int64_t)turns_from && w0.items != items && w1.items != items && w2.items != items;
  if (*turns) {
    int64_t at = 0;
    for (int k = 0; k < 3; ++k) {
      s.first[k] = (int)(at % most);          // item i of the launch belongs to CTA i % grid
      s.ctas[k] = w[k].items < most ? w[k].items : (int)most;
      at += w[k].items;
    }
    s.grid = (int)most;
    return s;
  }
  if (items > most) {
    const float all = w0.items * w0.cost + w1.items * w1.cost + w2.items * w2.cost;
    int left = (int)most;
    for (int k = 2; k >= 0; --k) {
      if (w[k].items == 0) continue;
      const int part = k == 0 ? left : (int)(w[k].items * w[k].cost / all * (float)most);
      s.ctas[k] = part < 1 ? 1 : part < w[k].items ? part : w[k].items;
      left -= s.ctas[k];
    }
  }
  s.grid = s.ctas[0] + s.ctas[1] + s.ctas[2];
  return s;
}

template <auto KERNEL>
cudaError_t launch_phase(const PrepArgs& a, const Share& sh, int nh, size_t smem, cudaStream_t s) {
  cudaError_t e = allow_smem<KERNEL>();
  if (e == cudaSuccess) e = launch_overlapped(KERNEL, dim3((unsigned)sh.grid), kThreads, smem, s, a, sh, nh);
  count_launches(1);
  return e;
}

template <int D, int BITS, bool FAST, int VARIANT>
cudaError_t run_phases(const Problem& pr, PrepArgs a, cudaStream_t s) {
  static_assert(kRowThreads * kTpr == kThreads, "the passes of a launch have the same block size");
  const size_t rope_bytes = ((a.flags & VC_FLAG_ROPE) && a.rope_in_smem) ? (size_t)a.rd.entries * 8 : 0;
  const size_t row_smem = 2 * (size_t)Geo<D>::stage_bytes + (size_t)kBlock * D + 3 * kBlock * 4 + 64 + D * 4 + rope_bytes;
  const size_t v_smem = 3 * (size_t)kBlock * 2 * D + 16 * D * 4 + 2 * kBlock * 4;
  const size_t sum_smem = 2 * (size_t)kThreads * (D / 16) * 16 + 8 * D * 4 + rope_bytes;
  const size_t smem = row_smem > v_smem ? row_smem : v_smem, rest_smem = sum_smem > v_smem ? sum_smem : v_smem;
  static_assert(2 * kThreads * (D / 16) * 16 + 8 * D * 4 <= 2 * Geo<D>::stage_bytes + kBlock * D, "the column sums fit the row pass's share");
  const bool ext = a.ext_k_mean != nullptr;     // the caller supplied the statistics: no statistics passes
  const bool tuned = D == 128 && BITS == 8 && !ext && (a.flags & VC_FLAG_K_SMOOTH);
  const int turns_from = tuned ? 80 : 16;
  // A grid with long axes has a table that leaves an SM room for one CTA of the row pass (at d128 from 27.6 KB on,
  // 3448 entries).  The rows then get launches of their own, so that the passes that need less do not come
  // down to one CTA per SM too.  8 bits, d128: 21 x 68 x 120 H3 332 -> 283 us, 1 x 128 x 128 H39 394 -> 337,
  // 33 x 90 x 160 H1 335 -> 318 (all passes in launches of their own: 321, 363, 347).
  const bool wide = smem > kHalfSm;
  cudaError_t e = cudaSuccess;
  int group = pr.heads_per_pass > 0 ? pr.heads_per_pass : pr.BH;
  if (group > 32768) group = 32768;
  for (int bh0 = 0; bh0 < pr.BH && e == cudaSuccess; bh0 += group) {
    const int nh = pr.BH - bh0 < group ? pr.BH - bh0 : group;
    const int per = pr.nb * nh;
    a.bh0 = bh0;
    const int sums = a.flags & VC_FLAG_K_SMOOTH ? per : 0;
    auto finalize = [&](auto kernel, int threads) {
      if (e == cudaSuccess) e = launch_overlapped(kernel, dim3((unsigned)nh), threads, 0, s, a);
      count_launches(1);
    };
    auto launch = [&](auto whole, auto in_turns, size_t bytes, Work w0, Work w1, Work w2, int z0) {
      bool turns;                                // (kinds do not meet on an SM that holds one CTA: no turns)
      const Share sh = bytes > kHalfSm ? share_ctas(w0, w1, w2, z0, 1, INT_MAX, &turns) : share_ctas(w0, w1, w2, z0, 2, turns_from, &turns);
      if (e == cudaSuccess) e = turns ? in_turns(a, sh, nh, bytes, s) : whole(a, sh, nh, bytes, s);
    };
    const Work none{0, 0.f}, rows{per, kCostRows}, amax{per, kCostAmax}, k_sums{sums, kCostSums}, v_stats{per, kCostVStats}, v_codes{per, kCostV8},
        v_codes4{per, kCostV4};
    if constexpr (BITS == 8) {
      const auto first = launch_phase<prep_kernel<D, 8, kPhase1, FAST, VARIANT, false>>, first_turns = launch_phase<prep_kernel<D, 8, kPhase1, FAST, VARIANT, true>>,
                 second = launch_phase<prep_kernel<D, 8, kPhase2, FAST, VARIANT, false>>, second_turns = launch_phase<prep_kernel<D, 8, kPhase2, FAST, VARIANT, true>>;
      if (!ext) {
        launch(first, first_turns, wide ? rest_smem : smem, wide ? none : rows, k_sums, v_stats, 0);
        finalize(prep_finalize_kernel<D, 8, kMeans>, 8 * D);
      }
      // (with supplied statistics there is no first launch for Q to share; on a wide grid it does not share one)
      const bool q_too = ext || wide;
      launch(second, second_turns, wide ? row_smem : smem, Work{q_too ? 2 * per : per, kCostRows}, wide ? none : v_codes, none, q_too ? 0 : 1);
      if (wide) launch(second, second_turns, v_smem, none, v_codes, none, 0);
    } else {
      const auto first = launch_phase<prep_kernel<D, 4, kPhase1, FAST, VARIANT, false>>, first_turns = launch_phase<prep_kernel<D, 4, kPhase1, FAST, VARIANT, true>>,
                 second = launch_phase<prep_kernel<D, 4, kPhase2, FAST, 0, false>>, second_turns = launch_phase<prep_kernel<D, 4, kPhase2, FAST, 0, true>>,
                 third = launch_phase<prep_kernel<D, 4, kPhase3, FAST, 0, false>>, third_outer = launch_phase<prep_kernel<D, 4, kPhase3, FAST, 1, false>>,
                 second_outer = launch_phase<prep_kernel<D, 4, kPhase2, FAST, FAST, false>>;
      launch(first, first_turns, wide ? rest_smem : smem, wide ? none : amax, k_sums, v_codes4, 0);
      if (wide) launch(first, first_turns, row_smem, amax, none, none, 0);
      // The outer scales.  K's in a launch of its own is some 0.6 us of the chain, Q's in the finalization 0.3; forming them in every
      // item costs 1 percent of the codes' passes.  So the items form them while a CTA has few.  By items / by launches, NVFP4:
      // B1 H12 N4096 d64 29.0 / 29.5 us, d128 41.6 / 42.2; H12 N16384 d64 81.0 / 81.6; H12 N32760 (10 items per CTA) d64 146.5 /
      // 146.4; H40 (35) d64 438 / 435; H24 N118800 (75) d64 908 / 899, d128 without RoPE 1506 / 1434.
      // Q's share a launch with another pass, which goes in turns beyond turns_from items per CTA of both (share_ctas): the items
      // form them only where it does not.  (And not in the general row body, which has no registers left for it.)
      const bool few = per <= 16 * 2 * sm_count(), q_too = FAST && 2 * per <= turns_from * 2 * sm_count();
      if (q_too) {
        finalize(prep_finalize_kernel<D, 4, kMeans>, 8 * D);
        launch(second_outer, second_outer, smem, rows, amax, none, 0);
      } else {
        finalize(prep_finalize_kernel<D, 4, kMeans | kOuter>, 8 * D);
        launch(second, second_turns, smem, rows, amax, none, 0);
      }
      if (!few) finalize(prep_finalize_kernel<D, 4, kOuter>, 32);
      const auto codes = few ? third_outer : third;
      launch(codes, codes, smem, rows, none, none, 1);
    }
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Short heads in front of an attention launch: the whole pass in one launch, a cluster of CTAs per head and tensor, a CTA
// per block.  Few blocks keep the GPU busy for a few microseconds, and what the pass then costs is its chain of
// launches: table, statistics, finalization, codes, at 4 bits one more, 0.8 to 1.5 us from the end of each to the start of
// the next beside its own filling of a pipeline (13.2 us from the table's start to the attention's at B1 H2 N1024 d128).  Here
//   - every CTA computes the RoPE tables it needs itself, in front of the wait for the kernel before it;
//   - a CTA keeps its block in shared memory, so V is read once, and K once unless a permutation gathers it; the statistics
//     of a head meet in distributed shared memory, behind one cluster barrier each;
//   - gathered K is staged twice: in sequence order for the column sums (and the head maximum), gathered for the codes
//     (from L2 as a rule).  The sums run over the same blocks, in the same order, as in the launches above.
// The row and value transforms are the ones of the other launches, and the bundle is the same, byte for byte.
// Whole calls, d128, a launch per phase -> this one: FP8 (four launches) B1 H1 N1024 23.1 -> 18.4 us, H12 25.9 -> 24.9, H9 N576
// 21.8 -> 18.0, H4 N200 18.0 -> 13.9; NVFP4 (five) H12 N1024 35.3 -> 30.3, H4 N200 25.6 -> 18.3.  What bounds it: latency. Tables
// 1.5 to 2.5 us, rows 1.5, column sums 2, barrier 0.8, fold 1, codes 2.
// The tables are hidden when calls of the library follow one another.  Behind a caller's kernel, which lets nothing start early,
// they are in the open: H1 N1024 20.4 us instead of 18.4, 1 x 1 x 64 tokens (1387 entries) 16.4 instead of 12.2 (a launch per phase
// 23.1 and 18.5 to 19.2 either way).  And every CTA computes its own: where many streams fill the GPU with such calls the sum of the
// work counts, NVFP4 H8 N1024 on eight streams 13.6 us a call (13.0 with a launch per phase; on two 16.1 against 18.7).
struct Short {
  double theta, n;           // n: tokens
  unsigned int* status;
};
enum { kShortK = 0, kShortV = 1, kShortQ = 2 };
// Blocks of a head at most: the CTAs of a portable cluster.  (Clusters of 16 find room on few GPCs at a time: B1 H6 N1955
// d64 35.1 us instead of 27.7 when calls follow one another.  Two blocks a CTA in clusters of 8: 27.7, no gain.)
constexpr int kShortCluster = 8;
constexpr int kShortEntries = 1408;    // RoPE table entries at most: at d128 two CTAs stay on an SM

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// The word at `p` of this CTA's shared memory, in the CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_word(const void* p, int rank) {
  uint32_t at, v;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  return v;
}
// x / n for an integer n <= 128 kShortCluster, correctly rounded, with inv = 1 / n (rounded) already at hand: a quotient and one
// correction by its remainder, three operations in place of a division behind the sums.  q is within 1.5 ulp of x / n (two
// roundings), so x - q n is a multiple of ulp(q) below 2^12 of them: exact.  What is added is then off by 2^-52 of an ulp, while
// x / n lies at least 1 / (2 n) of an ulp from a number halfway between two doubles (n times such a number has more than 53 bits, so
// no x reaches it): the sum rounds as x / n does.
__device__ __forceinline__ double divided(double x, double n, double inv) {
  const double q = x * inv;
  return isfinite(q) ? fma(fma(-q, n, x), inv, q) : q;
}

template <int D> struct ShortSmem {
  static constexpr int tile = 2 * Geo<D>::stage_bytes;     // behind the rows, in place and gathered: codes [128 x D]
  static constexpr int red = tile + kBlock * D;            // 8 D floats
  static constexpr int part = red + 8 * D * 4;             // column sums or value maxima [D]
  static constexpr int pm = part + D * 4;                  // (m+, m-) pairs [D]
  static constexpr int qred = pm + D * 4;                  // [2][8] floats, the block's and the head's maximum
  static constexpr int src = qred + 80;                    // source rows [128]
  static constexpr int freq = src + kBlock * 4;            // [D / 2] doubles
  static constexpr int plain = freq + D / 2 * 8;           // the tables
  static constexpr size_t bytes(int entries) { return (size_t)plain + 16 * (size_t)entries; }
};

// Source of row t of a block: the gather by `perm` (clamped: never a bad address), -1 behind the last token.
__device__ __forceinline__ int source_row(const PrepArgs& a, const int32_t* perm, int blk, int t) {
  const int pos = blk * kBlock + t;
  return pos >= a.N ? -1 : (perm ? min(max(__ldg(perm + pos), 0), a.N - 1) : pos);
}
// 128 threads (t) copy the rows of a block; `mine` is the source of row t.  The lanes of a warp fetch its 32 rows 16 bytes at a time.
template <int D>
__device__ __forceinline__ void fetch_block(const PrepArgs& a, const char* head, int mine, int pitch, unsigned char* dst, int t) {
  constexpr int LPR = D / 8, RPI = 32 / LPR;
  const int lane = t & 31;
  dst += (t & ~31) * pitch + (lane / LPR) * pitch + 16 * (lane % LPR);
  head += 16 * (lane % LPR);
#pragma unroll
  for (int k = 0; k < 32 / RPI; ++k) {
    const int sr = __shfl_sync(0xffffffffu, mine, k * RPI + lane / LPR);
    if (sr >= 0) cp_async16(dst + k * RPI * pitch, head + (int64_t)sr * a.stride_n_bytes);
  }
}

template <int D, int BITS, int VARIANT>
__global__ void __launch_bounds__(kThreads, 2) prep_short_kernel(const PrepArgs a, const Short s) {
  using L = ShortSmem<D>;
  constexpr int kQuant = BITS == 4 ? kStageQuant4 : (VARIANT ? kStageQuant8I : kStageQuant8);
  constexpr int kRowBytes = BITS == 4 ? D / 2 : D;
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int group = blockIdx.x / a.nb, blk = blockIdx.x - group * a.nb;  // (a cluster is a group: blk is the rank in it)
  const int kind = group / a.BH, bh = group - kind * a.BH;
  const bool full = a.N - blk * kBlock >= kBlock;
  float* part = reinterpret_cast<float*>(smem + L::part);
  const int64_t head = head_offset_bytes(a, bh);
  const int32_t* perm = a.perm ? a.perm + (size_t)bh * a.N : nullptr;

  if (kind == kShortV) {
    unsigned int* amax = reinterpret_cast<unsigned int*>(part);
    float* red = reinterpret_cast<float*>(smem + kBlock * 2 * D);          // 16 D floats, behind the value tile
    if (tid < D) amax[tid] = 0u;
    pdl_wait();
    if (warp >= 4) {
      fetch_block<D>(a, reinterpret_cast<const char*>(a.v) + head, source_row(a, perm, blk, tid - 128), 2 * D, smem, tid - 128);
      cp_async_commit();
      cp_async_wait<0>();
    }
    __syncthreads();
    pdl_allow();
    const int cp = tid % (D / 2);
    float2 am = make_float2(0.f, 0.f), mu = am;
    if constexpr (BITS == 8) {
      if (full) v_stats_item<D, true>(a, smem, red, bh, blk, amax);
      else v_stats_item<D, false>(a, smem, red, bh, blk, amax);
      cluster_arrive();
      cluster_wait();
      mu = *reinterpret_cast<const float2*>(a.v_mu + ((size_t)bh * a.nb + blk) * D + 2 * cp);
      unsigned int m0 = 0u, m1 = 0u;
#pragma unroll
      for (int r = 0; r < kShortCluster; ++r) {
        if (r >= a.nb) break;
        m0 = max(m0, peer_word(amax + 2 * cp, r));
        m1 = max(m1, peer_word(amax + 2 * cp + 1, r));
      }
      cluster_arrive();                       // (this CTA has read its peers)
      am = make_float2(__uint_as_float(m0), __uint_as_float(m1));
      if (blk == 0 && tid < D / 2) *reinterpret_cast<uint2*>(a.v_amax + (size_t)bh * D + 2 * cp) = make_uint2(m0, m1);
    }
    if (blk == 0 && tid < D / 2)
      *reinterpret_cast<float2*>(a.v_scale + (size_t)bh * D + 2 * cp) = BITS == 8 ? make_float2(value_scale(am.x), value_scale(am.y)) : make_float2(1.0f, 1.0f);
    constexpr int kV = BITS == 8 ? kVQuant8 : (VARIANT ? kVQuant4M : kVQuant4);
    if (full) v_item<D, kV, true>(a, smem, red, bh, blk, mu, am);
    else v_item<D, kV, false>(a, smem, red, bh, blk, mu, am);
    if constexpr (BITS == 8) cluster_wait();  // a CTA stays until its peers have read it
    return;
  }

  // ---- Q and K: the tables (warps 0 to 3) while the rows are on their way (warps 4 to 7)
  const int tensor = kind == kShortK ? 1 : 0;
  const bool smooth = tensor == 1 && (a.flags & VC_FLAG_K_SMOOTH), gather = tensor == 1 && perm;
  unsigned char *in_place = smem, *gathered = gather ? smem + Geo<D>::stage_bytes : smem, *out_tile = smem + L::tile;
  float *red = reinterpret_cast<float*>(smem + L::red), *pm = reinterpret_cast<float*>(smem + L::pm), *qred = reinterpret_cast<float*>(smem + L::qred);
  unsigned int* amax = reinterpret_cast<unsigned int*>(qred + 16);
  int* src = reinterpret_cast<int*>(smem + L::src);
  float2 *plain = reinterpret_cast<float2*>(smem + L::plain), *folded = plain + a.rd.entries;
  double inv_n = 0.0;
  if (warp < 4) {
    double* freq = reinterpret_cast<double*>(smem + L::freq);
    if (tid < D / 2) {
      const int ax = tid >= a.rd.pair_start[2] ? 2 : (tid >= a.rd.pair_start[1] ? 1 : 0);
      freq[tid] = rope_freq(s.theta, tid - a.rd.pair_start[ax], a.rd.pairs[ax]);
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll 1
    for (int e = tid; e < a.rd.entries; e += 128) {
      const int ax = e >= a.rd.off[2] ? 2 : (e >= a.rd.off[1] ? 1 : 0);
      const int pos = (e - a.rd.off[ax]) / a.rd.pairs[ax], i = e - a.rd.off[ax] - pos * a.rd.pairs[ax];
      rope_entry_of(pos, freq[a.rd.pair_start[ax] + i], plain + e, folded + e);
    }
    if (tid < D) pm[tid] = 0.f;
    if (tid == 0) *amax = 0u;
    inv_n = 1.0 / s.n;
    pdl_wait();
  } else {
    pdl_wait();
    const char* x = reinterpret_cast<const char*>(tensor ? a.k : a.q) + head;
    const int t = tid - 128, from = source_row(a, tensor ? perm : nullptr, blk, t);      // (asked for first: the copies in place cover the round trip)
    if (!gather || smooth || BITS == 4) fetch_block<D>(a, x, source_row(a, nullptr, blk, t), Geo<D>::pitch, in_place, t);
    cp_async_commit();
    src[t] = from;
    if (gather) fetch_block<D>(a, x, from, Geo<D>::pitch, gathered, t);
    cp_async_commit();
    cp_async_wait<1>();
  }
  constexpr int LPR = D / 8, RPL = LPR / 2;   // (a lane's place in the column sums)
  const int lr = lane % LPR, hb = lane / LPR;
  const PairSlots ps = pair_slots(a.rd, 4 * lr);
  __syncthreads();
  pdl_allow();
  if (blockIdx.x == 0 && tid == 0) *s.status = 0u;

  const int my_row = qk_row_of(tid), row0 = warp * (32 / kTpr);
  auto none = [] { return (unsigned int*)nullptr; };   // (what a stage does not ask for)
  if (tensor == 1) {
    if (smooth) {
      const RopeTab tab{smem_u32(plain), nullptr};
      k_colsum_item<D>(a, in_place + (16 * warp + RPL * hb) * Geo<D>::pitch + 16 * lr, Geo<D>::pitch, red, tab, ps, part, blk);
    }
    cp_async_wait<0>();
    cluster_arrive();
    cluster_wait();
    if (tid < D) {                            // the sums of the head's blocks, as the finalization launch adds them
      double sum = 0.0;
      if (smooth) {
        float p[kShortCluster];               // (all asked for, then added)
#pragma unroll
        for (int j = 0; j < kShortCluster; ++j) p[j] = j < a.nb ? __uint_as_float(peer_word(part + tid, j)) : 0.f;
#pragma unroll
        for (int j = 0; j < kShortCluster; ++j) sum += (double)p[j];
      }
      red[tid] = (float)divided(sum, s.n, inv_n);
      if (blk == 0) a.k_mean[(size_t)bh * D + tid] = red[tid];
    }
    cluster_arrive();
    __syncthreads();
    if (smooth && tid < D / 2) *reinterpret_cast<float2*>(pm + 2 * tid) = make_float2(red[2 * tid] + red[2 * tid + 1], red[2 * tid] - red[2 * tid + 1]);
    __syncthreads();
    if constexpr (BITS == 4) cluster_wait();
  }
  if constexpr (BITS == 4) {                  // the head maximum, over the rows in place
    const int pos = blk * kBlock + my_row;
    qk_row_item_fast<D, kStageAmax>(a, tensor, in_place, out_tile, qred, pm, smem_u32(folded), bh, blk, 0, false, pos < a.N ? pos : -1, [&] { return amax; }, none);
    cluster_arrive();
    cluster_wait();
    const unsigned int most = __reduce_max_sync(0xffffffffu, lane < a.nb ? peer_word(amax, lane) : 0u);
    cluster_arrive();
    if (tid == 0) amax[1] = most;
    __syncthreads();
  }
  auto outer = [&] {
    const float g = outer_scale(__uint_as_float(amax[1]));
    if (tid == 0 && blk == 0) (tensor ? a.k_scale : a.q_scale)[bh] = g;
    return g;
  };
  qk_row_item_fast<D, kQuant>(a, tensor, gathered, out_tile, qred, pm, smem_u32(folded), bh, blk, 1, false, src[my_row], none, outer);
  __syncwarp();                               // the warp's rows of the code tile are complete
  store_warp_rows<kRowBytes>(tensor ? a.k_codes : a.q_codes, (size_t)bh * a.n_pad + (size_t)blk * kBlock, out_tile, row0, lane);
  if (BITS == 4 || tensor == 1) cluster_wait();       // a CTA stays until its peers have read it
}

// Which calls take it: heads of at most eight blocks whose CTAs are resident at once at 8 bits (two per SM), or in two
// waves at 4 bits, where one more launch falls away.  Up to there it is the faster form in every format, at both widths and behind a
// caller's kernel too.  At the line and beyond, one launch / a launch per phase (us, whole calls, d128): FP8 N1024 H12 (288 CTAs)
// 24.9 / 25.9, H15 (360) 26.6 / 27.6, H18 (432) 28.8 / 29.1 and behind a caller's kernel 30.0 / 29.0, H30 (720) 39.2 / 36.4; N576
// H24 (360) 24.7 / 26.3, H28 (420) 31.6 / 31.3; NVFP4 N1024 H18 38.4 / 39.8, H24 (576) 42.2 / 47.6, H30 (720) 47.1 / 49.3; d64 H24
// 32.4 / 37.2.  So at 8 bits the line is where heads of eight blocks still gain behind anything; shorter heads gain beyond it as well
// (N100 H240, 720 CTAs, 30.1 / 37.6), which the rule leaves.
inline bool short_heads(const Problem& pr, const PrepArgs& a) {
  return pr.nb <= kShortCluster && a.rd.entries <= kShortEntries && !(pr.flags & VC_FLAG_CHECK_PERM) && 3 * pr.BH * pr.nb <= (pr.bits == 8 ? 2 : 4) * sm_count();
}
template <int D, int BITS, int VARIANT>
cudaError_t run_short(const PrepArgs& a, const Short& s, cudaStream_t stream) {
  constexpr auto kernel = prep_short_kernel<D, BITS, VARIANT>;
  cudaError_t e = allow_smem<kernel>();
  if (e == cudaSuccess)
    e = launch_clusters(kernel, dim3((unsigned)(3 * a.BH * a.nb)), a.nb, kThreads, ShortSmem<D>::bytes(a.rd.entries), stream, a, s);
  if (e != cudaSuccess) return e;
  count_launches(1);
  return cudaGetLastError();
}
template <int D, int BITS>
cudaError_t run_short(const Problem& pr, const PrepArgs& a, const Short& s, cudaStream_t stream) {
  const bool variant = BITS == 8 ? (a.flags & VC_FLAG_INT8_QK) != 0 : hybrid4(pr);
  return variant ? run_short<D, BITS, 1>(a, s, stream) : run_short<D, BITS, 0>(a, s, stream);
}

// The packed row transform serves the standard configuration.
inline bool fast_rows(const PrepArgs& a) {
  return (a.flags & VC_FLAG_ROPE) && (a.flags & VC_FLAG_HADAMARD) && a.rope_default && a.rope_in_smem;
}

template <int D, int BITS>
cudaError_t run(const Problem& pr, const PrepArgs& a, cudaStream_t s) {
  const bool variant = BITS == 8 ? (a.flags & VC_FLAG_INT8_QK) != 0 : hybrid4(pr);
  if (fast_rows(a)) return variant ? run_phases<D, BITS, true, 1>(pr, a, s) : run_phases<D, BITS, true, 0>(pr, a, s);
  return variant ? run_phases<D, BITS, false, 1>(pr, a, s) : run_phases<D, BITS, false, 0>(pr, a, s);
}

}  // namespace

cudaError_t launch_prep(const Problem& pr, const QuantLayout& ql, const WorkLayout& wl,
                        const void* q, const void* k, const void* v, const int32_t* perm,
                        uint8_t* quant, uint8_t* work, cudaStream_t stream, const vc_prep_stats* stats, bool then_attention) {
  PrepArgs a{};
  a.q = (const __nv_bfloat16*)q; a.k = (const __nv_bfloat16*)k; a.v = (const __nv_bfloat16*)v;
  a.perm = perm;
  a.stride_b = pr.stride_b; a.stride_h = pr.stride_h; a.stride_n = pr.stride_n;
  a.stride_n_bytes = (int)(2 * pr.stride_n);
  a.mul_H = ((1ull << 40) + pr.H - 1) / pr.H;
  a.H = pr.H; a.N = pr.N; a.n_pad = pr.n_pad; a.nb = pr.nb; a.bh0 = 0; a.flags = pr.flags; a.BH = pr.BH;
  a.q_codes = quant + ql.q_codes; a.k_codes = quant + ql.k_codes; a.v_codes = quant + ql.v_codes;
  a.q_micro = quant + ql.q_micro; a.k_micro = quant + ql.k_micro; a.v_micro = quant + ql.v_micro;
  a.q_scale = (float*)(quant + ql.q_scale); a.k_scale = (float*)(quant + ql.k_scale);
  a.v_scale = (float*)(quant + ql.v_scale); a.k_mean = (float*)(quant + ql.k_mean);
  a.v_means = (__nv_bfloat16*)(quant + ql.v_means);
  a.rope = (const float2*)(work + wl.rope);
  a.k_part = (float*)(work + wl.k_part); a.v_mu = (float*)(work + wl.v_mu);
  a.v_amax = (unsigned int*)(work + wl.amax);
  a.qk_amax = a.v_amax + (size_t)pr.BH * pr.d;
  const bool ext = stats != nullptr;
  if (ext) {   // K mean, V block means and residual maxima as the caller computed them
    a.ext_k_mean = stats->k_mean;
    a.v_mu = const_cast<float*>(stats->v_block_mean);
    a.v_amax = reinterpret_cast<unsigned int*>(const_cast<float*>(stats->v_amax));
  }
  const int len[3] = {pr.grid_t, pr.grid_h, pr.grid_w};
  int ps = 0;
  for (int ax = 0; ax < 3; ++ax) {
    a.rd.pair_start[ax] = ps;
    a.rd.pairs[ax] = pr.rope_dim[ax] / 2;
    a.rd.off[ax] = wl.rope_off[ax];
    a.rd.len[ax] = len[ax];
    ps += pr.rope_dim[ax] / 2;
  }
  a.rd.entries = wl.rope_entries;
  a.rd.grid_h = pr.grid_h; a.rd.grid_w = pr.grid_w;
  a.rd.mul_w = ((1ull << 40) + pr.grid_w - 1) / pr.grid_w;
  a.rd.mul_h = ((1ull << 40) + pr.grid_h - 1) / pr.grid_h;
  a.rope_in_smem = (size_t)wl.rope_entries * 8 <= 96 * 1024;
  {
    const int sdef = 2 * (pr.d / 6);
    a.rope_default = pr.rope_dim[0] == pr.d - 2 * sdef && pr.rope_dim[1] == sdef && pr.rope_dim[2] == sdef;
  }
  if (then_attention && !ext && fast_rows(a) && short_heads(pr, a)) {
    const Short s{(double)pr.rope_theta, (double)pr.N, reinterpret_cast<unsigned int*>(work + wl.status)};
    if (pr.d == 128) return pr.bits == 8 ? run_short<128, 8>(pr, a, s, stream) : run_short<128, 4>(pr, a, s, stream);
    return pr.bits == 8 ? run_short<64, 8>(pr, a, s, stream) : run_short<64, 4>(pr, a, s, stream);
  }
  // the table (one thread per entry), the words that start at zero, supplied statistics
  SetUp u{};
  u.status = reinterpret_cast<unsigned int*>(work + wl.status);
  if (ext) {
    u.n_ext = pr.BH * pr.d;
    u.ext_k_mean = (pr.flags & VC_FLAG_K_SMOOTH) ? stats->k_mean : nullptr;
    u.ext_v_amax = stats->v_amax;
    u.k_mean = a.k_mean;
    u.v_scale = a.v_scale;
  } else {
    u.zero = reinterpret_cast<unsigned int*>(work + wl.amax);
    u.n_zero = (int)(wl.amax_bytes / 4);
  }
  RopeDesc rd = a.rd;
  if (!(a.flags & VC_FLAG_ROPE)) rd.entries = 0;
  const int words = (u.n_zero + u.n_ext + 3) / 4, need = rd.entries > words ? rd.entries : words;
  cudaError_t e = launch_overlapped(rope_table_kernel, dim3((unsigned)(need / 64 + 1)), 64, 0, stream, reinterpret_cast<float2*>(work + wl.rope), rd,
                                    (double)pr.rope_theta, u);
  if (e != cudaSuccess) return e;
  count_launches(1);
  if ((e = launch_perm_check(pr, perm, wl, work, stream)) != cudaSuccess) return e;
  if (pr.d == 128) return pr.bits == 8 ? run<128, 8>(pr, a, stream) : run<128, 4>(pr, a, stream);
  return pr.bits == 8 ? run<64, 8>(pr, a, stream) : run<64, 4>(pr, a, stream);
}

}  // namespace vc

// ---------------------------------------------------------------------------------------
// vc_prep_noalloc: the preprocessing pass for callers that cannot provide a workspace.
// The scratch that vc_prep takes from the caller (RoPE tables, per-block partial sums, block
// means, amax words) lives here in a fixed array in device global memory, so the call needs no
// allocation of any kind; the price is a size limit and one array per GPU for the life of the
// process.
namespace {

// Held by every GPU that loads this library until the process exits.
static __device__ __align__(256) unsigned char g_prep_scratch[VC_NOALLOC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
unsigned char* g_scratch_addr[kMaxDevices] = {};   // device address of the array, per device

// In host code the array's name is only a handle; the device address has to be asked for,
// once per device, with that device current.
cudaError_t scratch_address(unsigned char** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  unsigned char* ptr = __atomic_load_n(&g_scratch_addr[dev], __ATOMIC_ACQUIRE);
  if (!ptr) {
    e = cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_prep_scratch);
    if (e != cudaSuccess) return e;
    __atomic_store_n(&g_scratch_addr[dev], ptr, __ATOMIC_RELEASE);   // same value from any thread
  }
  *out = ptr;
  return cudaSuccess;
}

}  // namespace

extern "C" vc_status vc_prep_noalloc(const vc_params* p, const void* q, const void* k, const void* v,
                                     const int32_t* perm, void* quant, void* stream) {
  vc::Problem pr;
  vc_status st = vc::resolve(p, &pr);
  if (st != VC_OK) return st;
  if (!q || !k || !v || !quant) return VC_ERR_INVALID_ARG;
  if (((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)quant | (uintptr_t)perm) & 15) return VC_ERR_INVALID_ARG;
  const vc::QuantLayout ql = vc::quant_layout(pr);
  const vc::WorkLayout wl = vc::work_layout(pr);
  if (wl.prep_end > (size_t)VC_NOALLOC_SCRATCH_BYTES) return VC_ERR_SCRATCH_LIMIT;
  unsigned char* scratch = nullptr;
  if (scratch_address(&scratch) != cudaSuccess) return VC_ERR_CUDA;
  // launch_prep clears the words that must start at zero (status, amax) on the stream itself
  cudaError_t e = vc::launch_prep(pr, ql, wl, q, k, v, perm, (uint8_t*)quant, scratch, (cudaStream_t)stream, nullptr, false);
  return e == cudaSuccess ? VC_OK : VC_ERR_CUDA;
}

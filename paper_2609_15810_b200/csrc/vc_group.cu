// Token grouping of VC-Attention for sm_100a (Sec. 3.2 "Value-guided permutation"): for every
// (batch, head) a k-means over the value tokens gives each token a label z_t, and the
// permutation handed to the preprocessing pass is pi = argsort(z), stable, so that every
// cluster becomes one contiguous run of key/value rows (Eq. 3).
//
// The paper fixes neither k nor the initialisation nor the iteration count ("lightweight
// online k-means", warm-started from the previous step's centroids).  This build takes plain
// Lloyd iterations: squared Euclidean distance on the fp32 value rows, centroids started at
// every (N / k)-th token unless warm-started, an empty cluster keeps its centroid, ties go to
// the lower cluster index, and the sort keeps token order inside a cluster.
//
// Everything is deterministic: no floating-point atomics.  A CTA owns a chunk of 1024
// consecutive tokens of one head and forms its per-cluster sums on the tensor core (fixed
// hardware order); a second kernel adds the chunks' partial sums in chunk order.
//
//   group_init_kernel     status word; centroids <- rows 0, N/k, 2 N/k, ... (cold start)
//   group_assign_kernel   labels, per-chunk cluster sums and counts      (once per iteration;
//                         distances on the tensor cores, see the kernel)
//   group_update_kernel   centroids <- sum of partial sums / counts      (once per iteration);
//                         behind the last one also the start of every (cluster, chunk) run in pi
//   group_scatter_kernel  pi: tokens of a chunk in order, behind their cluster's run
#include <cuda_bf16.h>

#include "vc_attn_shared.cuh"
#include "vc_internal.h"
#include "vc_launch.h"
#include "vc_sm100.cuh"

namespace vc {
namespace {

using namespace sm100;

constexpr int kGroupK = 64;          // clusters the kernels are laid out for (k <= 64)
constexpr int kChunkTiles = 8;       // 128-token tiles per chunk
constexpr int kChunk = kChunkTiles * kBlock;

struct GroupArgs {
  const __nv_bfloat16* v;
  int64_t stride_b, stride_h, stride_n;
  int H, N, k, chunks, all_chunks;   // chunks per head; of all heads
  float* centroids;      // [BH][k][D]
  int32_t* labels;       // [BH][N]
  float* psum;           // [BH][chunks][kGroupK][D]
  int32_t* counts;       // [BH][chunks][kGroupK]
  int32_t* offsets;      // [BH][chunks][kGroupK]
  int32_t* perm;         // [BH][N]
  uint32_t* status;      // status word (first word of the workspace)
  uint32_t wait_limit;   // polls after which a wait gives up
  uint32_t nonblocking;  // test hook: polls test the barrier without sleeping in hardware
};

template <int D>
__global__ void group_init_kernel(const GroupArgs a, int warm) {
  pdl_wait();
  pdl_allow();
  const int bh = blockIdx.y, j = blockIdx.x, c = threadIdx.x;
  if (bh == 0 && j == 0 && c == 0) *a.status = 0u;
  if (warm) return;
  const int b = bh / a.H, h = bh - b * a.H;
  const int step = a.N / a.k > 0 ? a.N / a.k : 1;
  const __nv_bfloat16* row = a.v + b * a.stride_b + h * a.stride_h + (int64_t)(j * step) * a.stride_n;
  if (c < D) a.centroids[((size_t)bh * a.k + j) * D + c] = __bfloat162float(row[c]);
}

// Assignment step on the tensor cores.  The scores v . c of a 128-token tile against the 64
// centroids are a 128 x 64 x d contraction: the value tile arrives by TMA as the bf16 A operand
// (exact: V is bf16), the fp32 centroids are split into three bf16 terms c = c_hi + c_mid + c_lo
// (8 + 8 + 8 mantissa bits, exact), and 3 x d/16 kind::f16 MMAs accumulate every product in FP32
// tensor memory.  label = argmin_c |c|^2 - 2 v.c  (|v|^2 is the same for every c), ties to the
// lower index.  The cluster sums are a contraction too: sums[64 x d] += onehot^T[64 x 128] V[128 x d],
// with the one-hot matrix of the tile's labels written by the token threads (one bf16 1.0 each) and
// the SAME value tile as the B operand, read MN-major (channels contiguous).  Products are exact
// and the accumulation order is the hardware's fixed one: deterministic, no atomics on floats.
//
// A CTA takes a run of consecutive chunks, so the centroids are split and laid out once per head it
// meets instead of once per chunk, and loads, products and labels run on from chunk to chunk.
//   warp 8      MMA issue (the issuing thread is held up while the tensor pipe's queue is full, so
//               nothing else may wait for it)
//   warp 9      TMA loads of the value tiles (4-stage ring)
//   warps 0-3   even tiles, warps 4-7 odd tiles of the run, one thread per token: scores from tensor
//               memory, argmin, label, one-hot entry; the warpgroup that had a chunk's last tile
//               writes the chunk's sums and counts out
// Tensor memory: two score buffers of 64 columns | two cluster-sum buffers (d columns, rows = clusters).
// What bounds it: at B1 H40 N32760 d128 it takes 125 us, about 3550 cycles per tile (190 us with a CTA per chunk, one
// label warpgroup and serial minima).  2176 of them are the products: 24 for the scores, 64 cycles each, as long as
// the A operand takes to read however few the centroids, and 8 of 80 for the sums; alone they would take 77 us.  Where
// the rest goes (hand-offs, chunk ends, a head's set-up) has not been measured.  The values at the copy rate: 51 us.
constexpr int kGStages = 4;
constexpr int kGThreads = 320;
constexpr uint32_t kGroupWaitLimit = 1u << 22;   // default number of polls of a wait

struct GroupSmem {
  uint64_t v_full[kGStages], v_free[kGStages], s_full[2], s_free[2], oh_full, oh_free, sum_done[2], sum_free[2];
  uint64_t drain;        // exit: "every MMA of the control warp has completed"
  alignas(16) float cnorm[kGroupK];
  int count[4][kGroupK]; // by chunk of the run, modulo 4: a warpgroup may be three tiles ahead of the other
  uint32_t tmem_base;
  int prev[kBlock];      // row of the one in every column of the one-hot tile, -1 none
  int abort;
};

// Bounded wait of a whole warp (see warp_wait2).  When it gives up, the labels of this run are garbage
// (but in range), its chunks count no tokens, positions that come of it are dropped outside [0, N), and the
// status word says so: vc_poll_status on the workspace returns VC_ERR_TIMEOUT.
__device__ __forceinline__ bool gwait(uint64_t* bar, uint32_t parity, GroupSmem* sh, const GroupArgs& a) {
  if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return true;
  if (!a.nonblocking) {
#pragma unroll 1
    for (uint32_t i = 0; i < a.wait_limit; ++i) {
      if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
      if ((i & 255u) == 255u && __any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&sh->abort))) return false;
    }
  } else {
#pragma unroll 1
    for (uint32_t i = 0; i < a.wait_limit; ++i) {
      if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return true;
      if ((i & 255u) == 255u && __any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&sh->abort))) return false;
    }
  }
  *reinterpret_cast<volatile int*>(&sh->abort) = 1;
  atomicExch(a.status, kStatusTimeout | 0x60u);
  return false;
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* m, uint64_t* bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}

// Shared-memory descriptor of an MN-major operand in the 128-byte swizzle: rows of 128 bytes hold
// 64 consecutive M/N elements of one k; 8 k-rows form a 1024-byte group (stride offset), the next
// 64 M/N elements start `mn_block_bytes` further (leading offset).
__device__ __forceinline__ uint64_t smem_desc_mnmajor(uint32_t saddr, uint32_t mn_block_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)(mn_block_bytes >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// A position in a CTA's run of chunks, tile by tile.
struct RunPos {
  int c, bh, chunk, tile, n_tiles;   // chunk over all heads; its head and number there; tile and tiles in it
};
__device__ __forceinline__ void at_chunk(RunPos& r, const GroupArgs& a, int c) {
  r.c = c;
  r.bh = c / a.chunks;
  r.chunk = c - r.bh * a.chunks;
  r.tile = 0;
  r.n_tiles = min(kChunkTiles, (a.N + kBlock - 1) / kBlock - r.chunk * kChunkTiles);
}
__device__ __forceinline__ void next_tile(RunPos& r, const GroupArgs& a) {
  if (++r.tile == r.n_tiles) at_chunk(r, a, r.c + 1);
}

constexpr int kSetUp = 288;              // threads that lay out a head's centroids (all but the loading warp)
__device__ __forceinline__ void set_up_barrier() { asm volatile("bar.sync 1, 288;" ::: "memory"); }

template <int D>
__global__ void __launch_bounds__(kGThreads, 1) group_assign_kernel(const __grid_constant__ CUtensorMap tm_v, const GroupArgs a) {
  constexpr int KH = D / 64;                        // 128-byte column halves of a bf16 tile
  constexpr uint32_t kVHalf = kBlock * 128, kVStage = KH * kVHalf;       // value tile: [KH][128 tokens][128 B]
  constexpr uint32_t kCHalf = kGroupK * 128, kCSplit = KH * kCHalf;      // centroid term: [KH][64 rows][128 B]
  constexpr uint32_t kOhHalf = 128 * 128, kOhBytes = 2 * kOhHalf;        // one-hot^T: [2][128 rows][64 tokens]
  constexpr uint32_t SUM_COL = 128;
  constexpr int kTmemCols = 512;
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* sV = smem;                                          // [kGStages] value tiles
  unsigned char* sC = sV + kGStages * kVStage;                       // [3] centroid terms
  unsigned char* sOh = sC + 3 * kCSplit;                             // one-hot^T of a tile's labels
  GroupSmem* sh = reinterpret_cast<GroupSmem*>(sOh + kOhBytes);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int per = a.all_chunks / (int)gridDim.x, more = a.all_chunks % (int)gridDim.x, b0 = blockIdx.x;
  const int c_begin = b0 * per + min(b0, more), c_end = c_begin + per + (b0 < more ? 1 : 0);

  if (tid == 0) {
    for (int i = 0; i < kGStages; ++i) { mbar_init(&sh->v_full[i], 1); mbar_init(&sh->v_free[i], 1); }
    mbar_init(&sh->oh_full, 128); mbar_init(&sh->oh_free, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh->s_full[i], 1); mbar_init(&sh->s_free[i], 4);
      mbar_init(&sh->sum_done[i], 1); mbar_init(&sh->sum_free[i], 2);
    }
    mbar_init(&sh->drain, 1);
    sh->abort = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tm_v);
  }
  for (int i = tid; i < (int)kOhBytes / 16; i += kGThreads) reinterpret_cast<uint4*>(sOh)[i] = make_uint4(0, 0, 0, 0);
  if (tid < 128) sh->prev[tid] = -1;
  if (tid < 4 * kGroupK) sh->count[tid / kGroupK][tid % kGroupK] = 0;
  if (warp == 8) { tmem_alloc<kTmemCols>(&sh->tmem_base); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // Behind the allocation (the next kernel may want tensor memory too) but in front of this kernel's own wait: the
  // kernel launched next, the update, must touch no global memory before its own.  (Behind the wait a warm
  // iteration at B1 H40 N32760 d128 takes 161 us instead of 157: the loading warp comes there last.)
  pdl_allow();
  const uint32_t tmem = sh->tmem_base;

  RunPos pos;                          // every role's own position in the run
  at_chunk(pos, a, c_begin);
  int g = 0, q = 0;                    // tiles and chunks of the run behind us
  bool ok = true;                      // false after a wait that gave up: no more waits, loads or products

  const uint32_t idesc_s = idesc_bf16(128, kGroupK);
  const uint32_t idesc_sum = idesc_bf16(128, D) | (1u << 16);        // B operand MN-major
  // operand descriptors (addresses in 16-byte units advance by additions)
  const uint64_t dv0 = smem_desc_kmajor(smem_u32(sV), 128), dc0 = smem_desc_kmajor(smem_u32(sC), 128);
  const uint64_t dvb0 = smem_desc_mnmajor(smem_u32(sV), kVHalf), doh0 = smem_desc_kmajor(smem_u32(sOh), 128);
  auto scores = [&](int i) {           // S[i % 2] = V_i C^T, three centroid terms
    const int st = i % kGStages, sb = i & 1;
    if (!ok || !(ok = gwait(&sh->v_full[st], (i / kGStages) & 1, sh, a))) return;
    if (i >= 2 && !(ok = gwait(&sh->s_free[sb], ((i >> 1) - 1) & 1, sh, a))) return;
    if (elect_one()) {
      tc_fence_after();
      const uint64_t dv = dv0 + (uint64_t)(st * (kVStage >> 4));
#pragma unroll
      for (int t = 0; t < 3; ++t)
#pragma unroll
        for (int kh = 0; kh < KH; ++kh)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_f16_ss(tmem + 64 * sb, dv + (kh * (kVHalf >> 4) + 2 * k), dc0 + (t * (kCSplit >> 4) + kh * (kCHalf >> 4) + 2 * k), idesc_s, (t | kh | k) != 0);
      mma_commit(&sh->s_full[sb]);
    }
    __syncwarp();
  };
  if (warp == 9) {
    // -------------------------------------------------------------------- loads, across chunks and heads
    // (the values are the caller's: they need not wait for the kernel in front)
    int loaded = 0;
    for (; pos.c < c_end; next_tile(pos, a), ++loaded) {
      const int st = loaded % kGStages;
      if (loaded >= kGStages && !gwait(&sh->v_free[st], (loaded / kGStages - 1) & 1, sh, a)) break;
      if (elect_one()) {
        const int b = pos.bh / a.H, h = pos.bh - b * a.H;
        mbar_expect_tx(&sh->v_full[st], kVStage);
        for (int kh = 0; kh < KH; ++kh)
          tma_load_4d(sV + st * kVStage + kh * kVHalf, &tm_v, &sh->v_full[st], 128 * kh, (pos.chunk * kChunkTiles + pos.tile) * kBlock, h, b);
      }
      __syncwarp();
    }
    // Nothing this CTA started may outlive it (shared and tensor memory are released at exit, also
    // after a wait gave up): wait for the copies nobody consumed; the MMA warp does the same.
    for (int jj = loaded > kGStages ? loaded - kGStages : 0; jj < loaded; ++jj)
      mbar_wait(&sh->v_full[jj % kGStages], (jj / kGStages) & 1, 1u << 22);
    pos.c = c_end;                     // (no part in the loop below)
  }
  pdl_wait();

  // ---- label warpgroups
  const int wg = warp >> 2, wtid = tid & 127;          // (warp 8: unused)
  const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  // my column of the one-hot^T tile: token wtid, 2 bytes inside a 16-byte chunk of row `label`
  unsigned char* oh = sOh + (wtid >> 6) * kOhHalf + (((wtid & 63) * 2) & 15);
  const int oh_chunk = ((wtid & 63) * 2) >> 4;

  while (pos.c < c_end) {
    // ---- the chunks of one head: centroids -> three bf16 terms in the swizzled K-major operand layout
    // (zero rows beyond k), squared norms.  Every score product of the previous head has been read.
    const int bh = pos.bh, head_end = min(c_end, (bh + 1) * a.chunks);
    set_up_barrier();
    for (int i = tid; i < kGroupK * (D / 8); i += kSetUp) {
      const int j = i / (D / 8), oct = i % (D / 8);      // centroid j, channels 8 oct .. 8 oct + 7
      float c[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (j < a.k) {
        const float4* src = reinterpret_cast<const float4*>(a.centroids + ((size_t)bh * a.k + j) * D + 8 * oct);
        const float4 lo = src[0], hi = src[1];
        c[0] = lo.x; c[1] = lo.y; c[2] = lo.z; c[3] = lo.w; c[4] = hi.x; c[5] = hi.y; c[6] = hi.z; c[7] = hi.w;
      }
      uint32_t w[3][4];
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        float r0 = c[e], r1 = c[e + 1];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          const __nv_bfloat162 p2 = __floats2bfloat162_rn(r0, r1);
          w[t][e >> 1] = *reinterpret_cast<const uint32_t*>(&p2);
          r0 -= __low2float(p2);
          r1 -= __high2float(p2);
        }
      }
      const int half = oct / 8, chunk16 = oct % 8;
      const uint32_t off = half * kCHalf + j * 128 + ((chunk16 ^ (j & 7)) << 4);
#pragma unroll
      for (int t = 0; t < 3; ++t) *reinterpret_cast<uint4*>(sC + t * kCSplit + off) = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
    }
    if (tid < kGroupK) {
      float s = INFINITY;                              // an infinite norm keeps the rows beyond k from ever winning
      if (tid < a.k) {
        // (sixteen loads at a time, then the squares in channel order)
        const float4* src = reinterpret_cast<const float4*>(a.centroids + ((size_t)bh * a.k + tid) * D);
        s = 0.f;
#pragma unroll 1
        for (int q0 = 0; q0 < D / 4; q0 += 16) {
          float4 c4[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) c4[e] = src[q0 + e];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            s = fmaf(c4[e].x, c4[e].x, s); s = fmaf(c4[e].y, c4[e].y, s);
            s = fmaf(c4[e].z, c4[e].z, s); s = fmaf(c4[e].w, c4[e].w, s);
          }
        }
      }
      sh->cnorm[tid] = s;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy stores -> tensor-core reads
    set_up_barrier();

    if (warp == 8) {
      // ---------------------------------------------------------------- MMA issue
      scores(g);
      while (pos.c < head_end) {
        const int st = g % kGStages;
        const bool first = pos.tile == 0, last = pos.tile + 1 == pos.n_tiles;
        if (!(last && pos.c + 1 == head_end)) scores(g + 1);           // scores run one tile ahead of the sums
        ok = ok && gwait(&sh->oh_full, g & 1, sh, a);
        if (ok && first && q >= 2) ok = gwait(&sh->sum_free[q & 1], ((q >> 1) - 1) & 1, sh, a);
        if (ok && elect_one()) {
          tc_fence_after();
          // sums += onehot^T (K-major, 128 tokens = two 64-token halves) x V_g (MN-major: 16 tokens = 2048 bytes per step)
          const uint64_t dvb = dvb0 + (uint64_t)(st * (kVStage >> 4));
          const uint32_t sum = tmem + SUM_COL + 128 * (q & 1);
#pragma unroll
          for (int half = 0; half < 2; ++half)
#pragma unroll
            for (int k = 0; k < 4; ++k)
              mma_f16_ss(sum, doh0 + (half * (kOhHalf >> 4) + 2 * k), dvb + 128 * (4 * half + k), idesc_sum, (!first) | (half > 0) | (k > 0));
          mma_commit(&sh->oh_free);
          mma_commit(&sh->v_free[st]);
          if (last) mma_commit(&sh->sum_done[q & 1]);
        }
        __syncwarp();
        ++g;
        if (last) ++q;
        next_tile(pos, a);
      }
    } else {
      // ---------------------------------------------------------------- labels and one-hot entries
      const uint64_t* cn = reinterpret_cast<const uint64_t*>(sh->cnorm);
      const uint64_t m2 = pack_f32x2(-2.0f, -2.0f);
      for (; pos.c < head_end; ++g, next_tile(pos, a)) {
        const bool last = pos.tile + 1 == pos.n_tiles;
        if ((g & 1) == wg) {
          const int t0 = (pos.chunk * kChunkTiles + pos.tile) * kBlock;
          ok = ok && gwait(&sh->s_full[wg], (g >> 1) & 1, sh, a);
          tc_fence_after();
          uint32_t s0[32], s1[32];
          tmem_ld32(lane_base + 64 * wg, s0);
          tmem_ld32(lane_base + 64 * wg + 32, s1);
          tmem_wait_ld();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh->s_free[wg]);
          // argmin of |c|^2 - 2 v.c over four runs of 16 clusters side by side; ties to the lower index
          float best[4];
          int arg[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) { best[r] = INFINITY; arg[r] = 0; }
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const int j = 16 * r + i;
              const uint64_t pair = j < 32 ? pack_b32x2(s0[j & 31], s0[(j & 31) + 1]) : pack_b32x2(s1[j & 31], s1[(j & 31) + 1]);
              float d0, d1;
              unpack2(fma2(pair, m2, cn[j >> 1]), d0, d1);
              if (d0 < best[r]) { best[r] = d0; arg[r] = j; }
              if (d1 < best[r]) { best[r] = d1; arg[r] = j + 1; }
            }
          }
          if (best[1] < best[0]) { best[0] = best[1]; arg[0] = arg[1]; }
          if (best[3] < best[2]) { best[2] = best[3]; arg[2] = arg[3]; }
          const int label = best[2] < best[0] ? arg[2] : arg[0];
          const bool valid = t0 + wtid < a.N;
          if (valid) {
            a.labels[(size_t)bh * a.N + t0 + wtid] = label;
            atomicAdd(&sh->count[q & 3][label], 1);
          }
          // the sums of the previous tile must have read the one-hot tile before it changes
          if (g >= 1) ok = ok && gwait(&sh->oh_free, (g - 1) & 1, sh, a);
          const int prev = sh->prev[wtid];               // the entry the other warpgroup left in my column
          if (prev >= 0) *reinterpret_cast<unsigned short*>(oh + prev * 128 + ((oh_chunk ^ (prev & 7)) << 4)) = 0;
          sh->prev[wtid] = valid ? label : -1;
          if (valid) *reinterpret_cast<unsigned short*>(oh + label * 128 + ((oh_chunk ^ (label & 7)) << 4)) = 0x3f80;   // bf16 1.0
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_arrive(&sh->oh_full);
          // ---- the chunk's cluster sums: row = cluster (lanes 0..63 of tensor memory), d columns
          if (last && (warp & 3) < 2) {
            ok = ok && gwait(&sh->sum_done[q & 1], (q >> 1) & 1, sh, a);
            tc_fence_after();
            const size_t at = (size_t)bh * a.chunks + pos.chunk;
            float* dst = a.psum + (at * kGroupK + wtid) * D;
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
              uint32_t r[32];
              tmem_ld32(lane_base + SUM_COL + 128 * (q & 1) + 32 * c, r);
              tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 8; ++e)
                reinterpret_cast<uint4*>(dst + 32 * c)[e] = make_uint4(r[4 * e], r[4 * e + 1], r[4 * e + 2], r[4 * e + 3]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->sum_free[q & 1]);
            // (a run that has given up reports no tokens: the other warpgroup may be anywhere, and what it adds to
            // this slot from here on would be counted for a later chunk)
            a.counts[at * kGroupK + wtid] = ok ? sh->count[q & 3][wtid] : 0;
            sh->count[q & 3][wtid] = 0;
          }
        }
        if (last) ++q;
      }
    }
  }
  if (warp == 8) {
    if (elect_one()) mma_commit(&sh->drain);
    __syncwarp();
    mbar_wait(&sh->drain, 0, 1u << 22);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) tmem_dealloc<kTmemCols>(tmem);
}

// Blocks j < k: centroid <- (sum over chunks, in chunk order) / count, a thread per channel with 32 partial
// sums in flight; an empty cluster keeps its centroid.  (Four channels per thread leave too few loads in
// flight: 24 us instead of 15 at B1 H40 N32760 d128, 42 MB of partial sums out of L2.)
// The last block, if it is there (behind the last iteration): offsets[chunk][label] = tokens with a
// smaller label + tokens of this label in earlier chunks.
template <int D>
__global__ void __launch_bounds__(D) group_update_kernel(const GroupArgs a) {
  const int bh = blockIdx.y, j = blockIdx.x, c = threadIdx.x;
  __shared__ int total[kGroupK], start[kGroupK];
  pdl_wait();
  pdl_allow();
  if (j < a.k) {
    const float* src = a.psum + ((size_t)bh * a.chunks * kGroupK + j) * D + c;
    const int32_t* cnt = a.counts + (size_t)bh * a.chunks * kGroupK + j;
    int n = 0;
    for (int ch = c & 31; ch < a.chunks; ch += 32) n += cnt[ch * kGroupK];
    float s = 0.f;
#pragma unroll 32
    for (int ch = 0; ch < a.chunks; ++ch) s += src[(size_t)ch * (kGroupK * D)];
    n = __reduce_add_sync(0xffffffffu, n);
    if (n > 0) a.centroids[((size_t)bh * a.k + j) * D + c] = s / (float)n;
    return;
  }
  const bool mine = c < kGroupK;                // one thread per label
  const int32_t* counts = a.counts + (size_t)bh * a.chunks * kGroupK + (mine ? c : 0);
  if (mine) {
    int n = 0;
#pragma unroll 8
    for (int ch = 0; ch < a.chunks; ++ch) n += counts[ch * kGroupK];
    total[c] = n;
  }
  __syncthreads();
  if (c == 0) {
    int run = 0;
    for (int l = 0; l < kGroupK; ++l) { start[l] = run; run += total[l]; }
  }
  __syncthreads();
  if (!mine) return;
  int run = start[c];
#pragma unroll 8
  for (int ch = 0; ch < a.chunks; ++ch) {
    a.offsets[((size_t)bh * a.chunks + ch) * kGroupK + c] = run;
    run += counts[ch * kGroupK];
  }
}

// A block per chunk, a warp per 128 of its tokens.  A label's tokens go behind its tokens in earlier warps
// (counted first); a warp walks its tokens in order, 32 at a time: a token goes behind the tokens of
// its label seen so far, and among the 32 of a step behind the lower lanes with the same label.
// (One warp walking all 32 steps of a chunk: 22 us instead of 12 at B1 H40 N32760.)
constexpr int kScatterWarps = kChunk / 128;
__global__ void __launch_bounds__(32 * kScatterWarps) group_scatter_kernel(const GroupArgs a) {
  const int chunk = blockIdx.x, bh = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ int next[kScatterWarps][kGroupK];
  for (int i = tid; i < kScatterWarps * kGroupK; i += 32 * kScatterWarps) (&next[0][0])[i] = 0;
  pdl_wait();
  pdl_allow();
  const int t_first = chunk * kChunk + warp * 128, t_end = min(a.N, (chunk + 1) * kChunk);
  int labs[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int t = t_first + 32 * i + lane;
    labs[i] = t < t_end ? a.labels[(size_t)bh * a.N + t] : -1 - lane;   // distinct dummies never match
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (labs[i] >= 0) atomicAdd(&next[warp][labs[i]], 1);
  __syncthreads();
  if (tid < kGroupK) {                       // counts -> first positions
    int run = a.offsets[((size_t)bh * a.chunks + chunk) * kGroupK + tid];
#pragma unroll
    for (int w = 0; w < kScatterWarps; ++w) {
      const int n = next[w][tid];
      next[w][tid] = run;
      run += n;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int lab = labs[i];
    const bool valid = lab >= 0;
    const unsigned int same = __match_any_sync(0xffffffffu, lab);
    const int rank = __popc(same & ((1u << lane) - 1u));
    int basepos = 0;
    if (valid) basepos = next[warp][lab];
    __syncwarp();
    if (valid) {
      // (after a wait that gave up the counts need not add up; they must not become an address for all that)
      const int at = basepos + rank;
      if ((unsigned)at < (unsigned)a.N) a.perm[(size_t)bh * a.N + at] = t_first + 32 * i + lane;
      if (rank == __popc(same) - 1) next[warp][lab] = basepos + rank + 1;     // the last of its group moves the cursor
    }
    __syncwarp();
  }
}

// 4-D byte tensor [B][H][N][2 d] with the caller's strides, box {128 bytes, 128 rows}, 128-byte swizzle.
bool make_value_map(CUtensorMap* m, const Problem& pr, const void* v) {
  attn::EncodeTiledFn fn = attn::encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)pr.d * 2, (cuuint64_t)pr.N, (cuuint64_t)pr.H, (cuuint64_t)pr.B};
  const cuuint64_t strides[3] = {(cuuint64_t)pr.stride_n * 2, (cuuint64_t)pr.stride_h * 2, (cuuint64_t)pr.stride_b * 2};
  const cuuint32_t box[4] = {128, 128, 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(v), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D>
cudaError_t run_group(const Problem& pr, GroupArgs a, int iters, int warm, cudaStream_t s) {
  constexpr size_t smem = (size_t)kGStages * kBlock * D * 2 + 3 * (size_t)kGroupK * D * 2 + 2 * 128 * 128 + sizeof(GroupSmem);
  static_assert(smem <= 227 * 1024, "shared memory of the assignment kernel exceeds the SM");
  alignas(64) CUtensorMap tm_v;
  if (!make_value_map(&tm_v, pr, a.v)) return cudaErrorUnknown;
  a.all_chunks = a.chunks * pr.BH;
  const int sms = sm_count(), grid = a.all_chunks < sms ? a.all_chunks : sms;
  cudaError_t e = allow_smem<group_assign_kernel<D>>();
  if (e == cudaSuccess) e = launch_overlapped(group_init_kernel<D>, warm ? dim3(1, 1) : dim3(a.k, pr.BH), D, 0, s, a, warm);
  for (int it = 0; it < iters && e == cudaSuccess; ++it) {
    e = launch_overlapped(group_assign_kernel<D>, dim3(grid), kGThreads, smem, s, tm_v, a);
    if (e == cudaSuccess) e = launch_overlapped(group_update_kernel<D>, dim3(a.k + (it + 1 == iters ? 1 : 0), pr.BH), D, 0, s, a);
    count_launches(2);
  }
  if (e == cudaSuccess) e = launch_overlapped(group_scatter_kernel, dim3(a.chunks, pr.BH), 32 * kScatterWarps, 0, s, a);
  count_launches(2);
  return e != cudaSuccess ? e : cudaGetLastError();
}

struct GroupLayout {
  size_t status, labels, psum, counts, offsets, total;
  int chunks;
};
GroupLayout group_layout(const Problem& pr) {
  GroupLayout g{};
  g.chunks = (pr.N + kChunk - 1) / kChunk;
  size_t off = 0;
  auto place = [&](size_t bytes) { size_t o = off; off = (off + bytes + 1023) / 1024 * 1024; return o; };
  g.status = place(VC_GROUP_LABELS_OFFSET);          // the status word, then the labels
  g.labels = place((size_t)pr.BH * pr.N * 4);
  g.psum = place((size_t)pr.BH * g.chunks * kGroupK * pr.d * 4);
  g.counts = place((size_t)pr.BH * g.chunks * kGroupK * 4);
  g.offsets = place((size_t)pr.BH * g.chunks * kGroupK * 4);
  g.total = off;
  return g;
}

}  // namespace
}  // namespace vc

using namespace vc;

extern "C" size_t vc_group_workspace_bytes(const vc_params* p) {
  Problem pr;
  if (resolve(p, &pr) != VC_OK) return 0;
  return group_layout(pr).total;
}

extern "C" vc_status vc_group(const vc_params* p, const void* v, int32_t k, int32_t iters, int32_t warm_start,
                              float* centroids, int32_t* perm, void* workspace, void* stream) {
  Problem pr;
  vc_status st = resolve(p, &pr);
  if (st != VC_OK) return st;
  if (!v || !centroids || !perm || !workspace) return VC_ERR_INVALID_ARG;
  if (((uintptr_t)v | (uintptr_t)centroids | (uintptr_t)perm | (uintptr_t)workspace) & 15) return VC_ERR_INVALID_ARG;
  if (k < 1 || iters < 1 || k > pr.N) return VC_ERR_INVALID_ARG;
  if (k > kGroupK) return VC_ERR_UNSUPPORTED;
  const GroupLayout gl = group_layout(pr);
  uint8_t* work = (uint8_t*)workspace;
  GroupArgs a{};
  a.v = (const __nv_bfloat16*)v;
  a.stride_b = pr.stride_b; a.stride_h = pr.stride_h; a.stride_n = pr.stride_n;
  a.H = pr.H; a.N = pr.N; a.k = k; a.chunks = gl.chunks;
  a.centroids = centroids;
  a.labels = (int32_t*)(work + gl.labels);
  a.psum = (float*)(work + gl.psum);
  a.counts = (int32_t*)(work + gl.counts);
  a.offsets = (int32_t*)(work + gl.offsets);
  a.perm = perm;
  a.status = (uint32_t*)(work + gl.status);
  const uint32_t lim = wait_limit_override();
  a.wait_limit = lim ? lim : kGroupWaitLimit;
  a.nonblocking = lim ? 1u : 0u;
  const cudaError_t e = pr.d == 128 ? run_group<128>(pr, a, iters, warm_start, (cudaStream_t)stream)
                                    : run_group<64>(pr, a, iters, warm_start, (cudaStream_t)stream);
  return e == cudaSuccess ? VC_OK : VC_ERR_CUDA;
}

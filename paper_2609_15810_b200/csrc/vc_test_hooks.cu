// Test hooks that run a piece of the attention kernels' arithmetic on its own.
#include "vc_internal.h"
#include "vc_nvfp4_codes.cuh"
#include "vc_sm100.cuh"

namespace vc {
namespace {

using namespace sm100;

// The ExpCast-FP8 code (Eq. 7) formed exactly as in the softmax stage of the attention kernels:
// per tile fa = cs / 16 and fb = (120 + beta - 8 m) / 128, then expcast_codes4 on four scores.
__global__ void expcast_codes_kernel(const float* __restrict__ s, int64_t n4, float cs, float m, float code_off,
                                     uint32_t* __restrict__ codes) {
  const float fa = cs * 0.0625f, fb = (code_off - 8.0f * m) * 0.0078125f;
  const uint64_t fa2 = pack_f32x2(fa, fa), fb2 = pack_f32x2(fb, fb);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
    const uint4 v = reinterpret_cast<const uint4*>(s)[i];
    codes[i] = expcast_codes4(v.x, v.y, v.z, v.w, fa2, fb2);
  }
}

// NVFP4 probabilities of rows of 128 scores under their running maxima, one thread per row as in the softmax stage.
template <int D, bool POLY>
__global__ void __launch_bounds__(128) nvfp4_codes_kernel(const float* __restrict__ s, const float* __restrict__ m, int64_t rows, float cs,
                                                          uint4* __restrict__ codes, uint2* __restrict__ factors) {
  __shared__ float table[128];
  table[threadIdx.x] = nvfp4::log2_entry(threadIdx.x);
  __syncthreads();
  for (int64_t r = (int64_t)blockIdx.x * 128 + threadIdx.x; r < rows; r += (int64_t)gridDim.x * 128) {
    const nvfp4::Row<D, POLY> nv(cs, m[r], smem_u32(table));
    const float4* src = reinterpret_cast<const float4*>(s + 128 * r);
    uint32_t sv[4][32], sfw[2] = {0u, 0u};
    float mx[8], off[8];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        const float4 v = src[8 * q + i / 4];
        sv[q][i] = __float_as_uint(v.x); sv[q][i + 1] = __float_as_uint(v.y);
        sv[q][i + 2] = __float_as_uint(v.z); sv[q][i + 3] = __float_as_uint(v.w);
      }
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      mx[g] = -INFINITY;
#pragma unroll
      for (int i = 0; i < 16; ++i) mx[g] = fmaxf(mx[g], __uint_as_float(sv[g / 2][16 * (g & 1) + i]));
    }
#pragma unroll
    for (int g = 0; g < 8; g += 2) nv.factors(g, mx, sfw, off);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint2 lo = nv.codes16(sv[q], 0, 2 * q, off), hi = nv.codes16(sv[q], 1, 2 * q + 1, off);
      codes[4 * r + q] = make_uint4(lo.x, lo.y, hi.x, hi.y);
    }
    factors[r] = make_uint2(sfw[0], sfw[1]);
  }
}

}  // namespace
}  // namespace vc

extern "C" vc_status vc_test_nvfp4_codes(const float* s, const float* m, int64_t rows, int32_t d, int32_t polynomial, float cs,
                                         uint8_t* codes, uint8_t* factors, void* stream) {
  if (rows < 0 || (d != 64 && d != 128) || !(cs > 0.f)) return VC_ERR_INVALID_ARG;
  if (rows == 0) return VC_OK;
  if (!s || !m || !codes || !factors || (((uintptr_t)s | (uintptr_t)m | (uintptr_t)codes | (uintptr_t)factors) & 15)) return VC_ERR_INVALID_ARG;
  const int blocks = (int)((rows + 127) / 128 < 4096 ? (rows + 127) / 128 : 4096);
  const auto kernel = polynomial ? (d == 128 ? vc::nvfp4_codes_kernel<128, true> : vc::nvfp4_codes_kernel<64, true>)
                                 : (d == 128 ? vc::nvfp4_codes_kernel<128, false> : vc::nvfp4_codes_kernel<64, false>);
  kernel<<<blocks, 128, 0, (cudaStream_t)stream>>>(s, m, rows, cs, reinterpret_cast<uint4*>(codes), reinterpret_cast<uint2*>(factors));
  vc::count_launches(1);
  return cudaGetLastError() == cudaSuccess ? VC_OK : VC_ERR_CUDA;
}

extern "C" vc_status vc_test_expcast_codes(const float* s, int64_t n, float cs, float m, float beta, uint8_t* codes, void* stream) {
  if (n < 0 || (n & 3) || !(cs > 0.f)) return VC_ERR_INVALID_ARG;
  if (n == 0) return VC_OK;
  if (!s || !codes || (((uintptr_t)s | (uintptr_t)codes) & 15)) return VC_ERR_INVALID_ARG;
  const int64_t n4 = n / 4;
  const int blocks = (int)((n4 + 255) / 256 < 4096 ? (n4 + 255) / 256 : 4096);
  vc::expcast_codes_kernel<<<blocks, 256, 0, (cudaStream_t)stream>>>(s, n4, cs, m, 120.0f + (beta != 0.f ? beta : -0.35f),
                                                                     reinterpret_cast<uint32_t*>(codes));
  vc::count_launches(1);
  return cudaGetLastError() == cudaSuccess ? VC_OK : VC_ERR_CUDA;
}

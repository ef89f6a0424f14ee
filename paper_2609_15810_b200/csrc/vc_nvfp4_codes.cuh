// NVFP4 probabilities: E4M3 factors of the 16-key groups of a row and E2M1 codes, as the softmax stage of the 4-bit attention
// kernel forms them (and the test hook that runs them on their own).
#pragma once
#include <cuda_fp8.h>

#include "vc_sm100.cuh"

namespace vc {
namespace nvfp4 {

using namespace sm100;

// Value of a non-negative E4M3 byte.
__device__ __forceinline__ float decode_ue4m3(uint32_t code) {
  return code >= 8u ? __uint_as_float((code + 960u) << 20) : (float)code * 0.001953125f;
}

// Entry i of the table of logarithms (128 floats): log2 of the E4M3 value with code i; a zero factor gives +infinity.
__device__ __forceinline__ float log2_entry(int i) { return i ? lg2_approx(decode_ue4m3(i)) : INFINITY; }

// E2M1 codes need no exponential, only something that lies on the right side of the format's seven rounding thresholds
// 0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.  This polynomial in x = log2(value) + 2 goes through all seven (x = 0 at the first),
// grows all the way to the top of the range and falls to minus infinity below zero, where the conversion clamps:
// degree 6 through the points plus 1.2e-4 times the product of their distances, in seven packed FMAs per two elements.
// Evaluated in FP32 its thresholds are within 2.4e-7 in the log2 domain (ex2.approx: 2^-22 of the value, 3.4e-7).
__device__ __forceinline__ uint64_t e2m1_poly2(uint64_t x) {
  constexpr float c[8] = {0.25f, 0.23001262545585632f, -0.06627432256937027f, 0.12829358875751495f,
                          -0.0517636276781559f, 0.014539925381541252f, -0.0019345706095919013f, 0.00011999999696854502f};
  uint64_t r = pack_f32x2(c[7], c[7]);
#pragma unroll
  for (int k = 6; k >= 0; --k) r = fma2(r, x, pack_f32x2(c[k], c[k]));
  return r;
}

// p = 2^(s cs - m') * 2688: the row maximum maps to 6 * 448, so the largest factor is 448.
// Per 16-key group: factor = E4M3(max p / 6); element / factor = 2^(s cs + c0 - log2 factor),
// a zero factor (log2: +infinity in the table) zeroes the group.  The logarithm comes from a table
// of the 128 codes, filled with what the instruction gives: decoding a code and taking its
// logarithm eight times per row and key tile cost 14 percent of the kernel (B1 H12 N32760 d128
// 5.25 -> 4.50 ms, B2 H16 N16384 d64 3.37 -> 2.83).
// Groups whose codes come from the polynomial (POLY): two of the eight at d = 128, three at d = 64 (the
// special-function unit is the longer queue there).  None 4.44 / 4.35 ms (B1 H12 N32760 d128 with / without value
// smoothing) and 2.89 (B2 H16 N16384 d64); groups 2 and 4 4.29 / 4.09 and 2.79; 1, 4 and 7 4.47 / 4.33 and 2.74;
// other pairs and threes lie between, four groups 4.43 / 4.37 and 2.89.
template <int D, bool POLY> struct Row {
  float cs, c0, c0p;                                    // log2(2688) - m'; ... + 2, where the polynomial's argument starts
  uint32_t lg2_at;                                      // the table, in shared memory
  __device__ __forceinline__ Row(float cs_, float m, uint32_t table) : cs(cs_), c0(11.39231742277876f - m), c0p(13.39231742277876f - m), lg2_at(table) {}
  static __device__ __forceinline__ constexpr bool by_poly(int g) { return POLY && (((D == 128 ? 0x14 : 0x92) >> g) & 1); }
  // factor bytes of groups g and g + 1 (maxima mx) into their words, and the exponents' offsets
  __device__ __forceinline__ void factors(int g, const float (&mx)[8], uint32_t (&sfw)[2], float (&off)[8]) const {
    const float p0 = ex2_approx(fmaf(mx[g], cs, c0)), p1 = ex2_approx(fmaf(mx[g + 1], cs, c0));
    const uint32_t sb = (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(p0 * (1.0f / 6.0f), p1 * (1.0f / 6.0f)), __NV_SATFINITE, __NV_E4M3);
    sfw[g >> 2] |= sb << (8 * (g & 2));
    off[g] = (by_poly(g) ? c0p : c0) - lds32(lg2_at + 4 * (sb & 0xffu));
    off[g + 1] = (by_poly(g + 1) ? c0p : c0) - lds32(lg2_at + 4 * (sb >> 8));
  }
  // codes of group g: sixteen scores from sv[16 * half] on, element 0 in the low nibble
  __device__ __forceinline__ uint2 codes16(const uint32_t (&sv)[32], int half, int g, const float (&off)[8]) const {
    float v[16];
    const uint64_t cs2 = pack_f32x2(cs, cs), off2 = pack_f32x2(off[g], off[g]);
    if (by_poly(g)) {
#pragma unroll
      for (int i = 0; i < 16; i += 2) unpack2(e2m1_poly2(fma2(pack_b32x2(sv[16 * half + i], sv[16 * half + i + 1]), cs2, off2)), v[i], v[i + 1]);
      return make_uint2(cvt_relu_e2m1x8(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]),
                        cvt_relu_e2m1x8(v[8], v[9], v[10], v[11], v[12], v[13], v[14], v[15]));
    }
#pragma unroll
    for (int i = 0; i < 16; i += 2) {                   // the exponent's FMA on two scores per instruction
      float x0, x1;
      unpack2(fma2(pack_b32x2(sv[16 * half + i], sv[16 * half + i + 1]), cs2, off2), x0, x1);
      v[i] = ex2_approx(x0);
      v[i + 1] = ex2_approx(x1);
    }
    return make_uint2(cvt_e2m1x8(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]),
                      cvt_e2m1x8(v[8], v[9], v[10], v[11], v[12], v[13], v[14], v[15]));
  }
};

}  // namespace nvfp4
}  // namespace vc

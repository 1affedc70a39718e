// Block integers for FP64 reals, shared by the FP64 hopping and force kernels (dhop_p64.cu gives the
// format, its ranges and its error): a block of reals has one binary exponent, that of the largest, and
// every real is x = d1 2^32 + 16 d0 with two signed digits.
#pragma once

#include "dwf_common.cuh"

namespace gdwf {

constexpr int FX_LO = 623, FX_HI = 1423;  // biased exponents 1023 -+ 400 of a block's largest real

// v >> k of an unsigned word, 0 for k >= 32 (the PTX shift clamps its count)
__device__ __forceinline__ uint32_t shr_clamp(uint32_t v, int k) {
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(k));
  return r;
}

// Magnitude digits (y1, y0) of the FP64 value with words (hi, lo) in a block whose largest
// magnitude has the exponent field emax (bits 20..30 of its high word):
// |v| = (y1 2^32 + 16 y0) 2^((emax >> 20) - 1075 - LEFT), truncated; LEFT = 9 (y1 < 2^30) or 8.
template <int LEFT>
__device__ __forceinline__ void fx_magnitude(uint32_t hi, uint32_t lo, uint32_t emax, int& y1, int& y0) {
  const int k = (int)((emax - (hi & 0x7ff00000u)) >> 20);  // >= 0
  const uint32_t m = (hi & 0x000fffffu) | 0x00100000u;
  const uint32_t xh = __funnelshift_l(lo, m, LEFT), xl = lo << LEFT;
  y1 = (int)shr_clamp(xh, k);
  y0 = (int)shr_clamp(__funnelshift_rc(xl, xh, k), max(k - 28, 4));  // low word of (x >> k), >> 4
}

// Largest high word (sign cleared) of n reals.
template <int N>
__device__ __forceinline__ uint32_t fx_max_hi(const double* v) {
  int smax = __double2hiint(v[0]);
  uint32_t umax = (uint32_t)__double2hiint(v[0]);
#pragma unroll
  for (int i = 1; i < N; ++i) {
    smax = max(smax, __double2hiint(v[i]));            // the largest of the non-negative ones
    umax = max(umax, (uint32_t)__double2hiint(v[i]));  // the largest of the negative ones, if any
  }
  return max((uint32_t)max(smax, 0), umax & 0x7fffffffu);
}

template <int N>
__device__ __forceinline__ bool fx_all_zero(const double* v) {
  uint32_t o = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) o |= ((uint32_t)__double2hiint(v[i]) & 0x7fffffffu) | (uint32_t)__double2loint(v[i]);
  return o == 0;
}

}  // namespace gdwf

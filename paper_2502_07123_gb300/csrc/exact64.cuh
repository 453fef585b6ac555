// The FP64 exact path's inverse Normal and path increments in 64-bit integers.
//
// FP64 arithmetic runs at 2 lanes per clock and SM on this GPU, 1/64 of the
// FP32 rate (a warp's FP64 instruction holds the SM's unit for 16 cycles, in
// which the four schedulers issue 64 others), so a library FP64 Phi^-1 -- about
// 60 FP64 operations -- bounded the FP64 kernels at 7.1e9 path-steps/s with the
// unit 85% busy.  Here Phi^-1 is a quintic by table evaluated on 32 x 32 -> 64
// integer multiplies, the increment c1 + c2 Z (+ c3 (Z^2 - 1)) is formed in
// 62 bits, and one FP64 multiply-add per path and step remains (S's update,
// whose rounding and range stay FP64's): about 120 instructions per Milstein
// path-step, bound by issue and the ALU pipe (53%) with the FP64 unit at 42%.
// 500,003 level-5 Milstein European samples: 2.25 -> 0.110 ms.  Absolute error of Phi^-1 at most
// 2^-54, root mean square 2^-57.8 (a correctly rounded FP64 value of [1, 2) is
// up to 2^-53 off).  An increment adds to c2 2^-54 and c3 |Z| 2^-53 of that at most
// 5 units 2^-qF (Euler: a product up to 4.4 low, the complement's one, q1's half; 10
// on the coarse path; Milstein 12 and 38; emulated over 3e5 draws 3.3, 5.7, 4.6 and
// 12.3).  qF is 58 for increments near 8 and 68 below 2^-7 (exact64_consts).
#pragma once
#include <stdint.h>

#include "device_common.cuh"
#include "phi_inv64_table.h"

namespace mlmc {

// The four octaves of u in [2^-5, 1/2) -- 15 of 16 draws -- are staged in shared
// memory (two arrays, so that a warp's 16-byte reads spread over all the bank
// groups: 2 x 8 KB); the other octaves' parts are read through L1.
constexpr int PHI64_HOT = 4 * PHI64_SUB;
__device__ __forceinline__ ulonglong2 *phi64_smem() {
  __shared__ ulonglong2 s_phi64[2 * PHI64_HOT];
  return s_phi64;
}
__device__ __forceinline__ void stage_phi64() {
  ulonglong2 *d = phi64_smem();
  for (int k = threadIdx.x; k < PHI64_HOT; k += blockDim.x) {
    copy16_async(d + k, k_phi64_a + k);
    copy16_async(d + PHI64_HOT + k, k_phi64_b + k);
  }
}

// Leading zeros of x != 0 in one instruction.
__device__ __forceinline__ uint32_t shift_to_top(uint32_t x) {
  uint32_t r;
  asm("bfind.shiftamt.u32 %0, %1;" : "=r"(r) : "r"(x));
  return r;
}

// y = -Phi^-1(2^-32 (J + 1/2)) 2^60 for J < 2^31 (u in (0, 1/2), y < 6.34 2^60).
// N = 2 J + 1, so u = N 2^-33; gen_phi_inv64_table.py tells the coefficients.
__device__ __forceinline__ uint64_t probit_q60(uint32_t J, const ulonglong2 *tab) {
  const uint32_t N = 2u * J + 1u;
  const uint32_t lz = shift_to_top(N);
  const uint32_t M = N << lz;
  const uint32_t t = 0x1000000u - (M & 0xFFFFFFu), T = t << 7;   // s 2^24, s 2^31
  const uint32_t k = lz * PHI64_SUB + (M >> 24) - PHI64_SUB;
  ulonglong2 a, b;
  if (k < (uint32_t)PHI64_HOT) {
    a = tab[k];
    b = tab[PHI64_HOT + k];
  } else {
    a = __ldg(&k_phi64_a[k]);
    b = __ldg(&k_phi64_b[k]);
  }
  const uint32_t a4 = (uint32_t)(b.y >> 32) + __umulhi((uint32_t)b.x & 0x7FFFFu, T);   // 2^-56
  const uint32_t a3 = (uint32_t)b.y + __umulhi(a4, T);                                 // 2^-55
  const uint64_t a2 = b.x + (uint64_t)a3 * t;                                          // 2^-79
  const uint64_t a1 = a.y + (uint64_t)(uint32_t)(a2 >> 32) * t + __umulhi((uint32_t)a2, t);   // 2^-71
  return a.x + (((uint64_t)(uint32_t)(a1 >> 32) * t + __umulhi((uint32_t)a1, t)) >> 3);       // 2^-60
}

// The high 64 bits of a b, up to 3 units low (the low words' product is left
// out).  hi(a) + hi(b) < 2^32, so that the cross products add in 32 bits.
__device__ __forceinline__ uint64_t mulhi64_3(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  return (uint64_t)ah * bh + (__umulhi(ah, bl) + __umulhi(al, bh));
}

// v 2^-F as a double by integer operations (a conversion instruction from 64
// bits runs at the FP64 rate).  hi0 = (1085 - F) << 20.  |v| is taken as v or
// ~v with its last bit set (one unit 2^-F, below the increment's own error); the
// 53rd bit stands for whatever is cut off below it, so the result is within one
// unit in the last place, without bias.  F >= 58, so a zero increment's 2^-F
// leaves S unchanged.
__device__ __forceinline__ double q_to_double(int64_t v, uint32_t hi0) {
  const uint32_t s = (uint32_t)((int32_t)((uint64_t)v >> 32) >> 31);
  uint32_t h = (uint32_t)((uint64_t)v >> 32) ^ s, l = ((uint32_t)v ^ s) | 1u;
  const bool small = h == 0u;   // |v| < 2^32: rare
  h = small ? l : h;
  l = small ? 0u : l;
  hi0 = small ? hi0 - (32u << 20) : hi0;
  const uint32_t lz = shift_to_top(h);
  h = __funnelshift_l(l, h, lz);
  l = l << lz;
  // the leading one adds 1 to the exponent field
  const uint32_t hi = (h >> 11) - (lz << 20) + hi0;
  return __hiloint2double((int)(hi | (s & 0x80000000u)), (int)(__funnelshift_r(l, h, 11) | 1u));
}

// min(x, y) of doubles by integer comparison (the FP64 comparison runs at the
// FP64 rate).  A NaN of positive sign loses, one of negative sign wins; the path
// minimum may be either, since the payoff subtracts it from a terminal value that
// is NaN from the same step on.
__device__ __forceinline__ double min_f64(double x, double y) {
  const int64_t a = __double_as_longlong(x), b = __double_as_longlong(y);
  const int64_t ka = a ^ (int64_t)((uint64_t)(a >> 63) >> 1), kb = b ^ (int64_t)((uint64_t)(b >> 63) >> 1);
  return ka < kb ? x : y;
}

// a > b for b >= 0 (positive zero), likewise; false for a NaN.
__device__ __forceinline__ bool above_f64(double a, double b) {
  const int64_t x = __double_as_longlong(a);
  return x > __double_as_longlong(b) && x <= 0x7FF0000000000000LL;
}

// 1 / x: the hardware's single-precision reciprocal r of x and one cubic step of
// Newton's iteration, r (1 + e + e^2) with e = 1 - x r (|e| < 2^-21, so what is
// left out is below 2^-63); by division outside the float range.
__device__ __forceinline__ double reciprocal(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const uint32_t mag = (uint32_t)hi & 0x7FFFFFFFu;
  if (mag - 0x39B00000u >= 0x0C800000u) return 1.0 / x;   // |x| outside [2^-100, 2^100)
  const float f = __uint_as_float(((mag - 0x38000000u) << 3) | ((uint32_t)lo >> 29));
  float rf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(f));
  const uint32_t b = __float_as_uint(rf);
  const double r = __hiloint2double((int)(((b >> 3) + 0x38000000u) | ((uint32_t)hi & 0x80000000u)), (int)(b << 29));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

}  // namespace mlmc

// Device building blocks of the level kernels: Philox4x32-10, the exact and
// approximate Normal maps of Sec. 3, fixed-point re-quantisation (Sec. 4.1)
// and 128-bit integer accumulation.
#pragma once
#include "phi_inv_table.h"
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "item.h"

namespace mlmc {

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds, each with two
// 32x32->64 products by the published multipliers; the round keys
// (key + r * Weyl increment) are precomputed on the host.
constexpr uint32_t PHILOX_M0 = 0xD2511F53u;
constexpr uint32_t PHILOX_M1 = 0xCD9E8D57u;
constexpr uint32_t PHILOX_W0 = 0x9E3779B9u;
constexpr uint32_t PHILOX_W1 = 0xBB67AE85u;

__device__ __forceinline__ uint4 philox_rounds(uint4 c, const RoundKeys &rk, int first) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r < first) continue;
    const uint64_t p0 = (uint64_t)PHILOX_M0 * c.x;
    const uint64_t p1 = (uint64_t)PHILOX_M1 * c.z;
    c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ rk.k[2 * r], (uint32_t)p1,
                   (uint32_t)(p0 >> 32) ^ c.w ^ rk.k[2 * r + 1], (uint32_t)p0);
  }
  return c;
}
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const RoundKeys &rk) { return philox_rounds(c, rk, 0); }

// Philox calls that differ in the counter's low word only: of the first two
// rounds' four products two are the same for all of them, as are the words
// they meet.
struct PhiloxStream {
  uint32_t z0, x1, z1, w1;
  __device__ __forceinline__ PhiloxStream(uint32_t q_hi, uint32_t ctr2, uint32_t ctr3, const RoundKeys &rk) {
    const uint64_t p = (uint64_t)PHILOX_M1 * ctr2;
    z0 = ctr3 ^ rk.k[1];
    x1 = (uint32_t)p ^ rk.k[2];
    const uint64_t q = (uint64_t)PHILOX_M0 * ((uint32_t)(p >> 32) ^ q_hi ^ rk.k[0]);
    z1 = (uint32_t)(q >> 32) ^ rk.k[3];
    w1 = (uint32_t)q;
  }
  __device__ __forceinline__ uint4 call(uint32_t q_lo, const RoundKeys &rk) const {
    const uint64_t p0 = (uint64_t)PHILOX_M0 * q_lo;
    const uint64_t p1 = (uint64_t)PHILOX_M1 * ((uint32_t)(p0 >> 32) ^ z0);
    return philox_rounds(make_uint4((uint32_t)(p1 >> 32) ^ x1, (uint32_t)p1, (uint32_t)p0 ^ z1, w1), rk, 2);
  }
};

__device__ __forceinline__ uint32_t word_of(const uint4 &w, int k) {
  return k == 0 ? w.x : k == 1 ? w.y : k == 2 ? w.z : w.w;
}

// 16 bytes from global to shared memory without waiting; the thread waits for
// all of its copies (copies_done) before the barrier that publishes them.
__device__ __forceinline__ void copy16_async(void *smem, const void *global) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(global)
               : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The inverse-Normal cubics (phi_inv_table.h) in shared memory.  A warp's 32
// random 16-byte reads of one copy cost 10.4 wavefronts on average (the fullest
// of 8 bank groups, per quarter warp); beside the pair table's 6.2 they held
// shared memory 76% busy in the correction kernels.  So there (OCT = 4) the parts
// of the four octaves [2^-5, 1/2) -- 15 of 16 draws -- are kept eight times, one
// copy per bank group, and lane l reads copy l mod 8: 4 wavefronts and about 1.7
// conflicts with a rarer part, which is kept once.  15 KB; 8,000,009 level-4
// corrections 317 -> 297 us.  The exact kernels, whose shared memory is 30% busy,
// keep one copy (OCT = 0, 8 KB): staging more slowed their short chunks by 5%.
constexpr int PHI_K0 = 94 << 4;   // exponent field and top four bits of the first part, u = 2^-33
template <int OCT>
struct PhiTable {
  static constexpr int COPIES = OCT ? 8 : 1, HOT0 = OCT ? (32 - OCT) * 16 : PHI_INV_PARTS;
  static constexpr int SIZE = HOT0 + (PHI_INV_PARTS - HOT0) * COPIES;   // in float4
  static __device__ __forceinline__ void stage(float4 *d) {
    for (int k = threadIdx.x; k < HOT0; k += blockDim.x) copy16_async(d + k, k_phi_inv + k);
    for (int k = threadIdx.x; k < SIZE - HOT0; k += blockDim.x)
      copy16_async(d + HOT0 + k, k_phi_inv + HOT0 + k / COPIES);
  }
  // What a hot part's index adds to COPIES x (exponent and top bits) for the calling lane's copy.
  static __device__ __forceinline__ uint32_t lane() {
    return (threadIdx.x & (COPIES - 1)) + (uint32_t)(PHI_K0 + HOT0 - COPIES * (PHI_K0 + HOT0));
  }
};

// Exact Normal Z = Phi^{-1}(2^-32 (J + 1/2)) in single precision (Sec. 3.1).
// The upper half uses Phi^{-1}(1 - u) = -Phi^{-1}(u): with J' = J or ~J below
// 2^31, u = 2^-32 (J' + 1/2) (J' rounded to nearest as a float) lies in
// [2^-33, 1/2].  Phi^{-1}(u) is the cubic of u's part (tab: staged as
// above, lane: PhiTable::lane()): u's exponent and the top four bits of its significand
// pick one of 512 parts of [2^-33, 1/2) (the 513th is u = 1/2), the other 19
// bits are the position t in [0, 1) within it, which as the low bits of a
// float of [16, 17) need no shift.  Error: about 1e-7 (1 + |Z|), unbiased
// (round to nearest).
template <int OCT>
__device__ __forceinline__ float exact_normal_f32(uint32_t J, const float4 *tab, uint32_t lane) {
  const uint32_t m = (uint32_t)((int32_t)J >> 31);
  const float u = fmaf(__uint2float_rn(J ^ m), 0x1p-32f, 0x1p-33f);
  const uint32_t b = __float_as_uint(u);
  uint32_t k = b >> 19;
  if (OCT > 0 && b >= (uint32_t)(PHI_K0 + PhiTable<OCT>::HOT0) << 19) k = k * PhiTable<OCT>::COPIES + lane;
  const float4 c = tab[(int)k - PHI_K0];
  const float t = __uint_as_float((b & 0x7FFFFu) | 0x41800000u) - 16.0f;
  const float z = fmaf(fmaf(fmaf(c.w, t, c.z), t, c.y), t, c.x);
  return __uint_as_float(__float_as_uint(z) ^ (J & 0x80000000u));
}

// Table index of the approximate Normal (Sec. 3.1): j = top d bits of J; the
// upper half (leading bit of j set) mirrors the index and flips the sign, so
// Z~ is the mean of Phi^{-1} over the 2^-d interval containing U.
struct ApproxIndex {
  uint32_t idx;
  bool neg;
};
__device__ __forceinline__ ApproxIndex approx_index(uint32_t J, int d) {
  const uint32_t j = J >> (32 - d);
  const uint32_t m = 0u - (j >> (d - 1));
  return ApproxIndex{(j ^ m) & ((1u << (d - 1)) - 1u), m != 0u};
}

// Method-3 class of a table index: {0,1} -> 0, [2^c, 2^(c+1)) -> c.
__device__ __forceinline__ int m3_class(uint32_t idx) {
  return 31 - __clz(idx | 1u);
}

// Fixed point: exact re-expression and rounding (ties toward +inf), saturation.
__device__ __forceinline__ int64_t requant(int64_t x, const Requant &q) {
  const int64_t y = (int64_t)((uint64_t)x << q.ls) + q.radd;
  return y >> q.rs;
}
__device__ __forceinline__ int64_t saturate(int64_t x, int64_t lim, uint32_t &sat) {
  const int64_t y = x > lim ? lim : (x < -lim ? -lim : x);
  sat |= (uint32_t)(y != x);
  return y;
}

// Half-precision helpers: one IEEE rounding per operation, never fused.
template <class H> struct HalfOps;
template <> struct HalfOps<__half> {
  static __device__ __forceinline__ __half mul(__half a, __half b) { return __hmul_rn(a, b); }
  static __device__ __forceinline__ __half add(__half a, __half b) { return __hadd_rn(a, b); }
  static __device__ __forceinline__ __half sub(__half a, __half b) { return __hsub_rn(a, b); }
  static __device__ __forceinline__ float to_f(__half a) { return __half2float(a); }
  static __device__ __forceinline__ __half from_bits(uint16_t b) { return __ushort_as_half(b); }
  static __device__ __forceinline__ __half from_f(float x) { return __float2half_rn(x); }
  static __device__ __forceinline__ __half neg(__half a) { return __hneg(a); }
};
template <> struct HalfOps<__nv_bfloat16> {
  static __device__ __forceinline__ __nv_bfloat16 mul(__nv_bfloat16 a, __nv_bfloat16 b) { return __hmul_rn(a, b); }
  static __device__ __forceinline__ __nv_bfloat16 add(__nv_bfloat16 a, __nv_bfloat16 b) { return __hadd_rn(a, b); }
  static __device__ __forceinline__ __nv_bfloat16 sub(__nv_bfloat16 a, __nv_bfloat16 b) { return __hsub_rn(a, b); }
  static __device__ __forceinline__ float to_f(__nv_bfloat16 a) { return __bfloat162float(a); }
  static __device__ __forceinline__ __nv_bfloat16 from_bits(uint16_t b) { return __ushort_as_bfloat16(b); }
  static __device__ __forceinline__ __nv_bfloat16 from_f(float x) { return __float2bfloat16_rn(x); }
  static __device__ __forceinline__ __nv_bfloat16 neg(__nv_bfloat16 a) { return __hneg(a); }
};

// Paired (x2) form: one instruction rounds both halves of a 32-bit register,
// each exactly as the scalar operation of HalfOps would.
template <class H> struct HalfOps2;
template <> struct HalfOps2<__half> {
  using T = __half2;
  static __device__ __forceinline__ T mul(T a, T b) { return __hmul2_rn(a, b); }
  static __device__ __forceinline__ T add(T a, T b) { return __hadd2_rn(a, b); }
  static __device__ __forceinline__ T sub(T a, T b) { return __hsub2_rn(a, b); }
  static __device__ __forceinline__ T pack(__half lo, __half hi) { return __halves2half2(lo, hi); }
  static __device__ __forceinline__ T splat(__half a) { return __half2half2(a); }
  static __device__ __forceinline__ __half lo(T a) { return __low2half(a); }
  static __device__ __forceinline__ __half hi(T a) { return __high2half(a); }
};
template <> struct HalfOps2<__nv_bfloat16> {
  using T = __nv_bfloat162;
  static __device__ __forceinline__ T mul(T a, T b) { return __hmul2_rn(a, b); }
  static __device__ __forceinline__ T add(T a, T b) { return __hadd2_rn(a, b); }
  static __device__ __forceinline__ T sub(T a, T b) { return __hsub2_rn(a, b); }
  static __device__ __forceinline__ T pack(__nv_bfloat16 lo, __nv_bfloat16 hi) { return __halves2bfloat162(lo, hi); }
  static __device__ __forceinline__ T splat(__nv_bfloat16 a) { return __bfloat162bfloat162(a); }
  static __device__ __forceinline__ __nv_bfloat16 lo(T a) { return __low2bfloat16(a); }
  static __device__ __forceinline__ __nv_bfloat16 hi(T a) { return __high2bfloat16(a); }
};

// 128-bit unsigned accumulation of squares of int64 values.
__device__ __forceinline__ void add_u128(uint64_t &lo, uint64_t &hi, uint64_t alo, uint64_t ahi) {
  const uint64_t nlo = lo + alo;
  hi += ahi + (uint64_t)(nlo < lo);
  lo = nlo;
}
__device__ __forceinline__ void add_square(uint64_t &lo, uint64_t &hi, int64_t y) {
  const uint64_t a = (uint64_t)(y < 0 ? -y : y);
  add_u128(lo, hi, a * a, __umul64hi(a, a));
}

}  // namespace mlmc

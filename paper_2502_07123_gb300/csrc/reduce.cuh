// Deterministic reduction of per-chunk partial sums, shared by the plan
// finalize kernel and the engine's accumulate kernel so that both produce the
// same bits for the same chunking.
#pragma once
#include <cuda_runtime.h>

#include "item.h"

namespace mlmc {

// The sum of partials[0, n) in a fixed order, by a CTA (the level kernels) or a
// warp (finalize_kernel, the engine), with the same bits: 128 columns, column v
// adding chunks v, v + 128, ... in turn; the 32 columns of each of the four
// groups meet in an xor butterfly; the four group totals are added in order.
// Integer sums are exact (Sigma Y^2 in 128 bits).
//
// The CTA that finishes an item last reads all its partials through L2: as one
// warp with one load in flight per lane, 388 dependent rounds for 12,401 chunks
// -- about 75 us with every other SM idle.  Now four warps, six chunks in flight
// per column, and only the sums that the estimator has.
struct PartialSum {
  int64_t isum = 0;
  uint64_t lo = 0, hi = 0, ns = 0;
  double ds = 0.0, dq = 0.0;
  template <bool INTS = true, bool REALS = true>
  __device__ __forceinline__ void add(int64_t i, uint64_t l, uint64_t h, uint64_t n, double s, double q) {
    if constexpr (INTS) {
      isum += i;
      const uint64_t nlo = lo + l;
      hi += h + (uint64_t)(nlo < lo);
      lo = nlo;
    }
    if constexpr (REALS) {
      ds += s;
      dq += q;
    }
    ns += n;
  }
  template <bool INTS = true, bool REALS = true>
  __device__ __forceinline__ void add(const PartialSum &o) {
    add<INTS, REALS>(o.isum, o.lo, o.hi, o.ns, o.ds, o.dq);
  }
};

constexpr uint32_t SUM_COLUMNS = 128;

// Column v's chunks.  CG: read through L2 only (partials written by other CTAs
// of the running kernel).  INTS, REALS: which sums the partials hold (the
// others are zero in all of them).
template <bool CG, bool INTS, bool REALS>
__device__ __forceinline__ PartialSum column_sum(const Partial *partials, uint32_t n, uint32_t v) {
  constexpr int DEPTH = 6;
  PartialSum t;
  auto u64 = [](const void *p) {
    const unsigned long long *q = reinterpret_cast<const unsigned long long *>(p);
    return CG ? __ldcg(q) : *q;
  };
  auto f64 = [](const double *p) { return CG ? __ldcg(p) : *p; };
  for (uint32_t c = v; c < n; c += SUM_COLUMNS * DEPTH) {
    unsigned long long is[DEPTH], lo[DEPTH], hi[DEPTH], ns[DEPTH];
    double ds[DEPTH], dq[DEPTH];
#pragma unroll
    for (int k = 0; k < DEPTH; ++k) {
      const uint32_t i = c + k * SUM_COLUMNS;
      const Partial *p = partials + (i < n ? i : v);
      is[k] = INTS ? u64(&p->isum) : 0;
      lo[k] = INTS ? u64(&p->isum2_lo) : 0;
      hi[k] = INTS ? u64(&p->isum2_hi) : 0;
      ds[k] = REALS ? f64(&p->dsum) : 0.0;
      dq[k] = REALS ? f64(&p->dsum2) : 0.0;
      ns[k] = u64(&p->nsat);
    }
#pragma unroll
    for (int k = 0; k < DEPTH; ++k)
      if (c + k * SUM_COLUMNS < n) t.add<INTS, REALS>((int64_t)is[k], lo[k], hi[k], ns[k], ds[k], dq[k]);
  }
  return t;
}

// Column v's only chunk (at most 32 of them in all): little code, which a small
// launch fetches for this one use.
template <bool INTS, bool REALS>
__device__ __forceinline__ PartialSum one_chunk(const Partial *partials, uint32_t n, uint32_t v) {
  PartialSum t;
  if (v < n) {
    const Partial *p = partials + v;
    if constexpr (INTS) {
      t.isum = __ldcg(reinterpret_cast<const long long *>(&p->isum));
      t.lo = __ldcg(reinterpret_cast<const unsigned long long *>(&p->isum2_lo));
      t.hi = __ldcg(reinterpret_cast<const unsigned long long *>(&p->isum2_hi));
    }
    if constexpr (REALS) {
      t.ds = __ldcg(&p->dsum);
      t.dq = __ldcg(&p->dsum2);
    }
    t.ns = __ldcg(reinterpret_cast<const unsigned long long *>(&p->nsat));
  }
  return t;
}

// The 32 columns of a group, one per lane: every lane gets their total.
template <bool INTS, bool REALS>
__device__ __forceinline__ PartialSum group_sum(PartialSum t) {
  for (int m = 16; m >= 1; m >>= 1) {
    PartialSum o;
    if constexpr (INTS) {
      o.isum = __shfl_xor_sync(0xffffffffu, (long long)t.isum, m);
      o.lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)t.lo, m);
      o.hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)t.hi, m);
    }
    if constexpr (REALS) {
      o.ds = __shfl_xor_sync(0xffffffffu, t.ds, m);
      o.dq = __shfl_xor_sync(0xffffffffu, t.dq, m);
    }
    o.ns = __shfl_xor_sync(0xffffffffu, (unsigned long long)t.ns, m);
    t.add<INTS, REALS>(o);
  }
  return t;
}

__device__ __forceinline__ DevSums to_sums(const PartialSum &t) {
  DevSums r;
  r.dsum = t.ds; r.dsum2 = t.dq; r.isum = t.isum; r.isum2_lo = t.lo; r.isum2_hi = t.hi; r.nsat = t.ns;
  return r;
}

// By all 32 lanes of a warp; every lane returns the total.
__device__ inline DevSums warp_sum_partials(const Partial *partials, uint32_t n) {
  const uint32_t lane = threadIdx.x & 31;
  PartialSum t = group_sum<true, true>(column_sum<false, true, true>(partials, n, lane));
  for (uint32_t w = 1; w < SUM_COLUMNS / 32; ++w)
    t.add(group_sum<true, true>(column_sum<false, true, true>(partials, n, 32 * w + lane)));
  return to_sums(t);
}

// By all threads of a CTA of one to four warps (the partials written by other
// CTAs of the running kernel); thread 0 returns the total.
template <bool INTS, bool REALS>
__device__ inline DevSums cta_sum_partials(const Partial *partials, uint32_t n) {
  __shared__ PartialSum group[SUM_COLUMNS / 32];
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t w = threadIdx.x >> 5; w < SUM_COLUMNS / 32; w += blockDim.x >> 5) {
    const PartialSum t = group_sum<INTS, REALS>(column_sum<true, INTS, REALS>(partials, n, 32 * w + lane));
    if (lane == 0) group[w] = t;
  }
  __syncthreads();
  PartialSum t = group[0];
  for (uint32_t w = 1; w < SUM_COLUMNS / 32; ++w) t.add<INTS, REALS>(group[w]);
  return to_sums(t);
}

// Unsigned 128-bit integer to the nearest double (ties to even).
__device__ inline double u128_to_double_rn(unsigned long long lo, unsigned long long hi) {
  if (hi == 0) return __ull2double_rn(lo);
  const int z = __clzll((long long)hi);
  unsigned long long m = z ? ((hi << z) | (lo >> (64 - z))) : hi;
  const unsigned long long rest = z ? (lo << z) : lo;
  m |= (rest != 0ULL) ? 1ULL : 0ULL;   // sticky bit below the 64 kept bits
  return ldexp(__ull2double_rn(m), 64 - z);
}

}  // namespace mlmc

// The MLMC level kernel: per-sample coupled fine/coarse GBM paths of one
// level (Sec. 2.1), exact Normals and/or table-based approximate Normals from
// the same uniform J (Sec. 3), the low-precision path in fixed point
// (Algorithm 1) or binary16/bfloat16, payoffs, the level difference / nested
// correction (eq. chap:nested_exp) and per-CTA sums of Y and Y^2.
//
// Layout: one CTA processes one chunk of one work item; each thread simulates
// groups of samples whose uniforms come from one Philox call per group (4
// packs per call on level 0, 2 on level 1, one pack over 2^l / 4 calls above;
// a pack is one sample, or three with packed draws), entirely in registers.  The approximate-Normal table of the item
// lives in shared memory.  The only global-memory traffic is the work-item
// descriptor, the table, one Partial record per CTA, the item's sums (written
// by the CTA that finishes its last chunk) and the optional dump.
#pragma once
#include <type_traits>

#include "device_common.cuh"
#include "exact64.cuh"
#include "mlmc.h"
#include "reduce.cuh"

namespace mlmc {

using mlmc_sample_rec = ::mlmc_sample;

// Words of "call" q when the table indices enumerate the samples (levels 0 and
// 1): sample s takes j_i = (s >> (d i)) mod 2^d at step i, placed in the top d
// bits; the word layout per call is the one of the Philox draws.
__device__ __forceinline__ uint4 enum_words(uint64_t q, int lev, int d) {
  const uint32_t mask = (1u << d) - 1u, sh = 32u - (uint32_t)d;
  if (lev == 0) {
    const uint32_t s = 4u * (uint32_t)q;
    return make_uint4((s & mask) << sh, ((s + 1u) & mask) << sh, ((s + 2u) & mask) << sh, ((s + 3u) & mask) << sh);
  }
  const uint32_t s0 = 2u * (uint32_t)q, s1 = s0 + 1u;
  return make_uint4((s0 & mask) << sh, ((s0 >> d) & mask) << sh, (s1 & mask) << sh, ((s1 >> d) & mask) << sh);
}

template <int XP> struct XType { using T = float; };
template <> struct XType<XP_F64> { using T = double; };
template <int AP> struct HType { using T = __half; };
template <> struct HType<AP_BF16> { using T = __nv_bfloat16; };
template <> struct HType<AP_BF16S> { using T = __nv_bfloat16; };

constexpr int MAX_THREADS = 256;
// Register budget: the approximate fixed-point Euler kernel with terminal payoffs
// (the bulk of the nested estimator) and the merged nested kernel run with 7
// resident 128-thread CTAs per SM (72 registers per thread, no spills): 2e8
// packed path-steps at level 4 172 us with 6, 158 with 7 and with 8 (64
// registers, which spill and cost level 2 1%).  The matching correction kernel
// (static launch) takes 6, 80 registers instead of 111 (its device-scheduled
// form would spill there and keeps its allocation); 5 cost it 0.5%.
// The approximate 32-bit fixed-point Asian kernels run 4 CTAs per SM (<= 128
// registers, measured 8-16% faster than their natural ~144), as do the
// corrections whose natural allocation lies just above.
// The FP32 exact kernels need 80-96 registers and are held to 80 but for three
// device-scheduled ones and the Asian ones, which take 5 CTAs (8,000 level-10
// samples 56 -> 53 us, 1.2e8 level-1 ones 459 -> 457); the binary16 / bfloat16
// corrections' static launches
// need up to 104 and are held to 96, and the unpacked binary16 / bfloat16
// approximate kernels' (two samples per thread from level 2), 84-96, to 80.
// Every other instantiation keeps its natural allocation (a cap there spills).
constexpr int LAUNCH_THREADS = 128;
template <int EST, int XP, int AP, int SCHEME, int PC, int KP, bool DYN = false> struct MinCtas {
  static constexpr bool EM_TERMINAL_FX32 = AP == AP_FX32 && SCHEME == 0 && PC == PC_TERMINAL;
  static constexpr bool FX = AP == AP_FX32 || AP == AP_FX64;
  static constexpr int value =
      EM_TERMINAL_FX32 && EST == EST_APPROX ? 7
      : EM_TERMINAL_FX32 && EST == EST_CORR && !DYN ? 6
      : EST == EST_EXACT && XP == XP_F32 ? (!DYN && PC == PC_ASIAN ? 5 : !DYN || (SCHEME == 0 && PC != PC_ASIAN) ? 6 : 1)
      : EST == EST_CORR && FX ? 4
      : EST == EST_CORR && AP != AP_FIXED && !DYN ? (SCHEME == 1 && PC == PC_ASIAN ? 4 : 5)
      : EST == EST_APPROX && AP == AP_FX32 && PC == PC_ASIAN ? 4
      : EST == EST_APPROX && KP == 1 && !DYN && AP != AP_FIXED && !FX ? 6 : 1;
};

// The inverse-Normal cubics of the FP32 exact path in shared memory, the same
// for every item.  Kernels whose chunks run an FP32 exact path stage them once
// per CTA, before their first chunk's table (whose barrier makes them visible).
template <int OCT>
__device__ __forceinline__ float4 *phi_inv_smem() {
  __shared__ float4 s_phi_inv[PhiTable<OCT>::SIZE];
  return s_phi_inv;
}
template <int OCT>
__device__ __forceinline__ void stage_phi_inv() {
  PhiTable<OCT>::stage(phi_inv_smem<OCT>());
}
constexpr int PHI_OCT_CORR = 4, PHI_OCT_EXACT = 0;

// The exact path's inverse-Normal table of a kernel, if it has one.
template <int EST, int XP>
__device__ __forceinline__ void stage_exact_table() {
  if constexpr (EST == EST_CORR && XP == XP_F32) stage_phi_inv<PHI_OCT_CORR>();
  if constexpr (EST == EST_EXACT && XP == XP_F32) stage_phi_inv<PHI_OCT_EXACT>();
  if constexpr (EST != EST_APPROX && XP == XP_F64) stage_phi64();
}

// Bytes per entry of the shared-memory approximate-Normal table of a datapath:
// the 32-bit fast fixed-point datapath keeps (Z~_j, sum1 of a fine step) pairs.
template <int AP>
struct TabBytes {
  static constexpr size_t value = AP == AP_FX32 ? 8 : ((AP == AP_FIXED || AP == AP_FX64) ? 4 : 2);
};

// sum1 of one fast fixed-point step of Algorithm 1 from its Normal increment z:
// mul1 = rd(con2 z), [Milstein: mul3 = rd(con3 (z^2 - m))], sum1 = rd(con1 + mul1
// [+ mul3]).  c1r: con1 (fine) or con1_c (coarse) with sum1's rounding half unit;
// m: 1 (fine) or 2 (coarse) in units 2^-2fZ.  F32: the host proved every
// rounding shift below 32, so a product's rounded value is one funnel shift of
// its two words.
template <bool MIL, bool F32>
__device__ __forceinline__ int32_t ff_sum1(const FastFixed &ff, int32_t z, int32_t c1r, int64_t m) {
  int32_t mul1;
  const int64_t p1 = (int64_t)ff.con2 * z + ff.radd1;
  if constexpr (F32) mul1 = (int32_t)__funnelshift_r((uint32_t)p1, (uint32_t)((uint64_t)p1 >> 32), ff.rs1);
  else mul1 = (int32_t)(p1 >> ff.rs1);
  int32_t acc = c1r + mul1 * ff.mulF1;
  if constexpr (MIL) {
    // |Z~^2 - m| < 2^31 on this datapath (host-checked): one 32 x 32 product
    const int32_t zz = z * z - (int32_t)m;
    const int64_t p3 = (int64_t)ff.con3 * zz + ff.radd3;
    int32_t mul3;
    if constexpr (F32) mul3 = (int32_t)__funnelshift_r((uint32_t)p3, (uint32_t)((uint64_t)p3 >> 32), ff.rs3);
    else mul3 = (int32_t)(p3 >> ff.rs3);
    acc += mul3 * ff.mulF1;
  }
  return acc >> ff.rs_sum1;
}

// KP > 1 (approximate-only estimators): KP samples advance in lockstep, lane L
// reading bits [32 - d(L+1), 32 - dL) of the shared word (packed draws).
// MSEL: 0 the item uses a table lookup (Methods 1 and 2), 1 the line
// evaluation of Method 3, 2 either, chosen per step (only the per-sample
// dump instantiation), 4 a table lookup whose exact path is coupled by Method
// 2's ranks (corrections); chosen once per chunk, so the hot step code has no
// branch on the method.  FP64 exact kernels: 0 increments in 64-bit integers
// (exact64.cuh), 1 in FP64.
// PRE: the 32-bit fast datapath in its pre-scaled form, for items whose bounds
// allow it (FastFixed::pre_ok).  sum1 is kept times 2^(32 - rs2), so the rounded
// product rd(S sum1) is the high word of one 64-bit multiply-add, with no
// shift; and, mul1 and sum1 having the same grid, sum1 is mul1 plus a constant.
// Euler: the table holds P_j = con2 Z~_j + radd1 alone (4 bytes): a fine step's
// mul1 is P_j >> rs1 and a coarse step's (P_j + P_j' - radd1) >> rs1.  The
// 8-byte pairs' random reads cost 6.2 shared-memory wavefronts a warp, which
// held shared memory 83% busy in the packed approximate kernel; 4-byte reads
// cost 3.5.  Milstein: the pairs (Z~_j, scaled sum1_j).
// MERGED: the merged nested kernel's instantiation, which takes no enumerated
// items (the plan keeps those apart), so its group code has no enumeration
// branch.
template <int EST, int XP, int AP, int SCHEME, int PC, int KP = 1, int MSEL = 0, bool PRE = false,
          bool MERGED = false>
struct LevelSim {
  static_assert(KP == 1 || EST == EST_APPROX, "packed draws feed approximate-only estimators");
  static constexpr bool ENUMERATE = !MERGED;   // the group code reads enumerated words when asked
  static constexpr bool HAS_EXACT = (EST != EST_APPROX);
  static constexpr bool HAS_APPROX = (EST != EST_EXACT);
  static constexpr bool MIL = (SCHEME == 1);
  static constexpr int PHI_OCT = EST == EST_CORR ? PHI_OCT_CORR : PHI_OCT_EXACT;
  // the calls of a path share the first Philox rounds' constants (PhiloxStream);
  // most packed kernels, whose calls feed three samples, keep the registers
  static constexpr bool STREAM = KP == 1 || (AP == AP_FX32 && SCHEME == 0 && PC == PC_TERMINAL);
  static constexpr bool PERM = EST == EST_CORR && MSEL >= 2;   // Method 2's coupling of the exact path
  static constexpr bool FAST = (AP == AP_FX32 || AP == AP_FX64);
  static constexpr bool FIXED = (AP == AP_FIXED || FAST);
  static constexpr bool HALF = (AP == AP_F16 || AP == AP_BF16 || AP == AP_F16S || AP == AP_BF16S);
  // half increments with S (and its average and minimum) in FP32
  static constexpr bool S32 = (AP == AP_F16S || AP == AP_BF16S);
  // Half arithmetic on two lanes at once, in paired (x2) registers: lanes 0 and 1
  // of packed draws (lane 2 is scalar), or two samples of one thread with words
  // of their own (DUO, KP = 2).  The half instructions run on the pipe of the
  // integer multiplies, at its rate whether they hold one value or two.
  static constexpr bool DUO = HALF && KP == 2;
  static constexpr bool PAIR = HALF && KP >= 2 && !S32;
  using AS = typename std::conditional<AP == AP_FX32, int32_t, int64_t>::type;  // fixed-point S
  // saturation flag of the fast datapath: OR of (clamped ^ unclamped) for a 32-bit S
  using SatT = typename std::conditional<AP == AP_FX32, uint32_t, bool>::type;
  // 32-bit datapath: when the host proved it exact (ff.lazy), a group of packs
  // (or a correction's samples) first runs with S unclamped, tracking only its running
  // maximum hi; if hi stayed at or below lim_S no clamp would have acted and the
  // values are final, otherwise the group runs again on the clamped (EAGER)
  // datapath.
  static constexpr bool LAZY = (AP == AP_FX32 && (EST == EST_APPROX || EST == EST_CORR));
  static constexpr bool P32 = AP == AP_FX32 && PRE && !MIL;   // the table holds P_j only
  static constexpr int KPV = KP;
  static constexpr int ESTV = EST;
  using X = typename XType<XP>::T;
  using H = typename HType<AP>::T;
  using HO = HalfOps<H>;
  using HO2 = HalfOps2<H>;
  using H2 = typename HO2::T;
  using HS = typename std::conditional<S32, float, H>::type;   // S of the half datapaths
  static __device__ __forceinline__ float sf(float x) { return x; }
  static __device__ __forceinline__ float sf(H x) { return HO::to_f(x); }

  // ---- per-item constants (registers) ----
  int level, nsteps, payoff, d, dshift, method;
  // FX32: byte offset of lane l's table entry = rotr(word, rot[l]) & off_mask
  // PRE: 2^(32 - rs2); radd2 times it; what the fine and the coarse step's sum1
  // add to mul1, times it
  int32_t pre2, c1p, c1cp;
  int64_t radd2p;
  static constexpr int LG = P32 ? 2 : 3;   // log2 of a table entry's bytes
  uint32_t rot[KP], off_mask;
  const uint16_t *perm_s;  // method 2 coupling of the exact path (shared memory), or nullptr
  const float4 *phi;       // FP32 exact path: the inverse-Normal cubics in shared memory
  uint32_t phil;           // and this lane's copy (PhiTable::lane)
  uint32_t low_mask;
  X c1, c2, c1c, c3, S0, K;
  // FP64 exact path: integer increments (exact64.cuh)
  int64_t q1;
  uint64_t q2, q3;
  int qF;
  uint32_t qhi;            // q_to_double's exponent word
  const ulonglong2 *phi64;
  // fixed point
  FixedConsts fx;
  FastFixed ff;
  // half
  H hc1, hc1c, hc2, hc3;
  HS hS0;
  H2 pc1, pc1c, pc2, pc3;
  float K32;
  float unit_scale;
  const void *smem_tab;

  // ---- per-sample state (approximate state per lane) ----
  X S, Sc, zprev, accF, accC, minF, minC;
  int64_t qprev;           // FP64 exact path: the even step's increment, -Phi^-1 and its sign mask
  uint64_t yprev;
  int32_t mprev;
  AS aS[KP], aSc[KP], aminF[KP], aminC[KP];
  SatT satb[KP];
  AS hi;   // LAZY: running maximum of S over a group's lanes and steps (reset by the caller)
  int64_t aaccF[KP], aaccC[KP];
  int32_t azprev[KP];
  HS hS[KP], hSc[KP], hminF[KP], hminC[KP];
  H hzprev[KP];
  H2 pS, pSc, pzprev;   // lanes 0 and 1 when PAIR (hS[0..1] etc. then unused)
  float haccF[KP], haccC[KP];
  uint32_t sat[KP];

  __device__ __forceinline__ void load(const ItemDesc &it, const void *tab) {
    level = it.level;
    nsteps = 1 << it.level;
    payoff = it.payoff;
    d = it.d;
    dshift = 32 - it.d;
    method = it.method;
    if constexpr (XP == XP_F64) {
      c1 = it.c1d; c2 = it.c2d; c1c = it.c1cd; c3 = it.c3d; S0 = it.S0d; K = it.Kd + 0.0;   // +0 for a strike of -0 (above_f64)
      q1 = it.q1; q2 = it.q2; q3 = it.q3; qF = it.qF; qhi = (uint32_t)(1085 - it.qF) << 20;
      phi64 = phi64_smem();
    } else {
      c1 = it.c1f; c2 = it.c2f; c1c = it.c1cf; c3 = it.c3f; S0 = it.S0f; K = it.Kf;
    }
    if constexpr (FIXED) fx = it.fx;
    if constexpr (FAST) ff = it.ff;
    if constexpr (AP == AP_FX32 && PRE) {
      pre2 = 1 << (32 - it.ff.rs2);
      radd2p = (int64_t)((uint64_t)it.ff.radd2 << (32 - it.ff.rs2));
      c1p = (int32_t)((uint32_t)(it.ff.con1r >> it.ff.rs_sum1) << (32 - it.ff.rs2));
      c1cp = (int32_t)((uint32_t)(it.ff.con1cr >> it.ff.rs_sum1) << (32 - it.ff.rs2));
    }
    if constexpr (HALF) {
      hc1 = HO::from_bits(it.h_c1); hc1c = HO::from_bits(it.h_c1c);
      hc2 = HO::from_bits(it.h_c2); hc3 = HO::from_bits(it.h_c3);
      if constexpr (S32) hS0 = it.S0f;
      else hS0 = HO::from_bits(it.h_S0);
      K32 = it.Kf;
      if constexpr (PAIR || DUO) {
        pc1 = HO2::splat(hc1); pc1c = HO2::splat(hc1c); pc2 = HO2::splat(hc2); pc3 = HO2::splat(hc3);
      }
    }
    unit_scale = it.unit_scale;
    smem_tab = tab;
    if constexpr (AP == AP_FX32) {
      // lane l's field, bits [32 - d(l+1), 32 - d l) of the word, lands at bits [LG, LG + d)
#pragma unroll
      for (int l = 0; l < KP; ++l) rot[l] = (uint32_t)(32 - it.d * (l + 1) - LG) & 31u;
      off_mask = ((1u << it.d) - 1u) << LG;
    }
    perm_s = nullptr;
    if constexpr (HAS_EXACT && XP == XP_F32) {
      phi = phi_inv_smem<PHI_OCT>();
      phil = PhiTable<PHI_OCT>::lane();
    }
    low_mask = (1u << dshift) - 1u;
    if constexpr (PERM) {
      if (it.perm) perm_s = (const uint16_t *)((const unsigned char *)tab + ((size_t)1 << it.d) * TabBytes<AP>::value);
    }
  }

  __device__ __forceinline__ void begin() {
    if constexpr (HAS_EXACT) {
      S = S0; Sc = S0; zprev = X(0);
      accF = X(0.5) * S0; accC = accF; minF = S0; minC = S0;
    }
#pragma unroll
    for (int l = 0; l < KP; ++l) {
      if constexpr (FIXED) {
        aS[l] = (AS)fx.S0; aSc[l] = (AS)fx.S0; aaccF[l] = 0; aaccC[l] = 0; aminF[l] = aS[l]; aminC[l] = aS[l];
        azprev[l] = 0;
        satb[l] = SatT(0);
      }
      if constexpr (HALF) {
        hS[l] = hS0; hSc[l] = hS0; hzprev[l] = HO::from_f(0.0f); hminF[l] = hS0; hminC[l] = hS0;
        haccF[l] = __fmul_rn(0.5f, sf(hS0)); haccC[l] = haccF[l];
      }
      sat[l] = 0;
    }
    if constexpr (PAIR) {
      pS = HO2::splat(hS0); pSc = pS;
    }
    if constexpr (PAIR || DUO) pzprev = HO2::splat(HO::from_f(0.0f));
  }
  // LAZY: did some S since hi was reset leave [-lim_S, lim_S]?  (The host
  // proved that it cannot leave below first.)
  __device__ __forceinline__ bool over() const { return hi > (AS)ff.limT; }

  // Asian sums leave out S_0 (the first step's S, and the first coarse step's): zero is
  // added there instead of branching round the sum.  As branches they cut the step loop
  // into blocks whose steps ran one after another: 8,000 level-10 corrections 92 -> 68 us,
  // Method 2's 108 -> 80; 1.5e7 level-4 ones 568 -> 523.  The binary16 / bfloat16 and
  // the FP32 exact kernels keep the branch: Method 2's binary16 corrections 70 against
  // 75 us, 1.5e7 level-4 FP32 samples 343 against 350.
  static constexpr bool BRANCH_INNER = HALF || (EST == EST_EXACT && XP == XP_F32);

  // ---- exact path (FP32 / FP64) ----
  static __device__ __forceinline__ X lower(X a, X b) {
    if constexpr (XP == XP_F64) return min_f64(b, a);
    else return fmin(a, b);
  }
  static __device__ __forceinline__ bool above(X a, X b) {   // a > b, b >= 0
    if constexpr (XP == XP_F64) return above_f64(a, b);
    else return a > b;
  }
  __device__ __forceinline__ X exact_inc(X z, X cc1, X mm) const {
    if constexpr (MIL) return fma(c3, fma(z, z, -mm), fma(c2, z, cc1));
    else return fma(c2, z, cc1);
  }

  // ---- fixed-point Algorithm-1 step ----
  __device__ __forceinline__ int64_t fx_step(int64_t s, int32_t z, int64_t con1A, int m, uint32_t &sat) {
    const int64_t mul1 = saturate(requant((int64_t)fx.con2 * z, fx.q_mul1), fx.lim[3], sat);
    int64_t acc = con1A + (int64_t)((uint64_t)mul1 << fx.sh_mul1_F1);
    if constexpr (MIL) {
      const int64_t zz = (int64_t)z * z - ((int64_t)m << fx.fZ2);
      const int64_t mul3 = saturate(requant((int64_t)fx.con3 * zz, fx.q_mul3), fx.lim[3], sat);
      acc += (int64_t)((uint64_t)mul3 << fx.sh_mul1_F1);
    }
    const int64_t sum1 = saturate(requant(acc, fx.q_sum1), fx.lim[4], sat);
    const int64_t mul2 = saturate(requant(s * sum1, fx.q_mul2), fx.lim[5], sat);
    const int64_t s2 = (int64_t)((uint64_t)s << fx.sh_S_F2) + (int64_t)((uint64_t)mul2 << fx.sh_mul2_F2);
    return saturate(requant(s2, fx.q_S), fx.lim[6], sat);
  }

  // ---- fast fixed-point Algorithm-1 step (same values as fx_step while S stays in range) ----
  // The S update of a step whose sum1 is known: mul2 = rd(S sum1), S = rd(S + mul2).
  // TRACK (lazy runs): count this S in the pack's maximum (fast_fixed's limT)
  template <bool EAGER, bool TRACK = true>
  __device__ __forceinline__ AS ff_apply(AS s, int32_t sum1, SatT &satb) {
    if constexpr (AP == AP_FX32 && PRE) {
      const int64_t p2 = (int64_t)s * sum1 + radd2p;
      const int32_t mul2 = (int32_t)((uint64_t)p2 >> 32);
      s = (int32_t)((uint32_t)s + (uint32_t)mul2 * (uint32_t)ff.mulS);
    } else if constexpr (AP == AP_FX32) {
      const int64_t p2 = (int64_t)s * sum1 + ff.radd2;
      const int32_t mul2 = (int32_t)__funnelshift_r((uint32_t)p2, (uint32_t)((uint64_t)p2 >> 32), ff.rs2);
      s = (int32_t)((uint32_t)s + (uint32_t)mul2 * (uint32_t)ff.mulS);
    } else {
      const int32_t mul2 = (int32_t)((int64_t)((uint64_t)s * (uint64_t)(int64_t)sum1 + (uint64_t)ff.radd2) >> ff.rs2);
      s = (int64_t)((uint64_t)s + (uint64_t)((int64_t)mul2 * ff.mulS));
    }
    if constexpr (LAZY && !EAGER) {
      if constexpr (TRACK) hi = max(hi, s);
      return s;
    }
    // saturation of S (the only variable the host could not bound)
    const AS lim = (AS)ff.limS;
    const AS c = min(max(s, -lim), lim);
    if constexpr (AP == AP_FX32) satb |= (uint32_t)(c ^ s);
    else satb |= (c != s);
    return c;
  }
  template <bool EAGER>
  __device__ __forceinline__ AS ff_step(AS s, int32_t z, int32_t c1r, int64_t m, SatT &satb) {
    return ff_apply<EAGER>(s, ff_sum1<MIL, AP == AP_FX32>(ff, z, c1r, m), satb);
  }
  // FX32: lane l's table entry for word w.  Lane 0's field (and the only one of an
  // unpacked word) is the top one: no mask.  The table sits at the start of the
  // dynamic shared memory: addressing it there, rather than through smem_tab,
  // leaves the base to the load's immediate offset, one add fewer per lookup.
  // SH: log2 of the entry's bytes in the table read.
  template <class E, int SH = LG>
  __device__ __forceinline__ E fx32_entry(uint32_t w, int l) const {
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    if (l == 0) return ((const E *)smem_dyn)[w >> dshift];
    return *(const E *)(smem_dyn + ((__funnelshift_r(w, w, rot[l]) & off_mask) >> (LG - SH)));
  }
  // The FX32 fine step of lane l on word w; returns what the coarse step needs of
  // it (Z~, or P_j).  TRACK as in ff_apply.
  template <bool EAGER, bool TRACK>
  __device__ __forceinline__ int32_t fx32_fine(uint32_t w, int l) {
    if constexpr (P32) {
      const int32_t q = fx32_entry<int32_t>(w, l);
      aS[l] = ff_apply<EAGER, TRACK>(aS[l], (q >> ff.rs1) * pre2 + c1p, satb[l]);
      return q;
    } else {
      const int2 e = fx32_entry<int2>(w, l);
      aS[l] = ff_apply<EAGER, TRACK>(aS[l], e.y, satb[l]);
      return e.x;
    }
  }
  // The FX32 coarse step from the two fine steps' values.
  template <bool EAGER>
  __device__ __forceinline__ void fx32_coarse(int l, int32_t x0, int32_t x1) {
    if constexpr (P32) {
      const int32_t q = x0 + x1 - (int32_t)ff.radd1;
      aSc[l] = ff_apply<EAGER>(aSc[l], (q >> ff.rs1) * pre2 + c1cp, satb[l]);
    } else if constexpr (PRE) {
      const int32_t z = x0 + x1;
      const int64_t p1 = (int64_t)ff.con2 * z + ff.radd1;
      const int64_t p3 = (int64_t)ff.con3 * (z * z - (int32_t)ff.mcoarse) + ff.radd3;
      const int32_t mul = (int32_t)__funnelshift_r((uint32_t)p1, (uint32_t)((uint64_t)p1 >> 32), ff.rs1) +
                          (int32_t)__funnelshift_r((uint32_t)p3, (uint32_t)((uint64_t)p3 >> 32), ff.rs3);
      aSc[l] = ff_apply<EAGER>(aSc[l], mul * pre2 + c1cp, satb[l]);
    } else {
      aSc[l] = ff_step<EAGER>(aSc[l], x0 + x1, ff.con1cr, ff.mcoarse, satb[l]);
    }
  }

  // ---- half-precision step (one rounding per operation) ----
  // With S32 only the increment sum1 is in half precision; S is updated in
  // FP32 (mul2 = fl32(S sum1), S = fl32(S + mul2)).
  __device__ __forceinline__ HS h_step(HS s, H z, H cc1, H mh) const {
    const H mul1 = HO::mul(hc2, z);
    H sum1 = HO::add(cc1, mul1);
    if constexpr (MIL) {
      const H sq = HO::mul(z, z);
      const H sqm = HO::sub(sq, mh);
      const H mul3 = HO::mul(hc3, sqm);
      sum1 = HO::add(sum1, mul3);
    }
    if constexpr (S32) {
      return __fadd_rn(s, __fmul_rn(s, HO::to_f(sum1)));
    } else {
      const H mul2 = HO::mul(s, sum1);
      return HO::add(s, mul2);
    }
  }
  // the same on two lanes at once: the increment, and the step
  __device__ __forceinline__ H2 h2_inc(H2 z, H2 cc1, H2 mh) const {
    const H2 mul1 = HO2::mul(pc2, z);
    H2 sum1 = HO2::add(cc1, mul1);
    if constexpr (MIL) {
      const H2 sq = HO2::mul(z, z);
      const H2 sqm = HO2::sub(sq, mh);
      const H2 mul3 = HO2::mul(pc3, sqm);
      sum1 = HO2::add(sum1, mul3);
    }
    return sum1;
  }
  __device__ __forceinline__ H2 h2_step(H2 s, H2 z, H2 cc1, H2 mh) const {
    return HO2::add(s, HO2::mul(s, h2_inc(z, cc1, mh)));
  }
  // lane l's half state (fine / coarse)
  __device__ __forceinline__ HS lane_S(int l) const {
    if constexpr (PAIR) { if (l == 0) return HO2::lo(pS); if (l == 1) return HO2::hi(pS); }
    return hS[l];
  }
  __device__ __forceinline__ HS lane_Sc(int l) const {
    if constexpr (PAIR) { if (l == 0) return HO2::lo(pSc); if (l == 1) return HO2::hi(pSc); }
    return hSc[l];
  }
  __device__ __forceinline__ static void lane_min(HS &mn, HS x) { mn = sf(x) < sf(mn) ? x : mn; }

  // Approximate Normal of J in Z's fixed-point format: Method 1 reads the
  // signed table at j = top d bits of J; Method 3 evaluates the class line.
  __device__ __forceinline__ int32_t fixed_z(uint32_t J) const {
    if constexpr (MSEL == 0 || MSEL == 4) return ((const int32_t *)smem_tab)[J >> dshift];
    if constexpr (MSEL == 2) {
      if (method != 3) return ((const int32_t *)smem_tab)[J >> dshift];
    }
    const ApproxIndex ai = approx_index(J, d);
    int32_t v;
    {
      const M3Coef *m3 = (const M3Coef *)smem_tab;
      const int c = m3_class(ai.idx);
      const int64_t t = m3->A[c] + m3->B[c] * (int64_t)ai.idx;
      const int sh = M3_FRAC - fx.fZ2 / 2;
      v = (int32_t)((t + ((int64_t)1 << (sh - 1))) >> sh);
    }
    return ai.neg ? -v : v;
  }

  __device__ __forceinline__ H half_z(uint32_t J) const {
    if constexpr (MSEL == 0 || MSEL == 4) return HO::from_bits(((const uint16_t *)smem_tab)[J >> dshift]);
    if constexpr (MSEL == 2) {
      if (method != 3) return HO::from_bits(((const uint16_t *)smem_tab)[J >> dshift]);
    }
    const ApproxIndex ai = approx_index(J, d);
    H v;
    {
      const M3Coef *m3 = (const M3Coef *)smem_tab;
      const int c = m3_class(ai.idx);
      v = HO::from_f(fmaf(m3->b[c], (float)ai.idx, m3->a[c]));
    }
    return ai.neg ? HO::neg(v) : v;
  }

  // One fine step i driven by J, and the coarse step after odd i (levels >= 1).
  // PAR: parity of i when known at compile time (0 even, 1 odd), -1 otherwise.
  // J1: the second sample's word (DUO).
  template <bool COARSE, int PAR = -1, bool EAGER = true>
  __device__ __forceinline__ void step(uint32_t J, int i, uint32_t J1 = 0) {
    const bool odd = PAR >= 0 ? (PAR == 1) : ((i & 1) != 0);
    if constexpr (HAS_EXACT) {
      // Method 2 (Sec. 3.2): the exact path takes the uniform in the interval
      // pi(j) that the approximate value of j is ranked at, with J's low bits
      uint32_t Je = J;
      if constexpr (PERM) {
        if (MSEL != 2 || perm_s) Je = ((uint32_t)perm_s[J >> dshift] << dshift) | (J & low_mask);
      }
      X z, inc;
      int64_t qi = 0;
      uint64_t y = 0;
      int32_t m = 0;
      const bool qinc = XP == XP_F64 && (MSEL == 2 ? qF != 0 : MSEL == 0);
      if constexpr (XP == XP_F64) {
        m = (int32_t)Je >> 31;   // Z = y in the upper half, -y below
        y = probit_q60(Je ^ (uint32_t)m, phi64);
        if (qinc) {
          // c2 Z = +-c2 y, the negative as the complement (one unit 2^-qF off)
          qi = q1 + (int64_t)(mulhi64_3(q2, y) ^ (uint64_t)(int64_t)~m);
          if constexpr (MIL) qi += (int64_t)mulhi64_3(q3, mulhi64_3(y, y));
          inc = q_to_double(qi, qhi);
        } else {
          z = q_to_double((int64_t)(y ^ (uint64_t)(int64_t)~m), (uint32_t)(1085 - 60) << 20);
          inc = exact_inc(z, c1, X(1));
        }
      } else {
        z = exact_normal_f32<PHI_OCT>(Je, phi, phil);
        inc = exact_inc(z, c1, X(1));
      }
      if constexpr (PC == PC_ASIAN) { if (!BRANCH_INNER || i > 0) accF = accF + (BRANCH_INNER || i > 0 ? S : X(0)); }
      S = fma(S, inc, S);
      if constexpr (PC == PC_LOOKBACK) minF = lower(minF, S);
      if constexpr (COARSE) {
        if (odd) {
          if constexpr (PC == PC_ASIAN) { if (!BRANCH_INNER || i > 1) accC = accC + (BRANCH_INNER || i > 1 ? Sc : X(0)); }
          if (qinc) {
            // c1_c = 2 c1 and (Z + Z')^2 - 2 = (Z^2 - 1) + (Z'^2 - 1) + 2 Z Z': the coarse
            // increment is the sum of the two fine ones (Milstein: + 2 c3 Z Z')
            int64_t qc = qprev + qi;
            if constexpr (MIL) {
              const uint64_t x = mulhi64_3(q3, mulhi64_3(yprev, y)) << 1;
              const uint64_t sg = (uint64_t)(int64_t)(mprev ^ m);
              qc += (int64_t)(x ^ sg);
            }
            inc = q_to_double(qc, qhi);
          } else {
            inc = exact_inc(zprev + z, c1c, X(2));
          }
          Sc = fma(Sc, inc, Sc);
          if constexpr (PC == PC_LOOKBACK) minC = lower(minC, Sc);
        } else if (qinc) {
          qprev = qi;
          yprev = y;
          mprev = m;
        } else {
          zprev = z;
        }
      }
    }
    if constexpr (PAIR) {
      // Algorithm-1 arithmetic of lanes 0 and 1 in paired instructions; lane 2 alone
      constexpr bool THIRD = KP == 3;
      const H2 z01 = HO2::pack(half_z(J), half_z(DUO ? J1 : J << d));
      H z2 = HO::from_f(0.0f);
      if constexpr (THIRD) z2 = half_z(J << (2 * d));
      if constexpr (PC == PC_ASIAN) {
        if (i > 0) {
          haccF[0] = __fadd_rn(haccF[0], HO::to_f(HO2::lo(pS)));
          haccF[1] = __fadd_rn(haccF[1], HO::to_f(HO2::hi(pS)));
          if constexpr (THIRD) haccF[2] = __fadd_rn(haccF[2], HO::to_f(hS[2]));
        }
      }
      pS = h2_step(pS, z01, pc1, HO2::splat(HO::from_f(1.0f)));
      if constexpr (THIRD) hS[2] = h_step(hS[2], z2, hc1, HO::from_f(1.0f));
      if constexpr (PC == PC_LOOKBACK) {
        lane_min(hminF[0], HO2::lo(pS)); lane_min(hminF[1], HO2::hi(pS));
        if constexpr (THIRD) lane_min(hminF[2], hS[2]);
      }
      if constexpr (COARSE) {
        if (odd) {
          const H2 zc01 = HO2::add(pzprev, z01);
          if constexpr (PC == PC_ASIAN) {
            if (i > 1) {
              haccC[0] = __fadd_rn(haccC[0], HO::to_f(HO2::lo(pSc)));
              haccC[1] = __fadd_rn(haccC[1], HO::to_f(HO2::hi(pSc)));
              if constexpr (THIRD) haccC[2] = __fadd_rn(haccC[2], HO::to_f(hSc[2]));
            }
          }
          pSc = h2_step(pSc, zc01, pc1c, HO2::splat(HO::from_f(2.0f)));
          if constexpr (THIRD) hSc[2] = h_step(hSc[2], HO::add(hzprev[2], z2), hc1c, HO::from_f(2.0f));
          if constexpr (PC == PC_LOOKBACK) {
            lane_min(hminC[0], HO2::lo(pSc)); lane_min(hminC[1], HO2::hi(pSc));
            if constexpr (THIRD) lane_min(hminC[2], hSc[2]);
          }
        } else {
          pzprev = z01;
          if constexpr (THIRD) hzprev[2] = z2;
        }
      }
    } else if constexpr (DUO) {
      // the increments of both samples in paired instructions, their FP32 S apart
      auto apply = [&](HS *s, H2 inc) {
        s[0] = __fadd_rn(s[0], __fmul_rn(s[0], HO::to_f(HO2::lo(inc))));
        s[1] = __fadd_rn(s[1], __fmul_rn(s[1], HO::to_f(HO2::hi(inc))));
      };
      const H2 z01 = HO2::pack(half_z(J), half_z(J1));
      if constexpr (PC == PC_ASIAN) {
        if (i > 0) {
          haccF[0] = __fadd_rn(haccF[0], sf(hS[0]));
          haccF[1] = __fadd_rn(haccF[1], sf(hS[1]));
        }
      }
      apply(hS, h2_inc(z01, pc1, HO2::splat(HO::from_f(1.0f))));
      if constexpr (PC == PC_LOOKBACK) { lane_min(hminF[0], hS[0]); lane_min(hminF[1], hS[1]); }
      if constexpr (COARSE) {
        if (odd) {
          if constexpr (PC == PC_ASIAN) {
            if (i > 1) {
              haccC[0] = __fadd_rn(haccC[0], sf(hSc[0]));
              haccC[1] = __fadd_rn(haccC[1], sf(hSc[1]));
            }
          }
          apply(hSc, h2_inc(HO2::add(pzprev, z01), pc1c, HO2::splat(HO::from_f(2.0f))));
          if constexpr (PC == PC_LOOKBACK) { lane_min(hminC[0], hSc[0]); lane_min(hminC[1], hSc[1]); }
        } else {
          pzprev = z01;
        }
      }
    } else if constexpr (AP == AP_FX32) {
      // the fine step's sum1 comes with Z~ from the table; the coarse step forms
      // its own from Z~_2k + Z~_2k+1
#pragma unroll
      for (int l = 0; l < KP; ++l) {
        if constexpr (PC == PC_ASIAN) aaccF[l] += i > 0 ? aS[l] : 0;
        // lazy runs track S after the odd fine steps only (limT); with the parity
        // unknown at compile time, after every step (more is as exact)
        constexpr bool TRACK_FINE = PAR == 1 || (PAR == -1 && COARSE);
        const int32_t x = fx32_fine<EAGER, TRACK_FINE>(J, l);
        if constexpr (PC == PC_LOOKBACK) aminF[l] = aS[l] < aminF[l] ? aS[l] : aminF[l];
        if constexpr (COARSE) {
          if (odd) {
            if constexpr (PC == PC_ASIAN) aaccC[l] += i > 1 ? aSc[l] : 0;
            fx32_coarse<EAGER>(l, azprev[l], x);
            if constexpr (PC == PC_LOOKBACK) aminC[l] = aSc[l] < aminC[l] ? aSc[l] : aminC[l];
          } else {
            azprev[l] = x;
          }
        }
      }
    } else if constexpr (HAS_APPROX) {
#pragma unroll
      for (int l = 0; l < KP; ++l) {
        const uint32_t Jl = l == 0 ? J : (J << (d * l));  // this lane's field at the top
        if constexpr (FIXED) {
          const int32_t z = fixed_z(Jl);
          if constexpr (PC == PC_ASIAN) aaccF[l] += i > 0 ? aS[l] : 0;
          if constexpr (FAST) aS[l] = ff_step<EAGER>(aS[l], z, ff.con1r, ff.mfine, satb[l]);
          else aS[l] = fx_step(aS[l], z, fx.con1A, 1, sat[l]);
          if constexpr (PC == PC_LOOKBACK) aminF[l] = aS[l] < aminF[l] ? aS[l] : aminF[l];
          if constexpr (COARSE) {
            if (odd) {
              if constexpr (PC == PC_ASIAN) aaccC[l] += i > 1 ? aSc[l] : 0;
              if constexpr (FAST) aSc[l] = ff_step<EAGER>(aSc[l], azprev[l] + z, ff.con1cr, ff.mcoarse, satb[l]);
              else aSc[l] = fx_step(aSc[l], azprev[l] + z, fx.con1cA, 2, sat[l]);
              if constexpr (PC == PC_LOOKBACK) aminC[l] = aSc[l] < aminC[l] ? aSc[l] : aminC[l];
            } else {
              azprev[l] = z;
            }
          }
        } else {
          const H z = half_z(Jl);
          if constexpr (PC == PC_ASIAN) { if (i > 0) haccF[l] = __fadd_rn(haccF[l], sf(hS[l])); }
          hS[l] = h_step(hS[l], z, hc1, HO::from_f(1.0f));
          if constexpr (PC == PC_LOOKBACK) lane_min(hminF[l], hS[l]);
          if constexpr (COARSE) {
            if (odd) {
              const H zc = HO::add(hzprev[l], z);
              if constexpr (PC == PC_ASIAN) { if (i > 1) haccC[l] = __fadd_rn(haccC[l], sf(hSc[l])); }
              hSc[l] = h_step(hSc[l], zc, hc1c, HO::from_f(2.0f));
              if constexpr (PC == PC_LOOKBACK) lane_min(hminC[l], hSc[l]);
            } else {
              hzprev[l] = z;
            }
          }
        }
      }
    }
  }

  // ---- payoffs ----
  // lg: log2 of the path's steps
  template <int PAY = -1>
  __device__ __forceinline__ X exact_payoff(X x, X acc, X mn, int lg) const {
    if constexpr (PC == PC_TERMINAL) {
      if (PAY >= 0 ? PAY == 1 : payoff == 1) return above(x, K) ? X(1) : X(0);
      const X dd = x - K;
      return above(dd, X(0)) ? dd : X(0);
    } else if constexpr (PC == PC_ASIAN) {
      // one explicit multiply-add: every instantiation rounds the average alike
      const X avg = fma(X(0.5), x, acc) * pow2_neg(lg);
      const X dd = avg - K;
      return above(dd, X(0)) ? dd : X(0);
    } else {
      return x - mn;
    }
  }
  // 2^-lg (an FP64 division would cost more than the payoff)
  static __device__ __forceinline__ X pow2_neg(int lg) {
    if constexpr (XP == XP_F64) return __hiloint2double((1023 - lg) << 20, 0);
    else return __int_as_float((127 - lg) << 23);
  }
  // PAY: the terminal payoff when known at compile time (0 European, 1 digital), -1 otherwise
  template <int PAY = -1>
  __device__ __forceinline__ int64_t fixed_payoff(int64_t x, int64_t inner, int64_t mn, int steps, bool coarse) const {
    if constexpr (PC == PC_TERMINAL && AP == AP_FX32) {
      // S, K < 2^31 on this datapath: 32-bit arithmetic
      const int32_t x32 = (int32_t)x, K32v = (int32_t)fx.K;
      const bool digital = PAY >= 0 ? PAY == 1 : payoff == 1;
      const int32_t v = digital ? (int32_t)1 << fx.fS : x32 - K32v;
      return x32 > K32v ? v : 0;
    } else if constexpr (PC == PC_TERMINAL) {
      if (payoff == 1) return x > fx.K ? ((int64_t)1 << fx.fS) : 0;
      return x > fx.K ? x - fx.K : 0;
    } else if constexpr (PC == PC_ASIAN) {
      const int64_t twice = fx.S0 + 2 * inner + x;
      const int64_t twoNK = 2 * (int64_t)steps * fx.K;
      const int64_t v = twice > twoNK ? twice - twoNK : 0;
      return coarse ? 2 * v : v;
    } else {
      return x - mn;
    }
  }
  __device__ __forceinline__ int64_t half_payoff(HS x, float acc, HS mn, int steps) const {
    float P;
    const float xf = sf(x);
    if constexpr (PC == PC_TERMINAL) {
      if (payoff == 1) {
        P = xf > K32 ? 1.0f : 0.0f;
      } else {
        const float dd = __fsub_rn(xf, K32);
        P = dd > 0.0f ? dd : 0.0f;
      }
    } else if constexpr (PC == PC_ASIAN) {
      const float tot = __fadd_rn(acc, __fmul_rn(0.5f, xf));
      const float avg = __fmul_rn(tot, 1.0f / (float)steps);
      const float dd = __fsub_rn(avg, K32);
      P = dd > 0.0f ? dd : 0.0f;
    } else {
      P = __fsub_rn(xf, sf(mn));
    }
    return __float2ll_rn(__fmul_rn(P, 16777216.0f));
  }

  // Finish the sample: payoffs, sample value, accumulation and optional dump
  // (EAGER false: a LAZY pack that stayed in range, so no saturation).
  // LV: 0 on level 0 (no coarse path), 1 on levels >= 1, -1 not known at compile time.
  // PAIRED: real samples are taken two at a time (levels 0 and 1; ThreadAcc).
  template <bool EAGER = true, int PAY = -1, int LV = -1, bool PAIRED = false, class Acc>
  __device__ __forceinline__ void finish(Acc &acc, int l, bool valid, mlmc_sample_rec *dump) {
    X pf = X(0), pc = X(0);
    int64_t qf = 0, qc = 0, afS = 0, acS = 0;
    uint32_t lsat = 0;
    const bool coarse = LV >= 0 ? LV == 1 : level > 0;
    if constexpr (HAS_EXACT) {
      pf = exact_payoff<PAY>(S, accF, minF, level);
      if (coarse) pc = exact_payoff<PAY>(Sc, accC, minC, level - 1);
    }
    if constexpr (FIXED) {
      qf = fixed_payoff<PAY>(aS[l], aaccF[l], aminF[l], nsteps, false);
      if (coarse) qc = fixed_payoff<PAY>(aSc[l], aaccC[l], aminC[l], nsteps >> 1, true);
      afS = aS[l];
      acS = aSc[l];
      if constexpr (FAST) lsat = (EAGER && satb[l]) ? 1u : 0u;
      else lsat = sat[l];
    }
    if constexpr (HALF) {
      if constexpr (HAS_APPROX) {
        qf = half_payoff(lane_S(l), haccF[l], hminF[l], nsteps);
        if (coarse) qc = half_payoff(lane_Sc(l), haccC[l], hminC[l], nsteps >> 1);
      }
    }
    double ydump;
    if constexpr (EST == EST_APPROX && AP == AP_FX32 && PC == PC_TERMINAL) {
      // a sample outside the item's range adds zero to the group sums, so the
      // range test does not branch the group's straight-line code (|Y| < 2^31
      // here and the host bounds a group's sum of squares below 2^64)
      const int32_t yi = valid ? (int32_t)(qf - qc) : 0;
      acc.add_group(yi);
      acc.nsat += valid ? lsat : 0u;
      if (!valid) return;
      ydump = (double)yi * (double)unit_scale;
    } else if constexpr (EST == EST_APPROX) {
      if (!valid) return;
      const int64_t yi = qf - qc;
      acc.add_int(yi);
      acc.nsat += lsat;
      ydump = (double)yi * (double)unit_scale;
    } else {
      // a sample outside the item's range adds zero: no branch
      if constexpr (EST == EST_EXACT) {
        const X y = valid ? pf - pc : X(0);
        acc.template add_real<PAIRED>(y);
        ydump = (double)y;
      } else {
        const float yx = (float)(pf - pc);
        const float ya = __fmul_rn(__ll2float_rn(qf - qc), unit_scale);
        const float y = valid ? __fsub_rn(yx, ya) : 0.0f;
        acc.template add_real<PAIRED>(y);
        ydump = (double)y;
      }
      acc.nsat += valid ? lsat : 0u;
      if (!valid) return;
    }
    if (dump) {
      mlmc_sample_rec r;
      r.pf = (double)pf; r.pc = (double)pc;
      r.sf = HAS_EXACT ? (double)S : 0.0;
      r.sc = (HAS_EXACT && level > 0) ? (double)Sc : 0.0;
      if constexpr (FIXED) {
        r.af = ldexp((double)afS, -fx.fS);
        r.ac = level > 0 ? ldexp((double)acS, -fx.fS) : 0.0;
      } else if constexpr (HALF) {
        r.af = HAS_APPROX ? (double)sf(lane_S(l)) : 0.0;
        r.ac = (HAS_APPROX && level > 0) ? (double)sf(lane_Sc(l)) : 0.0;
      } else {
        r.af = 0.0; r.ac = 0.0;
      }
      r.qf = qf; r.qc = qc; r.y = ydump; r.sat = lsat; r.pad = 0;
      *dump = r;
    }
  }
};

// Two floats in one 64-bit register pair and the instructions on both at once
// (each result rounded as the scalar operation's): half the issue slots.
struct F2 {
  uint64_t v;
  static __device__ __forceinline__ F2 of(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
  }
  __device__ __forceinline__ void get(float &a, float &b) const { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
};
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// a - b, exactly as a subtraction: -1 b + a is one rounding of a - b.
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { return fma2(F2{0xBF800000BF800000ULL}, b, a); }

// Samples of an FP32 real-valued estimator summed in a float pair before each
// FP64 flush: levels >= 2, and pairs of samples on levels 0 and 1 (see
// ThreadAcc::add_real).
constexpr int REAL_FLUSH_SAMPLES = 8, REAL_FLUSH_PAIRS = 6;

// Per-thread accumulator
template <int EST, int XP>
struct ThreadAcc {
  // integer estimators
  int64_t isum;
  uint64_t q_lo, q_hi;
  // real-valued estimators: FP64 sums (FP64 exact path: every sample; FP32
  // paths and corrections: the float pairs below, flushed)
  double ds, dq;
  // float pairs (s + c) of sum Y and sum Y^2 since the last flush: one of each
  // (os, oc, os2, oc2), or two, of every first and of every second sample
  float os, oc, os2, oc2;
  F2 fs, fc, fs2, fc2;
  float first;             // a first sample that waits for its second (have)
  bool have;
  uint32_t nsat;
  __device__ __forceinline__ void init() {
    isum = 0; q_lo = 0; q_hi = 0; gsum = 0; gq = 0; ds = 0.0; dq = 0.0; nsat = 0;
    os = 0.0f; oc = 0.0f; os2 = 0.0f; oc2 = 0.0f;
    fs = F2{0}; fc = fs; fs2 = fs; fc2 = fs; first = 0.0f; have = false;
  }
  __device__ __forceinline__ void add_int(int64_t y) {
    isum += y;
    add_square(q_lo, q_hi, y);
  }
  // Two wide multiply-adds per sample (FMA pipe): the group's sum of y and of
  // y^2 in 64 bits; flush_group() adds them into the totals (and
  // discard_group() drops a group that must be redone).
  int64_t gsum;
  uint64_t gq;
  __device__ __forceinline__ void add_group(int32_t y) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(gsum) : "r"(y), "r"(1));
    asm("mad.wide.s32 %0, %1, %1, %0;" : "+l"(gq) : "r"(y));
  }
  // two samples, 0 <= y <= 2^30 (payoffs of a 32-bit S): their sum fits 32 bits
  __device__ __forceinline__ void add_group2(int32_t y0, int32_t y1) {
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(gsum) : "r"((uint32_t)y0 + (uint32_t)y1), "r"(1));
    asm("mad.wide.s32 %0, %1, %1, %0;" : "+l"(gq) : "r"(y0));
    asm("mad.wide.s32 %0, %1, %1, %0;" : "+l"(gq) : "r"(y1));
  }
  __device__ __forceinline__ void flush_group() {
    isum += gsum;
    add_u128(q_lo, q_hi, gq, 0);
    gsum = 0;
    gq = 0;
  }
  __device__ __forceinline__ void discard_group() {
    gsum = 0;
    gq = 0;
  }
  // Sums at the start of a group, to undo the group's samples (the
  // path-dependent payoffs and the corrections add each sample directly).
  struct Mark {
    int64_t isum;
    uint64_t q_lo, q_hi;
    F2 fs, fc, fs2, fc2;
  };
  // (a group of levels 0 and 1 has an even number of samples: none waits there)
  __device__ __forceinline__ Mark mark() const { return Mark{isum, q_lo, q_hi, fs, fc, fs2, fc2}; }
  __device__ __forceinline__ void rewind(const Mark &m) {
    isum = m.isum; q_lo = m.q_lo; q_hi = m.q_hi;
    fs = m.fs; fc = m.fc; fs2 = m.fs2; fc2 = m.fc2; have = false;
  }
  // s + y = t + e exactly (Knuth's TwoSum, six FP32 operations): s becomes t, e is returned.
  static __device__ __forceinline__ F2 two_sum(F2 &s, F2 y) {
    const F2 t = add2(s, y);
    const F2 z = sub2(t, s);
    const F2 e = add2(sub2(s, sub2(t, z)), sub2(y, z));
    s = t;
    return e;
  }
  static __device__ __forceinline__ float two_sum(float &s, float y) {
    const float t = __fadd_rn(s, y);
    const float z = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(y, z));
    s = t;
    return e;
  }
  // A real sample.  FP64 samples are added in FP64.  An FP32 sample y enters the
  // float pair (os, oc) by TwoSum, so os + oc misses sum y only by the roundings
  // of the additions into oc; y^2 = p + pe exactly (p = fl(y y), pe = fma(y, y,
  // -p)) enters (os2, oc2) the same way.  With at most K = REAL_FLUSH_SAMPLES
  // samples between flushes (|oc| <= k u sum |y| after k of them, |oc2| <= (k+1) u
  // sum y^2, u = 2^-24) those roundings total at most u^2 K(K+1)/2 sum |y| and
  // 2 u^2 (K(K+1)/2 + K) sum y^2: below 1.3e-13 of sum |y| and 3.2e-13 of sum
  // y^2.  A flush adds each float, exactly widened, into the FP64 sums, so the
  // thread's sums are within about 3.5e-13 of the exact sums of its samples, at
  // one FP64 operation per sample.
  //
  // PAIRED (levels 0 and 1, where that is what bounds the kernel): two samples at
  // a time, each in its own pair of (fs, fc), on two-float instructions.  After K
  // = REAL_FLUSH_PAIRS a flush joins the two pairs of each sum by one more TwoSum,
  // whose error and the two companions are added (2 roundings of at most (2K+1) u
  // sum |y|), and adds two floats to the FP64 sum: at most u^2 (K(K+1)/2 + 2K + 1)
  // sum |y| and 2 u^2 (K(K+1)/2 + K + 2K + 3) sum y^2, below 1.3e-13 and 3.1e-13.
  // 9 instructions and 2/3 of an FP64 operation per sample, against 17 and one:
  // 67,108,864 level-0 FP32 samples 172 -> 159 us, the FP64 unit 73 -> 54% busy.
  template <bool PAIRED, class T>
  __device__ __forceinline__ void add_real(T y) {
    if constexpr (XP == XP_F64 && EST == EST_EXACT) {
      ds += (double)y;
      dq = fma((double)y, (double)y, dq);
    } else if constexpr (PAIRED) {
      if (have) add_pair(F2::of(first, (float)y));
      first = (float)y;
      have = !have;
    } else {
      const float yf = (float)y;
      oc = __fadd_rn(oc, two_sum(os, yf));
      const float p = __fmul_rn(yf, yf);
      const float pe = __fmaf_rn(yf, yf, -p);
      oc2 = __fadd_rn(__fadd_rn(oc2, two_sum(os2, p)), pe);
    }
  }
  __device__ __forceinline__ void add_pair(F2 y) {
    fc = add2(fc, two_sum(fs, y));
    const F2 p = mul2(y, y);
    const F2 pe = fma2(y, y, sub2(F2{0}, p));
    fc2 = add2(add2(fc2, two_sum(fs2, p)), pe);
  }
  static constexpr bool PAIRS = EST != EST_APPROX && !(XP == XP_F64 && EST == EST_EXACT);
  static __device__ __forceinline__ void flush_pair(F2 &s, F2 &c, double &d) {
    float a, b, ca, cb;
    s.get(a, b);
    c.get(ca, cb);
    const float t = __fadd_rn(a, b), z = __fsub_rn(t, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(t, z)), __fsub_rn(b, z));
    if (fabsf(t) <= 3.402823466e38f) {
      d += (double)t;
      d += (double)__fadd_rn(__fadd_rn(ca, cb), e);
    } else {   // the two sums together leave the float range
      d += (double)a + (double)ca;
      d += (double)b + (double)cb;
    }
    s = F2{0};
    c = F2{0};
  }
  template <bool PAIRED>
  __device__ __forceinline__ void flush_real() {
    if constexpr (PAIRS && PAIRED) {
      flush_pair(fs, fc, ds);
      flush_pair(fs2, fc2, dq);
    } else if constexpr (PAIRS) {
      ds += (double)os;
      ds += (double)oc;
      dq += (double)os2;
      dq += (double)oc2;
      os = 0.0f; oc = 0.0f; os2 = 0.0f; oc2 = 0.0f;
    }
  }
};

template <class T>
__device__ __forceinline__ T shfl_xor(T v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }

// Reduce the CTA's thread accumulators into one Partial (thread 0 writes it).
// Approximate-only estimators have integer sums only, the others real sums
// only, so each shuffles just its own.
template <int EST, int XP>
__device__ __forceinline__ void block_reduce_write(ThreadAcc<EST, XP> &a, Partial *out) {
  constexpr bool INT = EST == EST_APPROX;
  int64_t isum = INT ? a.isum : 0;
  uint64_t lo = INT ? a.q_lo : 0, hi = INT ? a.q_hi : 0;
  double ds = INT ? 0.0 : a.ds, dq = INT ? 0.0 : a.dq;
  uint32_t ns = a.nsat;
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    if constexpr (INT) {
      isum += shfl_xor((long long)isum, m);
      const uint64_t olo = (uint64_t)shfl_xor((unsigned long long)lo, m);
      const uint64_t ohi = (uint64_t)shfl_xor((unsigned long long)hi, m);
      add_u128(lo, hi, olo, ohi);
    } else {
      ds += shfl_xor(ds, m);
      dq += shfl_xor(dq, m);
    }
    ns += shfl_xor(ns, m);
  }
  __shared__ Partial wp[LAUNCH_THREADS / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    Partial p;
    p.isum = isum; p.isum2_lo = lo; p.isum2_hi = hi; p.dsum = ds; p.dsum2 = dq; p.nsat = ns;
    wp[warp] = p;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    Partial t = wp[0];
    const int nw = blockDim.x >> 5;
    for (int w = 1; w < nw; ++w) {
      t.isum += wp[w].isum;
      add_u128(t.isum2_lo, t.isum2_hi, wp[w].isum2_lo, wp[w].isum2_hi);
      t.dsum += wp[w].dsum;
      t.dsum2 += wp[w].dsum2;
      t.nsat += wp[w].nsat;
    }
    *out = t;
  }
}

template <int P> using PayTag = std::integral_constant<int, P>;

// The compiler may not reuse a value computed before this point: the clamped
// re-run of a LAZY group recomputes its draws instead of keeping the first
// run's live in registers through the group.
__device__ __forceinline__ void opaque(uint64_t &x) { asm volatile("" : "+l"(x)); }

// The item fields the group code reads, copied into registers once per chunk
// (read through the item reference they would be loaded again for every
// group: the kernel's stores to global memory might alias them).
struct GroupCtx {
  uint32_t ctr2, ctr3;
  int d, level, enumerate, lanes;
  uint64_t first, last;
};
// The Philox words of call q.
__device__ __forceinline__ uint4 draw(const GroupCtx &it, const LaunchArgs &args, uint64_t q) {
  return philox4x32_10(make_uint4((uint32_t)q, (uint32_t)(q >> 32), it.ctr2, it.ctr3), args.rk);
}

// The samples of group g of a chunk, for a level class LC known at compile
// time (0: level 0, 1: level 1, 2: levels >= 2).  A group is one Philox call's
// worth of packs (4 on level 0, 2 on level 1) or, from level 2, one pack over
// 2^l / 4 calls; a pack holds KP samples.  E: the clamped datapath (LAZY
// kernels; always true elsewhere); FULL: every sample of the group is in the
// item's range at compile time (then no per-sample range test splits the
// group's straight-line code); full: the same known at run time; PAY: the
// terminal payoff when fixed at compile time (0 European, 1 digital, -1 not).
template <int LC, bool E, bool FULL, int PAY, bool DUMP, class Sim, class Acc>
__device__ __forceinline__ void run_group(Sim &sim, Acc &acc, const LaunchArgs &args, const GroupCtx &it, uint64_t g,
                                          bool full, uint64_t first, uint64_t last, mlmc_sample_rec *dump) {
  constexpr int KP = Sim::KPV;
  if constexpr (LC == 2) {
    uint64_t P = g;
    uint32_t lsh = 0;   // lane-split packed draws: this sample's field to the top of the word
    if constexpr (KP == 1 && Sim::ESTV == EST_APPROX) {
      if (it.lanes > 1) {
        P = g / 3u;
        lsh = (uint32_t)it.d * (uint32_t)(g - P * 3u);
      }
    }
    const uint32_t calls = 1u << (it.level - 2);
    uint64_t qbase = P * calls;
    if constexpr (E && Sim::LAZY) opaque(qbase);
    sim.begin();
    // qbase is a multiple of calls (a power of two): the calls share its high word
    const PhiloxStream ps((uint32_t)(qbase >> 32), it.ctr2, it.ctr3, args.rk);
    for (uint32_t c = 0; c < calls; ++c) {
      const uint4 w = Sim::STREAM ? ps.call((uint32_t)qbase + c, args.rk) : draw(it, args, qbase + c);
      // (a step asks of its index whether it is the first; the binary16 / bfloat16
      // kernels were faster with the index itself)
      const int i0 = Sim::HALF ? (int)(c << 2) : c ? 4 : 0;
      sim.template step<true, 0, E>(w.x << lsh, i0);
      sim.template step<true, 1, E>(w.y << lsh, i0 + 1);
      sim.template step<true, 0, E>(w.z << lsh, i0 + 2);
      sim.template step<true, 1, E>(w.w << lsh, i0 + 3);
    }
    // a lazy correction that left its range adds nothing and runs again
    if (Sim::ESTV == EST_CORR && !E && sim.over()) return;
#pragma unroll
    for (int l = 0; l < KP; ++l) {
      const uint64_t s = KP == 1 ? g : P * KP + l;
      const bool valid = FULL || full || (s >= first && s < last);
      sim.template finish<E, PAY, 1>(acc, l, valid, DUMP && valid ? dump + (s - first) : nullptr);
    }
  } else {
    uint64_t gw = g;
    if constexpr (E && Sim::LAZY) opaque(gw);
    uint4 w;
    if (Sim::ENUMERATE && it.enumerate) w = enum_words(gw, LC, it.d);
    else w = draw(it, args, gw);
    constexpr int PPG = LC == 1 ? 2 : 4;  // packs per group
    const uint64_t s0 = (uint64_t)(PPG * KP) * g;
    // samples s0 + k are valid for k in [klo, khi)
    int klo = 0, khi = PPG * KP;
    if (!FULL && !full) {
      klo = s0 >= first ? 0 : (int)min(first - s0, (uint64_t)(PPG * KP));
      khi = last <= s0 ? 0 : (int)min(last - s0, (uint64_t)(PPG * KP));
    }
    if constexpr (LC == 1) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        sim.begin();
        sim.template step<true, 0, E>(u == 0 ? w.x : w.z, 0);
        sim.template step<true, 1, E>(u == 0 ? w.y : w.w, 1);
#pragma unroll
        for (int l = 0; l < KP; ++l) {
          const int k = u * KP + l;
          const bool valid = FULL || (k >= klo && k < khi);
          sim.template finish<E, PAY, 1, true>(acc, l, valid, DUMP && valid ? dump + (s0 + k - first) : nullptr);
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        sim.begin();
        sim.template step<false, -1, E>(word_of(w, u), 0);
#pragma unroll
        for (int l = 0; l < KP; ++l) {
          const int k = u * KP + l;
          const bool valid = FULL || (k >= klo && k < khi);
          sim.template finish<E, PAY, 0, true>(acc, l, valid, DUMP && valid ? dump + (s0 + k - first) : nullptr);
        }
      }
    }
  }
}

// One level-0 group of an item whose table holds each index's sample value
// (ItemDesc::tab_y0): per sample one table read and the two group sums.
// Samples k outside [klo, khi) add zero (FULL: the whole group is in range).
template <bool FULL, class Sim, class Acc>
__device__ __forceinline__ void y0_group(const Sim &sim, Acc &acc, const uint4 &w, int klo, int khi) {
  constexpr int KP = Sim::KPV;
  int32_t y[4 * KP];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
#pragma unroll
    for (int l = 0; l < KP; ++l) {
      const int k = u * KP + l;
      y[k] = sim.template fx32_entry<int32_t, 2>(word_of(w, u), l);
      if (!(FULL || (k >= klo && k < khi))) y[k] = 0;
    }
  }
#pragma unroll
  for (int k = 0; k < 4 * KP; k += 2) acc.add_group2(y[k], y[k + 1]);
}

// The groups of a chunk of such an item: the same samples and values as
// run_group's path (no saturation: see tab_y0_of).
template <class Sim, class Acc>
__device__ __forceinline__ void group_loop_y0(const Sim &sim, Acc &acc, const LaunchArgs &args, const GroupCtx &it,
                                              uint64_t gbeg, uint32_t ng, uint32_t rf0, uint32_t rf1, bool once) {
  constexpr int KP = Sim::KPV;
  const uint64_t first = it.first, last = it.last;
  // the chunk's Philox calls share the counter's high word but for one in 2^32;
  // once: a thread's whole sums stay in the 64-bit group sums, where they fit
  const uint32_t hi = (uint32_t)(gbeg >> 32);
  const bool one_hi = (uint32_t)((gbeg + ng) >> 32) == hi;
  const PhiloxStream ps(hi, it.ctr2, it.ctr3, args.rk);
  for (uint32_t r = threadIdx.x; r < ng; r += blockDim.x) {
    const uint64_t g = gbeg + r;
    uint4 w;
    if (Sim::ENUMERATE && it.enumerate) w = enum_words(g, 0, it.d);
    else if (one_hi) w = ps.call((uint32_t)g, args.rk);
    else w = draw(it, args, g);
    if (r >= rf0 && r < rf1) {
      y0_group<true>(sim, acc, w, 0, 0);
    } else {
      const uint64_t s0 = (uint64_t)(4 * KP) * g;
      const int klo = s0 >= first ? 0 : (int)min(first - s0, (uint64_t)(4 * KP));
      const int khi = last <= s0 ? 0 : (int)min(last - s0, (uint64_t)(4 * KP));
      y0_group<false>(sim, acc, w, klo, khi);
    }
    if (!once) acc.flush_group();
  }
  acc.flush_group();
}

// A thread's groups of one chunk, groups gbeg + r for r = threadIdx.x,
// threadIdx.x + blockDim.x, ... < ng, of level class LC; groups with r in
// [rf0, rf1) lie entirely in the item's range.  LAZY items run each such group
// first with S unclamped and its samples added tentatively; a group whose S
// went above lim_S is dropped and run again on the clamped datapath (rare).
// PAYF: the terminal payoff of the lazy run (terminal payoff classes).
template <int LC, int PAYF, bool DUMP, int EST, int XP, int AP, int PC, class Sim>
__device__ __forceinline__ void group_loop(Sim &sim, ThreadAcc<EST, XP> &acc, const LaunchArgs &args,
                                           const GroupCtx &it, uint64_t gbeg, uint32_t ng, uint32_t rf0, uint32_t rf1,
                                           bool lazy, mlmc_sample_rec *dump) {
  const uint64_t first = it.first, last = it.last;
  // Real-valued estimators flush their float pairs every FLUSH_GROUPS groups
  // (8 samples, or 6 pairs; a group of levels 0 and 1 has an even number of samples).
  constexpr bool REAL = ThreadAcc<EST, XP>::PAIRS;
  constexpr uint32_t FLUSH_GROUPS =
      LC == 2 ? (uint32_t)REAL_FLUSH_SAMPLES : (uint32_t)REAL_FLUSH_PAIRS / (LC == 1 ? 1u : 2u);
  uint32_t since_flush = 0;
  for (uint32_t r = threadIdx.x; r < ng; r += blockDim.x) {
    const uint64_t g = gbeg + r;
    const bool full = r >= rf0 && r < rf1;
    if constexpr (Sim::LAZY && !DUMP) {
      bool eager = true;
      if constexpr (EST == EST_CORR) {
        if (lazy) {
          sim.hi = 0;
          const auto saved = acc.mark();
          run_group<LC, false, false, PAYF, DUMP>(sim, acc, args, it, g, full, first, last, dump);
          eager = sim.over();
          if (LC != 2 && eager) acc.rewind(saved);
        }
      } else if (lazy && full) {
        sim.hi = 0;
        if constexpr (PC == PC_TERMINAL) {
          // the group's sums stay in their own accumulator until the group is kept
          run_group<LC, false, true, PAYF, DUMP>(sim, acc, args, it, g, true, first, last, dump);
          eager = sim.over();
          if (eager) acc.discard_group();
        } else {
          // path-dependent payoffs: one sample per step carries more state, and a
          // FULL instantiation costs registers more than the range test costs
          const auto saved = acc.mark();
          run_group<LC, false, false, -1, DUMP>(sim, acc, args, it, g, true, first, last, dump);
          eager = sim.over();
          if (eager) acc.rewind(saved);
        }
      }
      if (eager) run_group<LC, true, false, -1, DUMP>(sim, acc, args, it, g, full, first, last, dump);
    } else {
      // other datapaths: one instantiation (a FULL one beside it raised the
      // packed binary16 kernels from ~115 to ~165 registers and cost 9%)
      run_group<LC, true, false, -1, DUMP>(sim, acc, args, it, g, full, first, last, dump);
    }
    if constexpr (EST == EST_APPROX && AP == AP_FX32 && PC == PC_TERMINAL) acc.flush_group();
    if constexpr (REAL) {
      if (++since_flush == FLUSH_GROUPS) {
        acc.template flush_real<LC != 2>();
        since_flush = 0;
      }
    }
  }
  acc.template flush_real<LC != 2>();
}

// The first ng groups of a chunk, a multiple of 2 blockDim.x, two at a time
// (Sim::DUO; levels >= 2, one sample per group): groups r and r + blockDim.x.
// The binary16 kernel's integer-multiply pipe was 87% busy, half of it with
// scalar half instructions: 1,000,003 level-8 Milstein Asian samples 386 -> 276 us
// (with the larger chunks that give a thread two samples there).
template <class Sim, class Acc>
__device__ __forceinline__ void group_loop_duo(Sim &sim, Acc &acc, const LaunchArgs &args, const GroupCtx &it,
                                               uint64_t gbeg, uint32_t ng) {
  const uint32_t calls = 1u << (it.level - 2);
  for (uint32_t r = threadIdx.x; r < ng; r += 2u * blockDim.x) {
    const uint64_t q0 = (gbeg + r) * calls, q1 = q0 + (uint64_t)blockDim.x * calls;
    const PhiloxStream p0((uint32_t)(q0 >> 32), it.ctr2, it.ctr3, args.rk);
    const PhiloxStream p1((uint32_t)(q1 >> 32), it.ctr2, it.ctr3, args.rk);
    sim.begin();
    for (uint32_t c = 0; c < calls; ++c) {
      const uint4 w = p0.call((uint32_t)q0 + c, args.rk), v = p1.call((uint32_t)q1 + c, args.rk);
      const int i0 = (int)(c << 2);
      sim.template step<true, 0>(w.x, i0, v.x);
      sim.template step<true, 1>(w.y, i0 + 1, v.y);
      sim.template step<true, 0>(w.z, i0 + 2, v.z);
      sim.template step<true, 1>(w.w, i0 + 3, v.w);
    }
    sim.template finish<true, -1, 1>(acc, 0, true, nullptr);
    sim.template finish<true, -1, 1>(acc, 1, true, nullptr);
  }
}

// Simulate one chunk of an item (its table already in shared memory) and
// write the CTA's Partial for it.  The level class and (on the lazy terminal
// path) the payoff are fixed once per chunk, so the group loop carries no
// branch on them.  DYN (device-scheduled kernel) only keeps the
// instantiations of the static and device-scheduled kernels apart, so that
// each is compiled inline into its own kernel.
template <int EST, int XP, int AP, int SCHEME, int PC, int KP, int MSEL, bool DUMP, bool DYN, bool PRE = false,
          bool MERGED = false>
__device__ __forceinline__ void chunk_body(const LaunchArgs &args, const ItemDesc &it, int item, uint32_t gc,
                                           const unsigned char *smem_tab) {
  using Sim = LevelSim<EST, XP, AP, SCHEME, PC, KP, MSEL, PRE, MERGED>;
  // unpacked half-precision estimators take a thread's samples two at a time from
  // level 2 (a thread with one sample, or its odd last one, takes it alone; the
  // device-scheduled kernels, whose registers it would raise, always do)
  constexpr bool DUO = EST == EST_APPROX && Sim::HALF && KP == 1 && !DUMP && !DYN;
  ThreadAcc<EST, XP> acc;
  acc.init();

  const uint32_t chunk = gc - it.chunk_begin;
  const uint64_t per_chunk = (uint64_t)it.groups_per_thread * blockDim.x;
  uint64_t gbeg = it.g0 + (uint64_t)chunk * per_chunk;
  const uint64_t gend = min(it.g1, gbeg + per_chunk);
  uint32_t ng = gend > gbeg ? (uint32_t)(gend - gbeg) : 0u;
  // the chunk's groups [rf0, rf1) (relative to gbeg) lie entirely in the item's range
  const uint64_t gf0 = max(it.gf0, gbeg), gf1 = min(it.gf1, gend);
  uint32_t rf0 = gf0 < gf1 ? (uint32_t)(gf0 - gbeg) : 0u;
  uint32_t rf1 = gf0 < gf1 ? (uint32_t)(gf1 - gbeg) : 0u;
  // per-sample records only in the DUMP instantiation (parity runs)
  mlmc_sample_rec *dump = DUMP ? (mlmc_sample_rec *)it.dump : nullptr;
  const bool lazy = Sim::LAZY && !DUMP && it.ff.lazy;
  const int lc = it.level >= 2 ? 2 : it.level;
  const GroupCtx gx{it.ctr2, it.ctr3, it.d, it.level, it.enumerate, it.lanes, it.first, it.first + it.N};
  if constexpr (DUO) {
    const uint32_t pairs = it.level >= 2 && it.lanes <= 1 ? ng / (2u * blockDim.x) * (2u * blockDim.x) : 0u;
    if (pairs) {
      LevelSim<EST, XP, AP, SCHEME, PC, 2, MSEL> duo;
      duo.load(it, smem_tab);
      group_loop_duo(duo, acc, args, gx, gbeg, pairs);
      gbeg += pairs;
      ng -= pairs;
      rf0 = rf0 > pairs ? rf0 - pairs : 0u;
      rf1 = rf1 > pairs ? rf1 - pairs : 0u;
    }
  }
  Sim sim;
  sim.load(it, smem_tab);
  auto loop = [&](auto lctag, auto paytag) {
    group_loop<decltype(lctag)::value, decltype(paytag)::value, DUMP, EST, XP, AP, PC>(sim, acc, args, gx, gbeg, ng,
                                                                                      rf0, rf1, lazy, dump);
  };
  using L0 = std::integral_constant<int, 0>;
  using L1 = std::integral_constant<int, 1>;
  using L2 = std::integral_constant<int, 2>;
  if constexpr (Sim::LAZY && !DUMP && PC == PC_TERMINAL) {
    const bool dig = it.payoff == 1;
    const bool y0 = EST == EST_APPROX && it.tab_y0;
    if (lc == 0) {
      if (y0) {
        if constexpr (EST == EST_APPROX) {
          // samples of a thread (at most) times y^2 < 2^64
          const uint64_t most = (uint64_t)it.groups_per_thread * (4u * KP);
          group_loop_y0(sim, acc, args, gx, gbeg, ng, rf0, rf1, it.y0_bits < 64 && most <= (1ULL << it.y0_bits));
        }
      }
      else if (dig) loop(L0{}, PayTag<1>{});
      else loop(L0{}, PayTag<0>{});
    }
    else if (lc == 1) { if (dig) loop(L1{}, PayTag<1>{}); else loop(L1{}, PayTag<0>{}); }
    else { if (dig) loop(L2{}, PayTag<1>{}); else loop(L2{}, PayTag<0>{}); }
  } else {
    if (lc == 0) loop(L0{}, PayTag<-1>{});
    else if (lc == 1) loop(L1{}, PayTag<-1>{});
    else loop(L2{}, PayTag<-1>{});
  }
  block_reduce_write<EST, XP>(acc, args.partials + gc);
  if (!DYN && args.counters) {
    // the CTA that completes the item's last chunk sums all its partials, in a
    // fixed order; up to 32 of them (the other columns are empty: adding their
    // zeros changes nothing) are one warp's work, without the CTA's barriers
    const bool few = it.n_chunks <= 32u;
    __shared__ uint32_t s_last;
    uint32_t last = 0;
    if (threadIdx.x == 0) {
      __threadfence();
      last = atomicAdd(args.counters + item, 1u) + 1u == it.n_chunks;
      s_last = last;
    }
    if (few) {
      if (threadIdx.x < 32) last = __shfl_sync(0xffffffffu, last, 0);
    }
    else {
      __syncthreads();
      last = s_last;
    }
    if (last) {
      __threadfence();
      constexpr bool INTS = EST == EST_APPROX;
      const Partial *p = args.partials + it.chunk_begin;
      const DevSums r = few ? to_sums(group_sum<INTS, !INTS>(one_chunk<INTS, !INTS>(p, it.n_chunks, threadIdx.x)))
                            : cta_sum_partials<INTS, !INTS>(p, it.n_chunks);
      if (threadIdx.x == 0) {
        args.out[it.out_index] = r;
        args.counters[item] = 0u;   // ready for the next launch
      }
    }
  }
}

// Does an item run the pre-scaled form of the 32-bit fast datapath?  (Records
// take the plain form, as does Method 2's coupled exact path: pre_ok is 0 there.)
__device__ __forceinline__ bool fx32_pre(const ItemDesc &it) { return it.ff.pre_ok && !it.dump; }

// Find the item of chunk gc (the last with chunk_begin <= gc) and stage its
// approximate-Normal table in shared memory (unless *staged, when given, says
// that it is there already).  Every thread has finished the previous chunk
// before the table is overwritten (block_reduce_write ends with a barrier).
template <int AP, int SCHEME, bool PHI_BY_KIND = false>
__device__ __forceinline__ int stage_chunk(const ItemDesc *items, int n_items, uint32_t gc, const void **staged) {
  extern __shared__ __align__(16) unsigned char smem_tab[];
  __shared__ int s_item;
  if (n_items == 1) {
    if (threadIdx.x == 0) s_item = 0;
  } else if (threadIdx.x < 32) {
    // last item with chunk_begin <= gc (chunk_begin is non-decreasing and
    // items[0].chunk_begin <= gc): warp 0 samples 32 evenly spaced items per
    // round, one load each, and narrows to the stride after the last sample
    // at or before gc; one round for up to 32 items, two for up to 1024
    const int lane = threadIdx.x;
    int lo = 0, span = n_items;
    while (true) {
      const int stride = span > 32 ? (span + 31) / 32 : 1;
      const int k = lo + lane * stride;
      const bool le = lane * stride < span && items[k].chunk_begin <= gc;
      const int last = __popc(__ballot_sync(0xffffffffu, le)) - 1;
      lo += last * stride;
      if (stride == 1) break;
      span = min(stride, span - last * stride);
    }
    if (lane == 0) s_item = lo;
  }
  // the exact path's table, started before the first chunk: a static launch with an
  // approximate table waits for it at the barrier behind that table's stores
  if (AP == AP_NONE || staged) copies_done();
  __syncthreads();
  const int item = s_item;
  const ItemDesc &it = items[item];
  if constexpr (AP == AP_FX32) {
    // (Z~_j, sum1 of a fine step from Z~_j) for every index j, or in the
    // pre-scaled form of Euler items P_j = con2 Z~_j + radd1 (LevelSim's PRE):
    // Method 1 and 2 values from the item's table, Method 3 values from its
    // class lines (the arithmetic of LevelSim::fixed_z); sum1 by the datapath's
    // own step code.
    // The table depends on the item's constants as well, so a persistent CTA
    // (staged != nullptr) keeps it while its chunks stay in the same item.
    if (staged && *staged == (const void *)&it) return item;
    if (staged) *staged = (const void *)&it;
    // the item's constants in registers first: the table stores below go
    // through a pointer the compiler cannot tell apart from the item, so
    // fields read inside the loop would be loaded again after every store
    const FastFixed ff = it.ff;
    const int d = it.d, method = it.method, tab_y0 = it.tab_y0, payoff = it.payoff;
    const int fZh = it.fx.fZ2 / 2, fS = it.fx.fS;
    const int32_t S0q = (int32_t)it.fx.S0, Kq = (int32_t)it.fx.K;
    const void *ztab = it.ztab;
    const int n = 1 << d;
    // merged launch: only the correction chunks (kind 2) run the FP32 exact path;
    // the copies proceed while the pairs are formed
    if constexpr (PHI_BY_KIND) {
      if (it.kind == 2) stage_phi_inv<PHI_OCT_CORR>();
    }
    const bool pre = fx32_pre(it), p32 = pre && SCHEME == 0;
    int2 *dst = (int2 *)smem_tab;
    int32_t *dst4 = (int32_t *)smem_tab;
    const M3Coef *m3 = (const M3Coef *)ztab;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      int32_t z;
      if (method != 3) {
        z = ((const int32_t *)ztab)[k];
      } else {
        const ApproxIndex ai = approx_index((uint32_t)k << (32 - d), d);
        const int c = m3_class(ai.idx);
        const int64_t t = m3->A[c] + m3->B[c] * (int64_t)ai.idx;
        const int sh = M3_FRAC - fZh;
        const int32_t v = (int32_t)((t + ((int64_t)1 << (sh - 1))) >> sh);
        z = ai.neg ? -v : v;
      }
      if (p32 && !tab_y0) {
        dst4[k] = ff.con2 * z + (int32_t)ff.radd1;
        continue;
      }
      const int32_t sum1 = ff_sum1<SCHEME == 1, true>(ff, z, ff.con1r, ff.mfine);
      if (tab_y0) {
        // level 0: the sample is a function of j alone -- S after the one fine
        // step from S0 (mul2 = rd(S0 sum1), S = rd(S0 + mul2), clamped to lim_S
        // as on the clamped datapath) and its terminal payoff
        // (the host sets tab_y0 on lazy items only, whose S_0 <= limT keeps
        // that S within lim_S: the clamp changes nothing there).  The same
        // arithmetic as LevelSim::ff_apply's 32-bit step and fixed_payoff's
        // 32-bit terminal payoff; the level-0 parity tests hold the two equal.
        const int64_t p2 = (int64_t)S0q * sum1 + ff.radd2;
        const int32_t mul2 = (int32_t)__funnelshift_r((uint32_t)p2, (uint32_t)((uint64_t)p2 >> 32), ff.rs2);
        const int32_t s1 = (int32_t)((uint32_t)S0q + (uint32_t)mul2 * (uint32_t)ff.mulS);
        const int32_t lim = (int32_t)ff.limS;
        const int32_t c = min(max(s1, -lim), lim);
        const int32_t y = c > Kq ? (payoff == 1 ? (int32_t)1 << fS : c - Kq) : 0;
        dst4[k] = y;
      } else {
        dst[k] = make_int2(z, pre ? sum1 * (1 << (32 - ff.rs2)) : sum1);
      }
    }
    if (it.perm) {   // after the table: the method-2 interval ranks
      uint16_t *pd = (uint16_t *)(smem_tab + (size_t)n * TabBytes<AP>::value);
      for (int k = threadIdx.x; k < n; k += blockDim.x) pd[k] = it.perm[k];
    }
    copies_done();
    __syncthreads();
  } else if constexpr (AP != AP_NONE) {
    if (!staged || it.ztab != *staged) {
      if (staged) *staged = it.ztab;
      if (it.method != 3) {
        const int n = 1 << it.d;
        if constexpr (AP == AP_FIXED || AP == AP_FX64) {
          const int32_t *src = (const int32_t *)it.ztab;
          for (int k = threadIdx.x; k < n; k += blockDim.x) ((int32_t *)smem_tab)[k] = src[k];
        } else {
          const uint16_t *src = (const uint16_t *)it.ztab;
          for (int k = threadIdx.x; k < n; k += blockDim.x) ((uint16_t *)smem_tab)[k] = src[k];
        }
        if (it.perm) {   // after the table: the method-2 interval ranks
          uint16_t *dst = (uint16_t *)(smem_tab + (size_t)n * TabBytes<AP>::value);
          for (int k = threadIdx.x; k < n; k += blockDim.x) dst[k] = it.perm[k];
        }
      } else {
        const uint32_t *src = (const uint32_t *)it.ztab;
        for (int k = threadIdx.x; k < (int)(sizeof(M3Coef) / 4); k += blockDim.x)
          ((uint32_t *)smem_tab)[k] = src[k];
      }
      copies_done();
      __syncthreads();
    }
  }
  return item;
}

// A chunk of the 32-bit fast datapath in the form that its item takes.
template <int EST, int SCHEME, int PC, int KP, bool DYN, bool MERGED>
__device__ __forceinline__ void fx32_chunk(const LaunchArgs &args, const ItemDesc &it, int item, uint32_t gc,
                                           const unsigned char *smem_tab) {
  if (fx32_pre(it))
    chunk_body<EST, XP_F32, AP_FX32, SCHEME, PC, KP, 0, false, DYN, true, MERGED>(args, it, item, gc, smem_tab);
  else if (EST != EST_CORR || !it.perm)
    chunk_body<EST, XP_F32, AP_FX32, SCHEME, PC, KP, 0, false, DYN, false, MERGED>(args, it, item, gc, smem_tab);
  else if constexpr (EST == EST_CORR)
    chunk_body<EST, XP_F32, AP_FX32, SCHEME, PC, KP, 4, false, DYN, false, MERGED>(args, it, item, gc, smem_tab);
}

// One chunk (gc) of one launch: its item and table (stage_chunk), then the
// chunk's sample groups and the CTA's Partial for the chunk.
template <int EST, int XP, int AP, int SCHEME, int PC, int KP, bool ALLOW_DUMP, bool DYN>
__device__ __forceinline__ void run_chunk(const LaunchArgs &args, const ItemDesc *items, int n_items, uint32_t gc,
                                          const void **staged) {
  extern __shared__ __align__(16) unsigned char smem_tab[];
  const int item = stage_chunk<AP, SCHEME>(items, n_items, gc, staged);
  const ItemDesc &it = items[item];
  if (ALLOW_DUMP && it.dump) {
    if constexpr (ALLOW_DUMP) chunk_body<EST, XP, AP, SCHEME, PC, KP, 2, true, DYN>(args, it, item, gc, smem_tab);
  } else if constexpr (XP == XP_F64) {
    if (it.qF) chunk_body<EST, XP, AP, SCHEME, PC, KP, 0, false, DYN>(args, it, item, gc, smem_tab);
    else chunk_body<EST, XP, AP, SCHEME, PC, KP, 1, false, DYN>(args, it, item, gc, smem_tab);
  } else if constexpr (AP == AP_NONE) {
    chunk_body<EST, XP, AP, SCHEME, PC, KP, 0, false, DYN>(args, it, item, gc, smem_tab);
  } else if constexpr (AP == AP_FX32) {
    // no method choice: the table holds every method's values
    fx32_chunk<EST, SCHEME, PC, KP, DYN, false>(args, it, item, gc, smem_tab);
  } else {
    if (EST == EST_CORR && it.perm) {
      if constexpr (EST == EST_CORR) chunk_body<EST, XP, AP, SCHEME, PC, KP, 4, false, DYN>(args, it, item, gc, smem_tab);
    } else if (it.method == 3) chunk_body<EST, XP, AP, SCHEME, PC, KP, 1, false, DYN>(args, it, item, gc, smem_tab);
    else chunk_body<EST, XP, AP, SCHEME, PC, KP, 0, false, DYN>(args, it, item, gc, smem_tab);
  }
}

// Static launch: CTA b runs chunk chunk0 + b of the launch.
template <int EST, int XP, int AP, int SCHEME, int PC, int KP>
__global__ void __launch_bounds__(LAUNCH_THREADS, MinCtas<EST, XP, AP, SCHEME, PC, KP>::value)
level_kernel(const __grid_constant__ LaunchArgs args) {
  stage_exact_table<EST, XP>();
  run_chunk<EST, XP, AP, SCHEME, PC, KP, false, false>(args, args.use_one ? &args.one : args.items, args.n_items,
                                                      args.chunk0 + blockIdx.x, nullptr);
}

// The same for launches with per-sample records (parity runs): a kernel of
// its own, so that the record-writing code does not weigh on the register
// allocation of the launches without records.
template <int EST, int XP, int AP, int SCHEME, int PC, int KP>
__global__ void __launch_bounds__(LAUNCH_THREADS, MinCtas<EST, XP, AP, SCHEME, PC, KP>::value)
level_kernel_dump(const __grid_constant__ LaunchArgs args) {
  stage_exact_table<EST, XP>();
  run_chunk<EST, XP, AP, SCHEME, PC, KP, true, false>(args, args.items, args.n_items, args.chunk0 + blockIdx.x,
                                                     nullptr);
}

// Device-scheduled launch (fixed grid, captured once in a CUDA graph): the item
// and chunk counts come from args.dyn, written on the device before the
// launch; CTA b runs chunks b, b + gridDim.x, ...
template <int EST, int XP, int AP, int SCHEME, int PC, int KP>
__global__ void __launch_bounds__(LAUNCH_THREADS, MinCtas<EST, XP, AP, SCHEME, PC, KP, true>::value)
level_kernel_dyn(const __grid_constant__ LaunchArgs args) {
  const DynLaunch d = *args.dyn;
  const void *staged = nullptr;
  stage_exact_table<EST, XP>();
  for (uint32_t rel = blockIdx.x; rel < d.n_chunks; rel += gridDim.x)
    run_chunk<EST, XP, AP, SCHEME, PC, KP, false, true>(args, args.items + d.item_off, (int)d.n_items,
                                                        d.chunk0 + rel, &staged);
}

// A merged launch of the nested estimator's three 32-bit fixed-point kernel
// families for one (scheme, payoff class): approximate with packed draws
// (kind 0), approximate one sample per thread (kind 1) and correction (kind 2).
// Its chunks run the same chunk bodies as the separate launches, in one grid
// ordered by decreasing CTA cost, so the longest chains start first and the
// short chunks of every family fill in behind them.
// PRE: every item takes the pre-scaled form (family 24; else family 17).
template <int SCHEME, int PC, bool PRE>
__global__ void __launch_bounds__(LAUNCH_THREADS, 7) nested_kernel(const __grid_constant__ LaunchArgs args) {
  extern __shared__ __align__(16) unsigned char smem_tab[];
  const uint32_t gc = args.chunk0 + blockIdx.x;
  const int item = stage_chunk<AP_FX32, SCHEME, true>(args.items, args.n_items, gc, nullptr);
  const ItemDesc &it = args.items[item];
  if constexpr (PRE) {
    if (it.kind == 0)
      chunk_body<EST_APPROX, XP_F32, AP_FX32, SCHEME, PC, 3, 0, false, false, true, true>(args, it, item, gc, smem_tab);
    else if (it.kind == 1)
      chunk_body<EST_APPROX, XP_F32, AP_FX32, SCHEME, PC, 1, 0, false, false, true, true>(args, it, item, gc, smem_tab);
    else
      chunk_body<EST_CORR, XP_F32, AP_FX32, SCHEME, PC, 1, 0, false, false, true, true>(args, it, item, gc, smem_tab);
  } else {
    if (it.kind == 0) fx32_chunk<EST_APPROX, SCHEME, PC, 3, false, true>(args, it, item, gc, smem_tab);
    else if (it.kind == 1) fx32_chunk<EST_APPROX, SCHEME, PC, 1, false, true>(args, it, item, gc, smem_tab);
    else fx32_chunk<EST_CORR, SCHEME, PC, 1, false, true>(args, it, item, gc, smem_tab);
  }
}

}  // namespace mlmc

namespace mlmc {

template <int EST, int XP, int AP, int SCHEME, int PC, int KP>
cudaError_t launch_one(dim3 grid, dim3 block, size_t smem, cudaStream_t st, const LaunchArgs &a, int *occ) {
  auto k = (a.dyn || occ) ? level_kernel_dyn<EST, XP, AP, SCHEME, PC, KP>
            : a.dump       ? level_kernel_dump<EST, XP, AP, SCHEME, PC, KP>
                           : level_kernel<EST, XP, AP, SCHEME, PC, KP>;
  // above 48 KB of dynamic plus static shared memory (the static part holds
  // up to about 16.6 KB: the inverse-Normal cubics) the kernel must opt in
  if (smem > 24 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  // An approximate kernel alone runs with the shared memory that its own CTAs take, and
  // an enumerating one held up the correction kernel beside it (19-25 KB a CTA) until
  // its SMs were free.  With room for both, 132 KB for fixed point and 100 KB for the
  // 2-byte tables, an adaptive estimate with enumerated levels takes 49 -> 41 and 41 ->
  // 34 us.  (100 KB did nothing for fixed point; 132 KB cost 1e6 level-8 binary16 samples
  // 1.1 us, all 228 KB 4; 64 KB took residency from the deep bfloat16 items.)  Tables
  // above 16 KB keep the default.
  if constexpr (EST == EST_APPROX) {
    static int carved = cudaSharedmemCarveoutDefault, carved_on = -1;
    constexpr bool INT_TABLE = AP == AP_FIXED || AP == AP_FX32 || AP == AP_FX64;
    const int want = smem > 16 * 1024 ? (int)cudaSharedmemCarveoutDefault : INT_TABLE ? 58 : 44;   // percent of 228 KB
    int dev = 0;
    if (!a.dyn && !occ && !a.dump && cudaGetDevice(&dev) == cudaSuccess && (want != carved || dev != carved_on)) {
      const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, want);
      if (e != cudaSuccess) return e;
      carved = want;
      carved_on = dev;
    }
  }
  if (occ) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k, (int)block.x, smem);
  k<<<grid, block, smem, st>>>(a);
  return cudaGetLastError();
}

// All (scheme, payoff class) instantiations of one (estimator, precision) family.
template <int EST, int XP, int AP, int KP = 1>
cudaError_t launch_family(int scheme, int pc, dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                          const LaunchArgs &a, int *occ) {
  switch (scheme * 3 + pc) {
    case 0: return launch_one<EST, XP, AP, 0, PC_TERMINAL, KP>(grid, block, smem, st, a, occ);
    case 1: return launch_one<EST, XP, AP, 0, PC_ASIAN, KP>(grid, block, smem, st, a, occ);
    case 2: return launch_one<EST, XP, AP, 0, PC_LOOKBACK, KP>(grid, block, smem, st, a, occ);
    case 3: return launch_one<EST, XP, AP, 1, PC_TERMINAL, KP>(grid, block, smem, st, a, occ);
    case 4: return launch_one<EST, XP, AP, 1, PC_ASIAN, KP>(grid, block, smem, st, a, occ);
    case 5: return launch_one<EST, XP, AP, 1, PC_LOOKBACK, KP>(grid, block, smem, st, a, occ);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mlmc

// Error-model statistics of one MLMC level on the GPU (Sec. 4.2-4.3): for
// the discounted level difference DeltaP = P_f - P_c of a European call under
// Euler-Maruyama with exact FP64 Normals (stream 0, the correction
// estimator's uniforms), the sensitivities xbar = d DeltaP / d x of every
// intermediate variable of Algorithm 1 -- con1 (and the coarse constant for
// 2h), con2, Z_j, mul1_k, sum1_k, mul2_k, S_k on both paths, and S0 -- their
// second moments per variable type (V_indep, eq. optimistic) and per instance
// (V_corr, eq. pessimistic), the maxima |x| per type (exponents, Sec. 4.1),
// and the mean and variance of DeltaP.
//
// The reverse sweep of Algorithm 1 has a closed form for this graph: with
// S_{k+1} = S_k (1 + sum1_k), d S_n / d S_{k+1} = S_n / S_{k+1}, so every
// sensitivity is a_f S_n (resp. a_c S^c_m) times a per-step factor
// (1 / S_{k+1}, 1 / (1 + sum1_k), Z_k / (1 + sum1_k), ...), where
// a_f = e^{-rT} 1[S_n > K] and a_c = -e^{-rT} 1[S^c_m > K].
//
// FP64 operations (2 lanes per clock and SM here) are what the time goes to, so
// there are as few of them as the statistics need.  A CTA takes 128 samples at a
// time.  Pass 1, a thread per sample, runs both paths -- Normals and increments
// in integers (exact64.cuh), one reciprocal u = 1 / (1 + sum1) per step, 1 / S
// by 1 / S_{k+1} = u / S_k -- and writes u and 1 / S of every step to a tape in
// global memory (32 bytes at a time; it stays in L2 up to level 6 or so).  Pass
// 2, a thread per instance, adds the squares over the CTA's samples: no
// cross-lane sums, and the tape read in rows.  The per-type moments are sums of
// the per-instance ones.  About 25 FP64 operations per path-step against 258
// (two library Phi^-1, four divisions, 64-bit butterflies): 100,001 level-6
// samples 3.89 -> 0.42 ms a call, the FP64 unit 85 and 74% busy.
//
// Sums: a CTA's samples in a tree, the CTAs' partials by sens_finalize_kernel.
// Against 80-bit sums the instances' errors are no larger than those of division
// and butterflies per sample (20,000 / 2^l samples: 0.7-1.5 against 1.6-3.7 2^-53
// on levels 0 to 2), also where 1 / S has come through 1,024 factors (level 10,
// sigma 0.2: 11.7 against 12.0).  8,000,000 level-0 samples, 57,344 partials per
// value: 2.75 -> 2.09 ms with 128 threads a value instead of 32.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "device_common.cuh"
#include "exact64.cuh"
#include "host_api.h"
#include "item.h"
#include "mlmc.h"

using namespace mlmc;

namespace {

constexpr int SENS_THREADS = 128;
constexpr int SENS_MAX_LEVEL = 10;
// per-instance rows: S-type (= mul2 except S0), sum1-type (= mul1), Z
constexpr int SENS_ROWS = 3;
enum { T_Z = 0, T_CON1 = 1, T_CON2 = 2, T_MUL1 = 3, T_SUM1 = 4, T_MUL2 = 5, T_S = 6 };
// per-CTA scalars: sums, then maxima
enum { P_DP, P_DP2, P_C1F, P_C1C, P_C2, P_S0, P_SUMS, P_ZHI = P_SUMS, P_ZLO, P_ZCHI, P_ZCLO, P_MUL2, P_S, P_COUNT };

struct SensConsts {
  double con1, con1c, con2, S0, K, disc;
  int level, n, m, ni;
  uint64_t first, N;
  uint32_t ctr2, ctr3;
  int64_t q1;          // integer increments (exact64.cuh; qF 0: they may reach 8, formed in FP64)
  uint64_t q2;
  int qF;
};

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __forceinline__ double warp_max(double x) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

// The larger of |x| and the running maximum m >= 0, by integer comparison (a NaN loses).
__device__ __forceinline__ void max_abs(double &m, double x) {
  const long long b = __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFLL;
  if (b > __double_as_longlong(m) && b <= 0x7FF0000000000000LL) m = __longlong_as_double(b);
}

// Tape of a CTA's 128 samples: u and 1 / S of the fine steps [sample][n], then of
// the coarse steps [sample][m].
__host__ __device__ inline size_t tape_doubles(int n, int m) { return (size_t)SENS_THREADS * 2 * (n + m); }
// Accumulators of pass 2 in shared memory: 3 fine rows of max(n, 128) and 2
// coarse rows of max(m, 128) (below 128 instances several threads share one,
// each with the samples of its residue).
__host__ __device__ inline int slots(int n) { return n > SENS_THREADS ? n : SENS_THREADS; }

__global__ void __launch_bounds__(SENS_THREADS, 4) sens_kernel(const SensConsts c, const RoundKeys rk, uint64_t iters,
                                                            double *part, double *inst_part, double *tapes) {
  extern __shared__ double acc[];
  __shared__ double sF[SENS_THREADS], sG[SENS_THREADS], wp[P_COUNT][SENS_THREADS / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = c.n, m = c.m, nf = slots(n), nc = m > 0 ? slots(m) : 0;
  double *fine = acc, *coarse = acc + 3 * nf;
  for (int i = tid; i < 3 * nf + 2 * nc; i += SENS_THREADS) acc[i] = 0.0;
  stage_phi64();
  copies_done();
  __syncthreads();
  const ulonglong2 *phi = phi64_smem();
  double *tu = tapes + tape_doubles(n, m) * blockIdx.x, *tr = tu + (size_t)SENS_THREADS * n;
  double *tv = tr + (size_t)SENS_THREADS * n, *tw = tv + (size_t)SENS_THREADS * m;
  const uint32_t qhi = (uint32_t)(1085 - c.qF) << 20, zhi0 = (uint32_t)(1085 - 59) << 20;
  const double rS0 = 1.0 / c.S0;
  double ps[P_SUMS] = {0, 0, 0, 0, 0, 0}, mm2 = 0.0, mS = c.S0;
  // extremes of Z (units 2^-59) on the fine and the coarse path; a lane without a
  // sample of its own repeats sample `first`, which changes no extreme
  long long z_hi = -0x7FFFFFFFFFFFFFFFLL, z_lo = 0x7FFFFFFFFFFFFFFFLL, zc_hi = z_hi, zc_lo = z_lo;
  const uint64_t stride = (uint64_t)gridDim.x * SENS_THREADS;
  for (uint64_t it = 0; it < iters; ++it) {
    if (it * stride + (uint64_t)blockIdx.x * SENS_THREADS >= c.N) break;   // no sample for this CTA
    const uint64_t rel = it * stride + (uint64_t)blockIdx.x * SENS_THREADS + tid;
    const bool valid = rel < c.N;
    const uint64_t s = c.first + (valid ? rel : 0);
    // ---- pass 1: both paths, u and 1 / S of every step to the tape ----
    double S = c.S0, Sc = c.S0, r = rS0, rc = rS0, u1 = 0.0, zu = 0.0, v1 = 0.0, zcv = 0.0;
    long long zprev = 0, qprev = 0;
    // one step of a path from its Normal zq 2^-59 and increment q 2^-qF
    auto advance = [&](long long zq, long long q, double con1, double &St, double &rt, double &a1, double &az) {
      const double z = q_to_double(zq, zhi0);
      const double sum1 = c.qF ? q_to_double(q, qhi) : fma(c.con2, z, con1);
      const double mul2 = St * sum1;
      St = St + mul2;
      const double u = reciprocal(1.0 + sum1);
      rt *= u;
      a1 += u;
      az = fma(z, u, az);
      max_abs(mm2, mul2);
      max_abs(mS, St);
      return u;
    };
    for (int k0 = 0; k0 < n; k0 += 4) {
      const uint64_t wi = (s << c.level) + (uint64_t)k0;
      const uint4 w = philox4x32_10(make_uint4((uint32_t)(wi >> 2), (uint32_t)(wi >> 34), c.ctr2, c.ctr3), rk);
      double us[4], rs[4], vs[2], ws[2];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (k0 + j >= n) break;
        const uint32_t J = word_of(w, (int)((wi + j) & 3));
        const int32_t mk = (int32_t)J >> 31;   // Z = y in the upper half, -y below
        const uint64_t y = probit_q60(J ^ (uint32_t)mk, phi);
        const long long zq = mk ? (long long)(y >> 1) : -(long long)(y >> 1);
        const long long q = c.q1 + (long long)(mulhi64_3(c.q2, y) ^ (uint64_t)(int64_t)~mk);
        z_hi = max(z_hi, zq);
        z_lo = min(z_lo, zq);
        us[j] = advance(zq, q, c.con1, S, r, u1, zu);
        rs[j] = r;
        if (m > 0 && (j & 1)) {
          const long long zc = zprev + zq;
          zc_hi = max(zc_hi, zc);
          zc_lo = min(zc_lo, zc);
          vs[j >> 1] = advance(zc, qprev + q, c.con1c, Sc, rc, v1, zcv);
          ws[j >> 1] = rc;
        }
        zprev = zq;
        qprev = q;
      }
      const size_t f = (size_t)tid * n + k0, g = (size_t)tid * m + (k0 >> 1);
      if (n >= 4) {
        *(double2 *)(tu + f) = make_double2(us[0], us[1]);
        *(double2 *)(tu + f + 2) = make_double2(us[2], us[3]);
        *(double2 *)(tr + f) = make_double2(rs[0], rs[1]);
        *(double2 *)(tr + f + 2) = make_double2(rs[2], rs[3]);
        *(double2 *)(tv + g) = make_double2(vs[0], vs[1]);
        *(double2 *)(tw + g) = make_double2(ws[0], ws[1]);
      } else {
        tu[f] = us[0];
        tr[f] = rs[0];
        if (n == 2) {
          tu[f + 1] = us[1];
          tr[f + 1] = rs[1];
          tv[g] = vs[0];
          tw[g] = ws[0];
        }
      }
    }
    const bool inF = valid && S > c.K, inG = valid && m > 0 && Sc > c.K;
    const double F = inF ? c.disc * S : 0.0, G = inG ? -c.disc * Sc : 0.0;
    sF[tid] = F;
    sG[tid] = G;
    const double dp = (inF ? c.disc * (S - c.K) : 0.0) - (inG ? c.disc * (Sc - c.K) : 0.0);
    const double a1f = F * u1, a1c = G * v1, a2 = fma(F, zu, G * zcv), sS0 = (F + G) * rS0;
    ps[P_DP] += dp;
    ps[P_DP2] = fma(dp, dp, ps[P_DP2]);
    ps[P_C1F] = fma(a1f, a1f, ps[P_C1F]);
    ps[P_C1C] = fma(a1c, a1c, ps[P_C1C]);
    ps[P_C2] = fma(a2, a2, ps[P_C2]);
    ps[P_S0] = fma(sS0, sS0, ps[P_S0]);
    __syncthreads();
    // ---- pass 2: a thread per instance (several, each with a residue of the samples, below 128) ----
    for (int i = tid; i < nf; i += SENS_THREADS) {
      const int k = i & (n - 1), step = nf / n;
      double a0 = 0.0, a1 = 0.0, a2s = 0.0;
      for (int t = i / n; t < SENS_THREADS; t += step) {
        const double Ft = sF[t];
        const double a = Ft * tr[(size_t)t * n + k], b = Ft * tu[(size_t)t * n + k];
        const double z = m > 0 ? fma(sG[t], tv[(size_t)t * m + (k >> 1)], b) : b;
        a0 = fma(a, a, a0);
        a1 = fma(b, b, a1);
        a2s = fma(z, z, a2s);
      }
      fine[i] += a0;
      fine[nf + i] += a1;
      fine[2 * nf + i] += a2s;
    }
    for (int i = tid; i < nc; i += SENS_THREADS) {
      const int k = i & (m - 1), step = nc / m;
      double a0 = 0.0, a1 = 0.0;
      for (int t = i / m; t < SENS_THREADS; t += step) {
        const double Gt = sG[t];
        const double a = Gt * tw[(size_t)t * m + k], b = Gt * tv[(size_t)t * m + k];
        a0 = fma(a, a, a0);
        a1 = fma(b, b, a1);
      }
      coarse[i] += a0;
      coarse[nc + i] += a1;
    }
    __syncthreads();
  }
  // ---- CTA reduction (warp order) ----
  const double zs = 0x1p-59, cs = m > 0 ? zs : 0.0;
  const double mx[P_COUNT - P_SUMS] = {(double)z_hi * zs,  -(double)z_lo * zs, (double)zc_hi * cs,
                                       -(double)zc_lo * cs, mm2,                mS};
#pragma unroll
  for (int t = 0; t < P_COUNT; ++t) {
    const double x = t < P_SUMS ? warp_sum(ps[t < P_SUMS ? t : 0]) : warp_max(mx[t < P_SUMS ? 0 : t - P_SUMS]);
    if (lane == 0) wp[t][warp] = x;
  }
  __syncthreads();
  if (tid < P_COUNT) {
    double x = wp[tid][0];
    for (int w = 1; w < SENS_THREADS / 32; ++w) x = tid < P_SUMS ? x + wp[tid][w] : fmax(x, wp[tid][w]);
    part[(size_t)blockIdx.x * P_COUNT + tid] = x;
  }
  // the threads that shared an instance (below 128 of them), halves onto halves: at
  // level 0 the terms of a row are all alike, and 128 additions in a row rounded
  // them all the same way
  auto fold = [&](double *a, int row_count, int len, int instances) {
    for (int half = len / 2; half >= instances; half /= 2) {
      if (tid < half)
        for (int r = 0; r < row_count; ++r) a[r * len + tid] += a[r * len + tid + half];
      __syncthreads();
    }
  };
  fold(fine, 3, nf, n);
  if (m > 0) fold(coarse, 2, nc, m);
  double *out = inst_part + (size_t)blockIdx.x * SENS_ROWS * c.ni;
  for (int i = tid; i < SENS_ROWS * c.ni; i += SENS_THREADS) {
    const int row = i / c.ni, k = i - row * c.ni;
    out[i] = k < n ? fine[row * nf + k] : k < n + m && row < 2 ? coarse[row * nc + k - n] : 0.0;
  }
}

// The CTA partials' totals, a CTA per value: P_COUNT scalars, then the rows.
// Thread t adds the partials t, t + 128, ...  with the roundings collected in a
// second sum (TwoSum: there are up to 57,000 partials), then two butterflies.
__global__ void sens_finalize_kernel(const double *part, const double *inst_part, int n_ctas, int rows, double *res) {
  __shared__ double warp_total[SENS_THREADS / 32];
  const int v = blockIdx.x, tid = threadIdx.x;
  const double *p = v < P_COUNT ? part + v : inst_part + (v - P_COUNT);
  const size_t pitch = v < P_COUNT ? P_COUNT : rows;
  const bool is_max = v >= P_SUMS && v < P_COUNT;
  double x = is_max ? -1e300 : 0.0, err = 0.0;
  for (int b = tid; b < n_ctas; b += SENS_THREADS) {
    const double y = p[b * pitch];
    if (is_max) {
      x = fmax(x, y);
    } else {
      const double t = x + y, z = t - x;
      err += (x - (t - z)) + (y - z);
      x = t;
    }
  }
  x = is_max ? warp_max(x) : warp_sum(x + err);
  if ((tid & 31) == 0) warp_total[tid >> 5] = x;
  __syncthreads();
  if (tid == 0) {
    const double a = warp_total[0], b = warp_total[1], d = warp_total[2], e = warp_total[3];
    res[v] = is_max ? fmax(fmax(a, b), fmax(d, e)) : (a + b) + (d + e);
  }
}

// Device workspace and pinned result staging, kept between calls (under the
// library lock, each call synchronises): up to SENS_KEEP bytes, more is given
// back at the end of the call, and all of it when another allocation of the
// library fails (error_model_release).
constexpr size_t SENS_KEEP = (size_t)128 << 20, SENS_MAX_TAPE = (size_t)1 << 30;
struct SensSpace {
  int device = -1;
  char *d = nullptr;
  size_t cap = 0;
  double *h = nullptr;
  size_t h_cap = 0;
  bool reserve_device(int dev, size_t bytes) {
    if (d && (dev != device || bytes > cap)) release();
    if (!d) {
      if (cudaMalloc(&d, bytes) != cudaSuccess) {
        (void)cudaGetLastError();
        d = nullptr;
        return false;
      }
      cap = bytes;
      device = dev;
    }
    return true;
  }
  bool reserve_host(size_t doubles) {
    if (doubles <= h_cap) return true;
    if (h) cudaFreeHost(h);
    h = nullptr;
    h_cap = 0;
    if (cudaHostAlloc((void **)&h, sizeof(double) * doubles, cudaHostAllocDefault) != cudaSuccess) {
      (void)cudaGetLastError();
      h = nullptr;
      return false;
    }
    h_cap = doubles;
    return true;
  }
  void release() {
    if (d) cudaFree(d);
    d = nullptr;
    cap = 0;
  }
};
SensSpace g_sens;

}  // namespace

bool mlmc_host::error_model_release() {
  const bool had = g_sens.d != nullptr;
  g_sens.release();
  return had;
}

extern "C" mlmc_status mlmc_sensitivities(int level, uint64_t N, const mlmc_params *p, uint64_t seed,
                                          uint64_t first_sample, mlmc_sensitivity *out, double *inst_out) {
  MLMC_API_LOCK();
  using namespace mlmc_host;
  if (!out || !p || !params_ok(p) || level < 0 || level > SENS_MAX_LEVEL || N == 0) return MLMC_EINVAL;
  if (p->payoff != MLMC_EURO || p->scheme != MLMC_EULER) return MLMC_EINVAL;
  if (N > (1ULL << 40) || first_sample > (1ULL << (60 - level)) - N) return MLMC_EINVAL;
  mlmc_status s = ensure_ctx();
  if (s != MLMC_OK) return s;
  SensConsts c;
  std::memset(&c, 0, sizeof c);
  const double h = std::ldexp(p->T, -level);
  c.con1 = p->r * h;
  c.con1c = p->r * (2.0 * h);
  c.con2 = p->sigma * std::sqrt(h);
  c.S0 = p->S0;
  c.K = p->K;
  c.disc = std::exp(-p->r * p->T);
  c.level = level;
  c.n = 1 << level;
  c.m = level > 0 ? c.n / 2 : 0;
  c.ni = c.n + c.m + 1;
  c.first = first_sample;
  c.N = N;
  c.ctr2 = (uint32_t)level;   // stream 0
  c.ctr3 = p->request_id;
  RoundKeys rk;
  make_round_keys(seed, rk);
  {
    ItemDesc it;
    std::memset(&it, 0, sizeof it);
    it.level = level;
    it.c1d = c.con1; it.c1cd = c.con1c; it.c2d = c.con2;
    exact64_consts(it, false);
    c.q1 = it.q1; c.q2 = it.q2; c.qF = it.qF;
  }
  // a CTA per 128 samples while their tapes fit the kept workspace, at least the
  // four per SM that run at once (where the tape allows)
  const size_t tape = sizeof(double) * tape_doubles(c.n, c.m);
  const uint64_t want = std::max<uint64_t>(std::min<uint64_t>((uint64_t)4 * ctx_num_sms(), SENS_MAX_TAPE / tape),
                                           (SENS_KEEP - SENS_KEEP / 8) / tape);
  int n_ctas = (int)std::min<uint64_t>(want, (N + SENS_THREADS - 1) / SENS_THREADS);
  const size_t smem = sizeof(double) * (3 * (size_t)slots(c.n) + (c.m > 0 ? 2 * (size_t)slots(c.m) : 0));
  cudaStream_t st = ctx_stream();
  const size_t rows = (size_t)SENS_ROWS * c.ni, n_res = P_COUNT + rows;
  int dev = 0;
  MLMC_CK(cudaGetDevice(&dev));
  if (!g_sens.reserve_host(n_res)) return MLMC_ENOMEM;
  // any number of CTAs gives the statistics: half as many, down to one, where
  // the device has no room for their tapes
  while (!g_sens.reserve_device(dev, sizeof(double) * ((size_t)n_ctas * (tape / sizeof(double) + P_COUNT + rows) + n_res))) {
    if (n_ctas == 1) return MLMC_ENOMEM;
    n_ctas = (n_ctas + 1) / 2;
  }
  const uint64_t per = (uint64_t)n_ctas * SENS_THREADS, iters = (N + per - 1) / per;
  double *d_tape = (double *)g_sens.d, *d_part = d_tape + (size_t)n_ctas * (tape / sizeof(double));
  double *d_ip = d_part + (size_t)n_ctas * P_COUNT, *d_res = d_ip + (size_t)n_ctas * rows;
  mlmc_status rs = MLMC_OK;
  if (smem > 24 * 1024 &&
      cudaFuncSetAttribute(sens_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    rs = MLMC_ECUDA;
  if (rs == MLMC_OK) {
    sens_kernel<<<n_ctas, SENS_THREADS, smem, st>>>(c, rk, iters, d_part, d_ip, d_tape);
    sens_finalize_kernel<<<(unsigned)n_res, SENS_THREADS, 0, st>>>(d_part, d_ip, n_ctas, (int)rows, d_res);
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(g_sens.h, d_res, sizeof(double) * n_res, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      rs = MLMC_ECUDA;
  }
  if (g_sens.cap > SENS_KEEP) g_sens.release();
  if (rs != MLMC_OK) return rs;
  // per-instance second moments, type-major 7 x ni
  const double *res = g_sens.h, *rowsum = g_sens.h + P_COUNT;
  const int ni = c.ni, n = c.n, m = c.m;
  std::vector<double> E((size_t)7 * ni, 0.0);
  const double inv = 1.0 / (double)N;
  for (int i = 0; i < n + m; ++i) {
    E[(size_t)T_S * ni + i] = rowsum[i] * inv;
    E[(size_t)T_MUL2 * ni + i] = rowsum[i] * inv;
    E[(size_t)T_SUM1 * ni + i] = rowsum[ni + i] * inv;
    E[(size_t)T_MUL1 * ni + i] = rowsum[ni + i] * inv;
  }
  for (int j = 0; j < n; ++j) E[(size_t)T_Z * ni + j] = c.con2 * c.con2 * rowsum[2 * ni + j] * inv;
  E[(size_t)T_S * ni + n + m] = res[P_S0] * inv;
  E[(size_t)T_CON1 * ni + 0] = res[P_C1F] * inv;
  E[(size_t)T_CON1 * ni + 1] = res[P_C1C] * inv;
  E[(size_t)T_CON2 * ni + 0] = res[P_C2] * inv;
  std::memset(out, 0, sizeof *out);
  // maxima: sum1 and mul1 are monotone in Z, so its extremes give theirs
  auto larger = [](double a, double b) { return std::max(std::fabs(a), std::fabs(b)); };
  const double zh = res[P_ZHI], zl = -res[P_ZLO], ch = res[P_ZCHI], cl = -res[P_ZCLO];
  double mul1 = c.con2 * larger(zh, zl), sum1 = larger(c.con1 + c.con2 * zh, c.con1 + c.con2 * zl);
  if (m > 0) {
    mul1 = std::max(mul1, c.con2 * larger(ch, cl));
    sum1 = std::max(sum1, larger(c.con1c + c.con2 * ch, c.con1c + c.con2 * cl));
  }
  const double mx[7] = {larger(zh, zl), larger(c.con1, m > 0 ? c.con1c : 0.0), std::fabs(c.con2), mul1, sum1,
                        res[P_MUL2], res[P_S]};
  for (int t = 0; t < 7; ++t) {
    double a = 0.0, b = 0.0;
    for (int i = 0; i < ni; ++i) {
      a += E[(size_t)t * ni + i];
      b += std::sqrt(E[(size_t)t * ni + i]);
    }
    out->A[t] = a;
    out->B[t] = b;
    out->maxabs[t] = mx[t];
  }
  out->mean = res[P_DP] * inv;
  out->var = std::max(0.0, res[P_DP2] * inv - out->mean * out->mean);
  out->n = N;
  out->n_instances = ni;
  if (inst_out) std::memcpy(inst_out, E.data(), sizeof(double) * E.size());
  return MLMC_OK;
}

// descent.cuh -- strategy parameters, the state of a fresh descent and the
// restart, shared by the phase kernels (kernels_gen.cu) and the one-CTA
// generation of small searches (kernels_small.cu).
#pragma once
#include <cmath>
#include <cuda_bf16.h>
#include "device_common.cuh"

namespace cmaes_gb300 {

// --------------------------- strategy parameters ----------------------------
// Tutorial defaults (Hansen, arXiv:1604.00772) for the constants the paper
// leaves to the c-cmaes code (§4.1): log weights on the best floor(lambda/2)
// points summing to one (Eq. (2)), mu_eff, c_sigma, d_sigma, c_c, c_1, c_mu,
// E||N(0,I)||, the lazy eigendecomposition period, the history length of the
// "quality not improving" test and the iteration cap.
template <int NT>
__device__ void compute_params(Search& s, const DevOptions& o, double* sh) {
  const int n = s.n, lam = s.lam, mu = lam / 2;
  const double lw = log((lam + 1) / 2.0);
  double part = 0.0;
  for (int i = threadIdx.x; i < mu; i += NT) {  // (a logarithm is ~30 FP64 operations: each is taken once)
    const double v = lw - log(static_cast<double>(i + 1));
    s.w[i] = v;
    part += v;
  }
  const double sum = block_sum<NT>(part, sh);
  double sq = 0.0;
  for (int i = threadIdx.x; i < mu; i += NT) {
    const double wi = s.w[i] / sum;
    s.w[i] = wi;
    if (s.mixed) s.w32[i] = static_cast<float>(wi);
    sq += wi * wi;
  }
  const double ssq = block_sum<NT>(sq, sh);
  if (threadIdx.x == 0) {
    const double dn = static_cast<double>(n);
    const double mueff = 1.0 / ssq;
    s.mu = mu;
    s.mueff = mueff;
    s.cs = (mueff + 2.0) / (dn + mueff + 5.0);
    s.ds = 1.0 + 2.0 * fmax(0.0, sqrt((mueff - 1.0) / (dn + 1.0)) - 1.0) + s.cs;
    s.cc = (4.0 + mueff / dn) / (dn + 4.0 + 2.0 * mueff / dn);
    s.c1 = 2.0 / ((dn + 1.3) * (dn + 1.3) + mueff);
    s.cmu = fmin(1.0 - s.c1, 2.0 * (mueff - 2.0 + 1.0 / mueff) / ((dn + 2.0) * (dn + 2.0) + mueff));
    s.chin = sqrt(dn) * (1.0 - 1.0 / (4.0 * dn) + 1.0 / (21.0 * dn * dn));
    const int lazy = static_cast<int>(floor(1.0 / ((s.c1 + s.cmu) * dn * 10.0)));
    s.g_eig = o.eig_every > 0 ? o.eig_every : (lazy > 1 ? lazy : 1);
    s.hist_len = 10 + static_cast<int>(ceil(30.0 * dn / lam));
    s.max_iter = o.max_iter > 0
                     ? o.max_iter
                     : static_cast<int>(floor(100.0 + 50.0 * (dn + 3.0) * (dn + 3.0) / sqrt(static_cast<double>(lam))));
  }
  __syncthreads();
}

// Fresh descent state (Algorithm 2, "initialize"): C = B = I, D = 1, paths
// zero, sigma = sigma0. The mean is set by the caller.
template <int NT>
__device__ void reset_descent(Search& s) {
  const int n = s.n, ldn = s.ldn;
  for (int i = threadIdx.x; i < n; i += NT) {
    s.ps[i] = 0.0;
    s.pc[i] = 0.0;
    s.D[i] = 1.0;
  }
  for (long long e = threadIdx.x; e < static_cast<long long>(ldn) * n; e += NT) {
    const int i = static_cast<int>(e % ldn), j = static_cast<int>(e / ldn);
    const double v = (i == j) ? 1.0 : 0.0;
    s.C[e] = v;
    s.B[e] = v;
    s.BD[e] = v;
  }
  if (s.mixed) {  // tensor-core copy of B D: identity as well
    const int kp = s.kp;
    for (long long e = threadIdx.x; e < static_cast<long long>(n) * kp; e += NT) {
      const int i = static_cast<int>(e / kp), k = static_cast<int>(e % kp);
      const float v = (i == k) ? 1.0f : 0.0f;
      if (s.mixed == 2) static_cast<__nv_bfloat16*>(s.BDT)[e] = __float2bfloat16_rn(v);
      else static_cast<float*>(s.BDT)[e] = v;
    }
  }
  if (threadIdx.x == 0) {
    s.sigma = s.sigma0;
    s.gen = 0;
    s.hist_count = 0;
    s.eig_due = 0;
  }
}

// The restart of Algorithm 2: lambda doubled (or kept), a uniform mean in the
// box, C = B = I.
template <int NT>
__device__ void restart_descent(Search& s, const DevOptions& o, double* sh) {
  __syncthreads();
  if (threadIdx.x == 0) {
    s.restart += 1;
    if (o.ipop_double) s.lam *= 2;
  }
  __syncthreads();
  reset_descent<NT>(s);
  for (int i = threadIdx.x; i < s.n; i += NT)
    s.m[i] = restart_mean_coord(i, s.index, s.restart, o.key0, o.key1, o.box_lo, o.box_hi);
  __syncthreads();
  compute_params<NT>(s, o, sh);
}

// The formulas that the phase kernels, the one-CTA generations and the allocation-free
// evaluation share, with the rounding of each operation written out: the same state
// gives the same bits through any of them.
__device__ __forceinline__ double objective_term(int obj, double lam, double u) {
  return obj == 1 ? __dmul_rn(__dmul_rn(lam, u), u) : fma(u, u, __dmul_rn(-10.0, cospi(2.0 * u)));
}
// x = m + sigma y, also the mean's step
__device__ __forceinline__ double step_from(double m, double sigma, double y) { return fma(sigma, y, m); }
// (1 - c) p + coef v of the two paths
__device__ __forceinline__ double path_step(double c, double p, double coef, double v) {
  return fma(coef, v, __dmul_rn(1.0 - c, p));
}
// Eq. (2): the weight of the old C, and an entry of the new one
__device__ __forceinline__ double cov_keep(double c1, double cmu, double cc, double hsig) {
  return fma(__dmul_rn(__dmul_rn(c1, 1.0 - hsig), cc), 2.0 - cc, 1.0 - c1 - cmu);
}
__device__ __forceinline__ double cov_entry(double keep, double c, double c1, double pi, double pj, double cmu,
                                            double acc) {
  return fma(cmu, acc, fma(__dmul_rn(c1, pi), pj, __dmul_rn(keep, c)));
}

// Order-preserving 64-bit integer key of f: NaN -> +inf, -0 -> +0, then the
// IEEE bit pattern with the sign folded so that unsigned order = numeric order.
// (Comparing integers keeps the O(lambda^2) count off GB300's slow FP64 pipe.)
__device__ __forceinline__ unsigned long long rank_key(double f) {
  if (isnan(f)) f = INFINITY;
  if (f == 0.0) f = 0.0;
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(f));
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

}  // namespace cmaes_gb300

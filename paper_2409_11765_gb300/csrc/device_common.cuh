// device_common.cuh -- device helpers shared by the engine's kernels:
// Philox4x32-10 draws, tile lookup over uneven searches, fixed-order block
// reductions and the FP64 GEMM tile used by the sampling, objective,
// covariance and eigensolver-setup products.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include "engine.h"

namespace cmaes_gb300 {

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of
//   (hi0, lo0) = M0 * c0, (hi1, lo1) = M1 * c2,
//   c = (hi1 ^ c1 ^ k0, lo1, hi0 ^ c3 ^ k1, lo0),
// with the key bumped by the Weyl constants between rounds.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * c.x;
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
  }
  return c;
}

// 52-bit uniform in (0, 1) from two words: (top 52 bits + 1/2) * 2^-52, exact.
__device__ __forceinline__ double uniform52(uint32_t a, uint32_t b) {
  const unsigned long long v = ((static_cast<unsigned long long>(a) << 32) | b) >> 12;
  return (static_cast<double>(v) + 0.5) * 0x1p-52;
}

__device__ __forceinline__ uint32_t stream_word(int search, int restart) {
  return (static_cast<uint32_t>(search) << 8) | (static_cast<uint32_t>(restart) & 255u);
}

// Box-Muller pair for coordinates (2j, 2j+1) of candidate k in generation g.
__device__ __forceinline__ void normal_pair(uint32_t j, uint32_t k, uint32_t g, uint32_t sw,
                                            uint32_t k0, uint32_t k1, double& z0, double& z1) {
  const uint4 w = philox4x32_10(make_uint4(j, k, g, sw), k0, k1);
  const double u1 = uniform52(w.x, w.y);
  const double u2 = uniform52(w.z, w.w);
  const double r = sqrt(-2.0 * log(u1));
  const double a = (2.0 * 3.141592653589793) * u2;
  double s, c;
  sincos(a, &s, &c);
  z0 = r * c;
  z1 = r * s;
}

// Uniform coordinate i of the mean of descent `restart` in [lo, hi].
__device__ __forceinline__ double restart_mean_coord(int i, int search, int restart, uint32_t k0,
                                                     uint32_t k1, double lo, double hi) {
  const uint4 w = philox4x32_10(
      make_uint4(static_cast<uint32_t>(i) >> 1, 0xFFFFFFFFu, 0xFFFFFFFFu, stream_word(search, restart)),
      k0, k1);
  const double u = (i & 1) ? uniform52(w.z, w.w) : uniform52(w.x, w.y);
  return lo + (hi - lo) * u;
}

// ---------------------------------------------------------------------------
// Tile lookup: the launch covers searches [s0, s1); tile blockIdx.x maps to
// the search whose prefix range holds off[s0] + blockIdx.x.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int find_search(const TileMap& tm, int& local) {
  const int t = tm.off[tm.s0] + static_cast<int>(blockIdx.x);
  int lo = tm.s0, hi = tm.s1 - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tm.off[mid] <= t) lo = mid; else hi = mid - 1;
  }
  local = t - tm.off[lo];
  return lo;
}

// Fixed-order block reductions (the same blockDim always sums in the same
// order, so results are reproducible run to run).
template <int NT>
__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0) {
    for (int w = 0; w < NT / 32; ++w) r += sh[w];
    sh[0] = r;
  }
  __syncthreads();
  r = sh[0];
  __syncthreads();
  return r;
}

template <int NT>
__device__ __forceinline__ double block_max(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = sh[0];
    for (int w = 1; w < NT / 32; ++w) r = fmax(r, sh[w]);
    sh[0] = r;
  }
  __syncthreads();
  const double r = sh[0];
  __syncthreads();
  return r;
}

template <int NT>
__device__ __forceinline__ int block_or(int v, int* sh) {
  v = __reduce_or_sync(0xffffffffu, v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  int r = 0;
  for (int w = 0; w < NT / 32; ++w) r |= sh[w];
  __syncthreads();
  return r;
}

// ---------------------------------------------------------------------------
// FP64-accurate GEMM tile: out(i, j) = sum_k a(i, k) b(k, j) over a 64 x 64
// tile, K in steps of 32, 256 threads with 4 x 4 outputs each. The operand
// accessors are functors so that gathers (selected columns), offsets
// (x - x*) and transposes are applied while staging into shared memory;
// A_I_CONTIG / B_K_CONTIG say which index is contiguous in memory so the
// staging loads coalesce. The order of every sum is fixed.
//
// GB300 issues 1.7 FP64 FMAs per clock and SM and 28 32 x 32 + 64-bit integer
// multiply-adds, so the products run on integers: within a K step row i of A
// (and column j of B) is scaled by the power of two above its largest entry and
// rounded to 57 bits, x = (h 2^29 + l) 2^(e - 57) with |h|, |l| <= 2^28; h h and
// h l + l h are summed exactly (below 2^61 and 2^62 over 32 k), and the step's
// sum, to within 2^-57 of the two scales, is added to the FP64 accumulator: three
// integer multiply-adds per term instead of one FP64 FMA, two FP64 operations per
// output and step.
//
// The step's error, ~2^-57 of the product of the scales (rms), is small against
// sum |a b| only where large entries of the row meet large ones of the column; an
// axis-aligned rotation, or a row graded over many orders, has outputs where they
// do not. So sum |a b| is also formed to 8 bits a factor (eight dp4a per output and
// step), and an output where it is below 2^-4 of the scales' product, so that the
// error could pass an FP64 rounding of sum |a b|, takes the step's FMAs in FP64 from
// the entries themselves; so does one whose row or column has an infinite or NaN
// entry or scales near the ends of the exponent range. No output depends on which
// others share its tile. Rotated and evenly scaled operands have no such output:
// against 113-bit arithmetic the objectives come out 1.2 to 3 times closer than with
// FMAs (n = 100, rastrigin: 1.1e-16 rms, was 2.3e-16; n = 1000: 7.8e-17, was
// 2.5e-16). The steps split K evenly: a last step of a few k would meet them by chance.
// Bound by the integer multiply-adds and, beside them, by staging, which two CTAs per SM
// overlap (PER_SM = 2, 128 registers) where there are more tiles than SMs; a tile that
// has an SM to itself runs faster with the registers that the compiler takes (PER_SM = 1,
// 172). n = 500, 88 tiles and 168: 229 and 442 us with one, 248 and 384 with two.
// Evaluating 8704 points of n = 100: 305 us in FP64 FMAs, 143 here (its multiply-adds
// alone, tile padding included, take ~40), 270 if every output were to go to FP64.
// ---------------------------------------------------------------------------
constexpr int kGBM = 64, kGBN = 64, kGBK = 32, kGNT = 256;
constexpr int kGSms = 152;  // tiles from which on two CTAs share an SM

struct GemmSmem {
  int2 As[kGBK][kGBM + 1];  // limbs (h, l), or the doubles themselves
  int2 Bs[kGBK][kGBN + 1];
  unsigned ma[kGBK / 4][kGBM + 1];  // the entries' magnitudes to 8 bits, four k a word
  unsigned mb[kGBK / 4][kGBN + 1];
  int ea[kGBM], eb[kGBN];
};

// k per step: K split evenly into as few steps as there can be.
__host__ __device__ inline int gemm_step(int K) {
  const int steps = (K + kGBK - 1) / kGBK;
  return steps > 0 ? (K + steps - 1) / steps : kGBK;
}

// The biased exponent of x for the scales (1 for a subnormal number).
__device__ __forceinline__ int gemm_exponent(double x) {
  const int hi = __double2hiint(x), be = (hi >> 20) & 0x7ff;
  return be | static_cast<int>(be == 0 && ((hi << 1) | __double2loint(x)) != 0);
}

// The limbs of x for a scale with biased exponent E (|x| < 2^(E - 1022)): x rounded
// to 2 H - 1 bits of it, x = (h 2^H + l) 2^(E - 1022 - (2 H - 1)), |h|, |l| <= 2^(H - 1).
template <int H>
__device__ __forceinline__ int2 gemm_limbs(double x, int E) {
  const int hi = __double2hiint(x), be = (hi >> 20) & 0x7ff;
  long long m = (static_cast<long long>((hi & 0xfffff) | 0x100000) << 32) | static_cast<unsigned>(__double2loint(x));
  const int s = E - be - (2 * H - 54);
  if (s <= 0) m <<= -s;
  else m = s > 54 ? 0 : (m + (1LL << (s - 1))) >> s;
  if (be == 0) m = 0;
  if (hi < 0) m = -m;
  const int h = static_cast<int>((m + (1LL << (H - 1))) >> H);
  return make_int2(h, static_cast<int>(m - (static_cast<long long>(h) << H)));
}

// 8 bits of the magnitude of an entry with limb h (of gemm_limbs<29>), 2^-8 of the
// scale each.
__device__ __forceinline__ unsigned gemm_byte(int h) { return min(static_cast<unsigned>(abs(h)) >> 20, 255u); }

// Whether a step's output goes to FP64: `sum` is the dot product of those bytes, ea and
// eb the scales' biased exponents (0: only zeros there).
__device__ __forceinline__ bool gemm_in_f64(unsigned sum, int ea, int eb) {
  constexpr unsigned kLeast = 1u << 12;  // 2^-4 of the scales' product
  return ea != 0 && eb != 0 && (sum < kLeast || min(ea, eb) < 64 || max(ea, eb) == 0x7ff);
}

// The value of sum (h h) + sum (h l + l h) / 2^H over two operands of that form
// whose scales have the biased exponents ea and eb, e2 = ea + eb.
template <int H>
__device__ __forceinline__ double gemm_scaled(long long hh, long long mid, int e2) {
  const long long s = hh + ((mid + (1LL << (H - 1))) >> H);
  const int e = e2 - 2042 - 2 * H;
  const double d = static_cast<double>(s);
  const int hi = __double2hiint(d), be = ((hi >> 20) & 0x7ff) + e;
  if (s == 0) return 0.0;
  if (be <= 0 || be >= 2047) return scalbn(d, e);
  return __hiloint2double(hi + (e << 20), __double2loint(d));
}

template <int PER_SM, bool A_I_CONTIG, bool B_K_CONTIG, class LA, class LB, class EPI>
__device__ __forceinline__ void gemm_tile_f64(int M, int N, int K, int i0, int j0, const LA& la,
                                              const LB& lb, const EPI& epi, GemmSmem& sm) {
  const int tid = threadIdx.x;
  const int tr = tid & 15, tc = tid >> 4;
  constexpr int Q = kGBM * kGBK / kGNT;  // elements of each operand per thread
  double acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.0;
  // element q of this thread: A(ai, ak), B(bk, bj)
  auto ai = [&](int q) { return A_I_CONTIG ? (tid & 63) : (tid >> 5) + 8 * q; };
  auto ak = [&](int q) { return A_I_CONTIG ? (tid >> 6) + 4 * q : (tid & 31); };
  auto bj = [&](int q) { return B_K_CONTIG ? (tid >> 5) + 8 * q : (tid & 63); };
  auto bk = [&](int q) { return B_K_CONTIG ? (tid & 31) : (tid >> 6) + 4 * q; };
  const int step = gemm_step(K);
  for (int k0 = 0; k0 < K; k0 += step) {
    const int kn = min(step, K - k0);
    double av[Q], bv[Q];
    auto load = [&] {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int gi = i0 + ai(q), k = ak(q);
        av[q] = (gi < M && k < kn) ? la(gi, k0 + k) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int k = bk(q), gj = j0 + bj(q);
        bv[q] = (k < kn && gj < N) ? lb(k0 + k, gj) : 0.0;
      }
    };
    load();
    if (tid < kGBM) sm.ea[tid] = 0;
    else if (tid < kGBM + kGBN) sm.eb[tid - kGBM] = 0;
    __syncthreads();
    // scales: the largest biased exponent of every row of A and column of B
    auto scale = [&](const double (&v)[Q], bool column_per_warp, int* e, auto index) {
      int mx = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int be = gemm_exponent(v[q]);
        if (column_per_warp) {
          const int m = static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<unsigned>(be)));
          if ((tid & 31) == 0) e[index(q)] = m;
        } else {
          mx = max(mx, be);
        }
      }
      if (!column_per_warp) atomicMax(&e[index(0)], mx);
    };
    scale(av, !A_I_CONTIG, sm.ea, ai);
    scale(bv, B_K_CONTIG, sm.eb, bj);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int2 a = gemm_limbs<29>(av[q], sm.ea[ai(q)]), b = gemm_limbs<29>(bv[q], sm.eb[bj(q)]);
      sm.As[ak(q)][ai(q)] = a;
      sm.Bs[bk(q)][bj(q)] = b;
      reinterpret_cast<unsigned char*>(&sm.ma[ak(q) >> 2][ai(q)])[ak(q) & 3] = static_cast<unsigned char>(gemm_byte(a.x));
      reinterpret_cast<unsigned char*>(&sm.mb[bk(q) >> 2][bj(q)])[bk(q) & 3] = static_cast<unsigned char>(gemm_byte(b.x));
    }
    __syncthreads();
    unsigned f64 = 0;  // bit 4 r + c: this output's step is summed in FP64
    {
      unsigned sum[4][4] = {};
#pragma unroll(PER_SM == 1 ? kGBK / 4 : 2)
      for (int w = 0; w < kGBK / 4; ++w) {
        unsigned a[4], b[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) a[r] = sm.ma[w][tr + 16 * r];
#pragma unroll
        for (int c = 0; c < 4; ++c) b[c] = sm.mb[w][tc + 16 * c];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) sum[r][c] = __dp4a(a[r], b[c], sum[r][c]);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          f64 |= static_cast<unsigned>(gemm_in_f64(sum[r][c], sm.ea[tr + 16 * r], sm.eb[tc + 16 * c])) << (4 * r + c);
    }
    long long hh[4][4], mid[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) hh[r][c] = mid[r][c] = 0;
#pragma unroll 2
    for (int kk = 0; kk < kn; ++kk) {
      int2 a[4], b[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = sm.As[kk][tr + 16 * r];
#pragma unroll
      for (int c = 0; c < 4; ++c) b[c] = sm.Bs[kk][tc + 16 * c];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          hh[r][c] += static_cast<long long>(a[r].x) * b[c].x;
          mid[r][c] += static_cast<long long>(a[r].x) * b[c].y;
          mid[r][c] += static_cast<long long>(a[r].y) * b[c].x;
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (!(f64 >> (4 * r + c) & 1u))
          acc[r][c] += gemm_scaled<29>(hh[r][c], mid[r][c], sm.ea[tr + 16 * r] + sm.eb[tc + 16 * c]);
    if (!__syncthreads_or(static_cast<int>(f64))) continue;
    load();
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      *reinterpret_cast<double*>(&sm.As[ak(q)][ai(q)]) = av[q];
      *reinterpret_cast<double*>(&sm.Bs[bk(q)][bj(q)]) = bv[q];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (!(f64 >> (4 * r + c) & 1u)) continue;
#pragma unroll 4
        for (int kk = 0; kk < kn; ++kk)
          acc[r][c] = fma(*reinterpret_cast<const double*>(&sm.As[kk][tr + 16 * r]),
                          *reinterpret_cast<const double*>(&sm.Bs[kk][tc + 16 * c]), acc[r][c]);
      }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = i0 + tr + 16 * r, j = j0 + tc + 16 * c;
      if (i < M && j < N) epi(i, j, acc[r][c]);
    }
}

// ---------------------------------------------------------------------------
// Plane rotation of the cyclic Jacobi method for the symmetric 2 x 2 block
// [[app, apq], [apq, aqq]] (Golub & Van Loan, Matrix Computations, §8.5):
// t = tan(phi) is the root of smaller magnitude of apq t^2 + d t - apq = 0 with
// d = aqq - app (t = sgn(theta) / (|theta| + sqrt(theta^2 + 1)), theta = d / (2 apq)),
// c = 1 / sqrt(1 + t^2), s = t c, and the rotated block is
// diag(app - t apq, aqq + t apq).
//
// GB300 runs FP64 at 1/64 of the FP32 rate and an FP64 divide or square root
// expands into a long sequence on that pipe, so t and c start from FP32 values
// and are finished in FP64 by Newton's method:
//   t: two steps on g(t) = apq t^2 + d t - apq with an FP32 reciprocal of g'(t)
//      (each step multiplies the relative error by about 2^-22);
//   c: two steps of y <- y (3 - x y^2) / 2 on x = 1 + t^2, Newton's iteration
//      for 1/y^2 = x (each step squares the relative error).
// d and apq are first scaled by a power of two (exactly) so that the larger of
// the two lies in [1, 4): the FP32 values neither overflow nor underflow.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void jacobi_rotation(double app, double aqq, double apq, double& t,
                                                double& c, double& s) {
  const double d = aqq - app;
  const double mx = fmax(fabs(d), fabs(apq));
  const int e = static_cast<int>((__double_as_longlong(mx) >> 52) & 0x7ff);
  const double sc = __longlong_as_double(static_cast<long long>(2046 - min(e, 2045)) << 52);
  const double ds = d * sc, as = apq * sc;
  const float df = static_cast<float>(ds), af = static_cast<float>(as);
  float tf;
  if (fabsf(af) * 0x1p40f < fabsf(df)) {
    tf = __fdividef(af, df);  // |theta| > 2^39: t = 1 / (2 theta) to FP32 precision
  } else {
    const float th = __fdividef(df, af + af);
    tf = __fdividef(th >= 0.f ? 1.f : -1.f, fabsf(th) + sqrtf(fmaf(th, th, 1.f)));
  }
  double tt = static_cast<double>(tf);
  const double as2 = as + as;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const double g = fma(fma(as, tt, ds), tt, -as);
    const double r = static_cast<double>(__fdividef(1.f, static_cast<float>(fma(as2, tt, ds))));
    tt = fma(-g, r, tt);
  }
  const double x = fma(tt, tt, 1.0), hx = 0.5 * x;
  double y = static_cast<double>(rsqrtf(static_cast<float>(x)));
#pragma unroll
  for (int it = 0; it < 2; ++it) y = fma(y, fma(-hx * y, y, 0.5), y);
  t = tt;
  c = y;
  s = tt * y;
}

// Rotation test of the cyclic Jacobi method: the pair turns when
// |apq| > tol sqrt(|app aqq|), evaluated as apq^2 > tol^2 |app aqq| (the same
// test without an FP64 square root for entries between 1e-150 and 1e150).
__device__ __forceinline__ bool jacobi_rotates(double app, double aqq, double apq, double tol2) {
  return apq != 0.0 && apq * apq > tol2 * fabs(app * aqq);
}

// The same test with an absolute floor: entries at or below `floor` never turn.
__device__ __forceinline__ bool jacobi_rotates(double app, double aqq, double apq, double tol2, double floor) {
  return fabs(apq) > floor && apq * apq > tol2 * fabs(app * aqq);
}

}  // namespace cmaes_gb300

// kernels_eig_trd.cu -- the tridiagonal route of the eigendecomposition
// C = B D^2 B^T (32 < n <= kEigBigMaxN; the default route).
//
// The paper computes B and D with LAPACK's dsyev (§3.1), i.e. Householder
// reduction to tridiagonal form followed by a tridiagonal eigensolver. On
// GB300 FP64 issues at 1/64 of the FP32 rate, so the route is built for few
// FP64 flops and few sequential steps, all to FP64 accuracy (no refinement needed):
//   1. Householder tridiagonalisation T = Q^T C Q (kernels_eig_trd_reduce.cu).
//   2. Splitting: off-diagonal entries below 4 sqrt(n) eps64 ||T|| are set to
//      zero, which cuts T into independent blocks (this is where the repeated
//      eigenvalues of a low-rank update of a multiple of I separate).
//   3. Eigenvalues of each block by bisection on Sturm counts (one thread per
//      eigenvalue), to an absolute accuracy of 4 eps64 ||T||.
//   4. Eigenvectors of each block by inverse iteration (Gaussian elimination
//      with partial pivoting on T - lambda I, three solves from a
//      pseudo-random start); vectors of one block whose eigenvalues lie within
//      1e-13 ||T|| of each other (where inverse iteration may return nearly
//      parallel vectors) are orthogonalised by Gram-Schmidt (twice; classical
//      on a whole CTA for long chunks, modified on one warp for short ones),
//      in chunks of at most 64 consecutive vectors: a longer chain is a
//      repeated eigenvalue spread by rounding, whose vectors come from
//      independent pseudo-random starts and overlap little across chunks.
//   5. Newton-Schulz steps V <- V + V (I - V^T V) / 2 restore orthogonality
//      to rounding: inverse iteration leaves pairs with small absolute gaps
//      (the small eigenvalues of an ill-conditioned C, the spread-out copies
//      of a repeated eigenvalue) off by about eps64 ||T|| / gap, at most
//      ~1e-3 outside the Gram-Schmidt clusters. V^T V is formed in FP64, the
//      correction (of the size of that defect) in FP32; up to three steps,
//      each after the first only when the previous one started from a defect
//      above 5e-9.
//   6. Back-transformation B = Q V with the stored reflectors, then the
//      canonical form shared with the Jacobi route: columns in ascending
//      eigenvalue order, each column's entry of largest magnitude positive,
//      the PD guard on the eigenvalues.
// Every reduction has a fixed order, so a search gives the same bits alone
// and inside any batch.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <type_traits>
#include "device_common.cuh"
#include "ozaki.cuh"
#include "trd_common.cuh"

namespace cmaes_gb300 {

// --------------------------------------------------------------------------
// Scans of one CTA over n entries (n <= 4096): last index u <= t with
// flag(u) (prefix) or first index u >= t with flag(u) (suffix).
// --------------------------------------------------------------------------
template <int NT, class F>
__device__ void scan_last_start(int n, const F& flag, int* out, int* sh) {
  const int chunk = ceil_div(n, NT), c0 = threadIdx.x * chunk;
  int last = -1;
  for (int u = c0; u < c0 + chunk && u < n; ++u)
    if (flag(u)) last = u;
  sh[threadIdx.x] = last;
  __syncthreads();
  int carry = -1;
  for (int q = 0; q < static_cast<int>(threadIdx.x); ++q) carry = max(carry, sh[q]);
  for (int u = c0; u < c0 + chunk && u < n; ++u) {
    if (flag(u)) carry = u;
    out[u] = carry;
  }
  __syncthreads();
}

template <int NT, class F>
__device__ void scan_first_end(int n, const F& flag, int* out, int* sh) {
  const int chunk = ceil_div(n, NT), c0 = threadIdx.x * chunk;
  int first = 0x7fffffff;
  for (int u = min(c0 + chunk, n) - 1; u >= c0; --u)
    if (flag(u)) first = u;
  sh[threadIdx.x] = first;
  __syncthreads();
  int carry = 0x7fffffff;
  for (int q = NT - 1; q > static_cast<int>(threadIdx.x); --q) carry = min(carry, sh[q]);
  for (int u = min(c0 + chunk, n) - 1; u >= c0; --u) {
    if (flag(u)) carry = u;
    out[u] = carry + 1;  // block end (exclusive)
  }
  __syncthreads();
}

// --------------------------------------------------------------------------
// 2. ||T|| bound, splitting and the blocks of T (one CTA per search).
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(kTrdNT) k_trd_blocks(Search* S, int s0) {
  __shared__ double red[32];
  __shared__ int shi[kTrdNT];
  Search& s = S[s0 + blockIdx.x];
  if (!trd_due(s)) return;
  const int n = s.n;
  double* d = tv(s, TV_D);
  double* e = tv(s, TV_E);
  double* es = tv(s, TV_ES);
  double* e2 = tv(s, TV_E2);
  double* sc = tv(s, TV_SCAL);
  {  // from the reduction's integers: d in q above mu, tau in 2^-61, e in 2^(x - 62) q with x in TV_ES
    const double q = sc[8], mu = sc[9];
    double* tau = tv(s, TV_TAU);
    for (int i = threadIdx.x; i < n; i += kTrdNT) {
      d[i] = fma(static_cast<double>(__double_as_longlong(d[i])), q, mu);
      if (i + 1 < n) {
        e[i] = scalbn(static_cast<double>(__double_as_longlong(e[i])), static_cast<int>(__double_as_longlong(es[i])) - 62) * q;
        tau[i] = static_cast<double>(__double_as_longlong(tau[i])) * 0x1p-61;
      }
    }
    __syncthreads();
  }
  double tn = 0.0, em = 0.0;
  for (int i = threadIdx.x; i < n; i += kTrdNT) {
    const double lo = i > 0 ? fabs(e[i - 1]) : 0.0, hi = i + 1 < n ? fabs(e[i]) : 0.0;
    tn = fmax(tn, fabs(d[i]) + lo + hi);
    em = fmax(em, hi);
  }
  tn = block_max<kTrdNT>(tn, red);
  em = block_max<kTrdNT>(em, red);
  const double split = kTrdSplit * sqrt(static_cast<double>(n)) * kTrdEps * tn;
  for (int i = threadIdx.x; i + 1 < n; i += kTrdNT) es[i] = fabs(e[i]) <= split ? 0.0 : e[i];
  // d (TV_SD) and e^2 (TV_E2) scaled by a power of two (|d| <= 1) for the
  // bisection, and as pairs hi + lo of floats (hi the rounded value, lo the
  // rounded rest): d at TV_P0 (hi, then lo from ldn on), e^2 at TV_P1 likewise
  // (the reduction's buffers are free now)
  const double scl = tn > 0.0 ? exp2(-static_cast<double>(ilogb(tn) + 1)) : 1.0;
  double* sd = tv(s, TV_SD);
  float* d32 = reinterpret_cast<float*>(tv(s, TV_P0));
  float* e32 = reinterpret_cast<float*>(tv(s, TV_P1));
  const long long L2 = s.ldn;
  for (int i = threadIdx.x; i < n; i += kTrdNT) {
    const double ds = d[i] * scl;
    sd[i] = ds;
    d32[i] = static_cast<float>(ds);
    d32[L2 + i] = static_cast<float>(ds - static_cast<double>(d32[i]));
    if (i + 1 < n) {
      const double x = fabs(e[i]) <= split ? 0.0 : e[i] * scl;
      const double x2 = x * x;
      e2[i] = x2;
      e32[i] = static_cast<float>(x2);
      e32[L2 + i] = static_cast<float>(x2 - static_cast<double>(e32[i]));
    }
  }
  if (threadIdx.x == 0) {
    sc[7] = scl;
    sc[0] = tn;
    sc[1] = DBL_MIN * fmax(1.0, em * em);
    sc[2] = split;
    sc[3] = kTrdClus * tn;
    sc[4] = 0.0;  // orthogonality defects before the Newton-Schulz steps
    sc[5] = 0.0;
    sc[6] = 0.0;
  }
  __syncthreads();
  int* b0 = ti(s, TI_B0);
  int* b1 = ti(s, TI_B1);
  scan_last_start<kTrdNT>(n, [&](int u) { return u == 0 || es[u - 1] == 0.0; }, b0, shi);
  scan_first_end<kTrdNT>(n, [&](int u) { return u == n - 1 || es[u] == 0.0; }, b1, shi);
}

// --------------------------------------------------------------------------
// 3. Bisection: a group of LANES lanes finds eigenvalue t - b0 (ascending) of its
// block; each round the lanes take the Sturm counts at the LANES - 1 points (one
// point where a lane is alone) of the next log2(LANES) halvings and then walk those
// halvings on the counts: fewer sequential rounds for more counts in all. A
// precision's points lie on one grid, its last halving's, so the walk meets the same
// points and counts with any number of lanes: the number, which the whole handle
// decides, does not show in the bits.
//
// A Sturm count is the number of sign changes of the leading minors of T - x I,
//   p_j = (d_j - x) p_{j-1} - e_{j-1}^2 p_{j-2},
// rescaled by a power of two every few rows. Per row the dependent chain is one
// FMA (the quotient form p_j / p_{j-1} has a reciprocal on it: FP64 ~600 clocks
// a row against ~75) and the FP64 work three operations against ten. As with
// the quotients, the computed signs are exact for a T whose d_j - x and e_j^2
// are off by a few rounding errors each. A zero p_j takes the sign opposite to
// p_{j-1} (a pivot -0), shrunk far below it.
// --------------------------------------------------------------------------
// Threads per tile of the per-eigenvalue kernels: one warp, so that the warps
// of a single search spread over the SMs and their FP64 pipes.
constexpr int kTrdTT = 32;
int tiles_trd(int n) { return ceil_div(n, kTrdTT); }
int tiles_trd_bis(int n, int lanes) { return ceil_div(n * lanes, kTrdTT); }

// Lanes per eigenvalue (a power of two) by the number of eigenvalues of the handle's
// searches: the rounds' latency against the counts' FP64 work (three operations of ~19
// clocks per warp and row on each SM). The eigenvalue stage with 16 / 8 / 4 / 1 lanes, us:
//   1000 (1 search) 1203 / 1459 / 2020 / 3915, 1800 (2) 1270 / 1332 / 1837 / 3534,
//   2000 (8) 459 / 446 / 581 / 1097, 4000 (4) 2488 / 1873 / 2056 / 3910,
//   5000 (20) 906 / 683 / 649 / 1099, 12000 (12) 5519 / 4023 / 3361 / 3968,
//   14000 (4) 22277 / 15817 / 13249 / 13611, 15000 (15) 6893 / 4864 / 4252 / 4006,
//   38000 (76) 7909 / 5228 / 4088 / 2829.
int trd_bis_lanes(long long eigenvalues) {
  return eigenvalues <= 1900 ? 16 : eigenvalues <= 4500 ? 8 : eigenvalues <= 14000 ? 4 : 1;
}

// Eigenvalues of block [b0, b1) below x; d and e2 the scaled copies (|d| <= 1).
__device__ __forceinline__ int sturm64(const double* __restrict__ d, const double* __restrict__ e2, int b0, int b1,
                                       double x) {
  double p0 = 1.0, p1 = d[b0] - x;
  int cnt = 0;
  auto row = [&](double p, double before) -> double {  // counts the sign change from `before`
    if (((__double2hiint(p) & 0x7fffffff) | __double2loint(p)) == 0)
      p = __hiloint2double((__double2hiint(before) ^ static_cast<int>(0x80000000u)) - (100 << 20), 0);
    cnt += static_cast<int>(static_cast<unsigned>(__double2hiint(p) ^ __double2hiint(before)) >> 31);
    return p;
  };
  p1 = row(p1, p0);
  int j = b0 + 1;
  for (; j + 8 <= b1; j += 8) {
    double dd[8], ee[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      dd[u] = d[j + u];
      ee[u] = e2[j + u - 1];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double p = row(fma(dd[u] - x, p1, -(ee[u] * p0)), p1);
      p0 = p1;
      p1 = p;
    }
    const int ex = max(__double2hiint(p1) & 0x7ff00000, __double2hiint(p0) & 0x7ff00000);
    if (ex < ((1023 - 200) << 20) || ex > ((1023 + 200) << 20)) {
      const double sc = __hiloint2double((2046 << 20) - ex, 0);
      p0 *= sc;
      p1 *= sc;
    }
  }
  for (; j < b1; ++j) {
    const double p = row(fma(d[j] - x, p1, -(e2[j - 1] * p0)), p1);
    p0 = p1;
    p1 = p;
  }
  return cnt;
}

// The power of two that brings the larger of two floats near 1.
__device__ __forceinline__ float rescale32(float a, float b) {
  const int ex = max(__float_as_int(a) & 0x7f800000, __float_as_int(b) & 0x7f800000);
  return __int_as_float((254 << 23) - min(max(ex, 1 << 23), 253 << 23));
}

// The same in FP32.
__device__ __forceinline__ int sturm32(const float* __restrict__ d, const float* __restrict__ e2, int b0, int b1,
                                       float x) {
  float p0 = 1.0f, p1 = d[b0] - x;
  int cnt = 0;
  auto row = [&](float p, float before) -> float {
    if (p == 0.0f) p = before * -0x1p-30f;
    cnt += static_cast<int>(static_cast<unsigned>(__float_as_int(p) ^ __float_as_int(before)) >> 31);
    return p;
  };
  p1 = row(p1, p0);
  int j = b0 + 1;
  for (; j + 4 <= b1; j += 4) {
    float dd[4], ee[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      dd[u] = d[j + u];
      ee[u] = e2[j + u - 1];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float p = row(fmaf(dd[u] - x, p1, -(ee[u] * p0)), p1);
      p0 = p1;
      p1 = p;
    }
    const float sc = rescale32(p0, p1);
    p0 *= sc;
    p1 *= sc;
  }
  for (; j < b1; ++j) {
    const float p = row(fmaf(d[j] - x, p1, -(e2[j - 1] * p0)), p1);
    p0 = p1;
    p1 = p;
  }
  return cnt;
}

// The same in double-float arithmetic (each value a pair hi + lo of floats,
// ~46 significant bits; error-free sums and products from FMA) on the scaled
// pairs: d at dh / dl, e^2 at eh / el, x = xh + xl.
struct Df {
  float h, l;
};
__device__ __forceinline__ void df_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ Df df_sub(Df a, Df b) {
  float s, e;
  df_two_sum(a.h, -b.h, s, e);
  e = __fadd_rn(e, __fsub_rn(a.l, b.l));
  const float h = __fadd_rn(s, e);
  return Df{h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ Df df_mul(Df a, Df b) {
  const float h = __fmul_rn(a.h, b.h);
  return Df{h, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -h)))};
}
__device__ __forceinline__ int sturm_df(const float* __restrict__ dh, const float* __restrict__ dl,
                                        const float* __restrict__ eh, const float* __restrict__ el, int b0, int b1,
                                        float xh, float xl) {
  const Df x{xh, xl};
  Df p0{1.0f, 0.0f}, p1 = df_sub(Df{dh[b0], dl[b0]}, x);
  int cnt = 0;
  auto row = [&](Df p, float before) -> Df {
    if (p.h == 0.0f) p = Df{before * -0x1p-30f, 0.0f};
    cnt += static_cast<int>(static_cast<unsigned>(__float_as_int(p.h) ^ __float_as_int(before)) >> 31);
    return p;
  };
  p1 = row(p1, p0.h);
  int j = b0 + 1;
  for (; j + 4 <= b1; j += 4) {
    Df dd[4], ee[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      dd[u] = Df{dh[j + u], dl[j + u]};
      ee[u] = Df{eh[j + u - 1], el[j + u - 1]};
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const Df p = row(df_sub(df_mul(df_sub(dd[u], x), p1), df_mul(ee[u], p0)), p1.h);
      p0 = p1;
      p1 = p;
    }
    const float sc = rescale32(p0.h, p1.h);
    p0 = Df{p0.h * sc, p0.l * sc};
    p1 = Df{p1.h * sc, p1.l * sc};
  }
  for (; j < b1; ++j) {
    const Df p = row(df_sub(df_mul(df_sub(Df{dh[j], dl[j]}, x), p1), df_mul(Df{eh[j - 1], el[j - 1]}, p0)), p1.h);
    p0 = p1;
    p1 = p;
  }
  return cnt;
}

// Eigenvalue t of its block by bisection in three precisions on the scaled copies: FP32 down to
// a width of 2^-19 ||T||, widened by 2^-18 ||T|| (eight times the backward
// error of an FP32 Sturm count, ~10 eps32 ||T||); double-float down to
// 2^-42 ||T||, widened by 2^-41 ||T|| (several times that of a double-float
// count, ~10 2^-46 ||T||); each widened bracket checked with two counts of
// the next precision (the previous bracket kept if the check fails), the
// last step in FP64 to 4 eps64 ||T||. FP32 and double-float rows cost a warp
// ~4 and ~10 clocks of an SM, an FP64 row 57, so every precision goes as far as
// its counts stay reliable.
template <int LANES>
__global__ void __launch_bounds__(kTrdTT) k_trd_bisect(Search* S, TileMap tm) {
  int tile;
  const int si = find_search(tm, tile);
  const Search& s = S[si];
  if (!trd_due(s)) return;
  const int n = s.n;
  const int q = threadIdx.x % LANES;
  const int t = tile * (kTrdTT / LANES) + threadIdx.x / LANES;
  if (t >= n) return;  // uniform across the lanes of a group
  const int base = (threadIdx.x & 31) & ~(LANES - 1);
  const unsigned gmask = static_cast<unsigned>((1ull << LANES) - 1) << base;
  const double* d = tv(s, TV_SD);
  const double* e2 = tv(s, TV_E2);
  const float* d32 = reinterpret_cast<const float*>(tv(s, TV_P0));
  const float* e32 = reinterpret_cast<const float*>(tv(s, TV_P1));
  const double* sc = tv(s, TV_SCAL);
  double* lamb = tv(s, TV_LAMB);
  const int b0 = ti(s, TI_B0)[t], b1 = ti(s, TI_B1)[t];
  if (b1 - b0 == 1) {
    if (q == 0) lamb[t] = tv(s, TV_D)[t];
    return;
  }
  // the start bracket: [-||T||, ||T||] with ||T|| the largest Gershgorin row
  // sum of the unsplit T (it holds every block's spectrum), widened for rounding
  const double scl = sc[7], tn = sc[0] * scl;  // in [1/2, 1), or 0
  const double atol = 4.0 * kTrdEps * tn;
  const double fudge = 2.0 * kTrdEps * tn * (b1 - b0) + 0x1p-1000;
  double lo = -tn - fudge, hi = tn + fudge;
  const int idx = t - b0;
  // halves [lo_, hi_] to a width of at most tol; cnt(x): the Sturm count at x
  auto halve = [&](auto& lo_, auto& hi_, auto tol, auto cnt) {
    using V = std::remove_reference_t<decltype(lo_)>;
    constexpr int kBits = LANES == 1 ? 1 : LANES == 4 ? 2 : LANES == 8 ? 3 : 4;
    const V width = hi_ - lo_;
    if (!(width > tol) || !(tol > V(0))) return;
    int left = ilogb(width) - ilogb(tol) + 1;  // halvings: at most 54
    if (ldexp(width, 1 - left) <= tol) --left;
    const V w = ldexp(width, -left);  // the grid's spacing
    long long at = 0;                 // the bracket's left end on the grid
    while (left > 0) {
      const int b = min(kBits, left);
      left -= b;
      const long long p = min(q + 1, (1 << b) - 1);
      const int c = cnt(fma(w, static_cast<V>(at + (p << left)), lo_));
      const unsigned le = (__ballot_sync(gmask, c <= idx) & gmask) >> base;
      int pos = 0;
#pragma unroll
      for (int h = kBits - 1; h >= 0; --h)
        if (h < b && (le >> (pos + (1 << h) - 1) & 1u)) pos += 1 << h;
      at += static_cast<long long>(pos) << left;
    }
    hi_ = fma(w, static_cast<V>(at + 1), lo_);
    lo_ = fma(w, static_cast<V>(at), lo_);
  };
  // the two ends of a candidate bracket checked by the counts `cnt` (lane 0
  // the left end, lane 1 the right one; one lane does both)
  auto check = [&](auto cnt, double a, double b) -> bool {
    if (LANES == 1) return cnt(a) <= idx && cnt(b) > idx;
    const int c = cnt(q == 0 ? a : b);
    const bool mine = q == 0 ? c <= idx : q == 1 ? c > idx : true;
    return (__ballot_sync(gmask, !mine) & gmask) == 0;
  };
  if (tn > 0.0) {
    const long long L2 = s.ldn;
    // FP32
    float lo32 = static_cast<float>(lo), hi32 = static_cast<float>(hi);
    halve(lo32, hi32, 0x1p-19f, [&](float x) { return sturm32(d32, e32, b0, b1, x); });
    auto cnt_df = [&](double xs) {
      const float xh = static_cast<float>(xs);
      return sturm_df(d32, d32 + L2, e32, e32 + L2, b0, b1, xh, static_cast<float>(xs - static_cast<double>(xh)));
    };
    double los = lo, his = hi;
    {
      const double a = fmax(los, static_cast<double>(lo32) - 0x1p-18), b = fmin(his, static_cast<double>(hi32) + 0x1p-18);
      if (a < b && check(cnt_df, a, b)) {
        los = a;
        his = b;
      }
    }
    // double-float
    halve(los, his, 0x1p-42, cnt_df);
    const double lo2 = fmax(lo, los - 0x1p-41), hi2 = fmin(hi, his + 0x1p-41);
    if (lo2 < hi2 && check([&](double x) { return sturm64(d, e2, b0, b1, x); }, lo2, hi2)) {
      lo = lo2;
      hi = hi2;
    }
  }
  halve(lo, hi, atol, [&](double x) { return sturm64(d, e2, b0, b1, x); });
  if (q == 0) lamb[t] = 0.5 * (lo + hi) / scl;
}

// --------------------------------------------------------------------------
// 4a. Ranks of the eigenvalues (ascending, ties by block-major index; one thread
// each) and the clusters of close eigenvalues within a block (one CTA per
// search).
// --------------------------------------------------------------------------
constexpr int kTrdSortNT = 1024;

__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}

__global__ void __launch_bounds__(kTrdTT) k_trd_rank(Search* S, TileMap tm) {
  int tile;
  const int si = find_search(tm, tile);
  const Search& s = S[si];
  if (!trd_due(s)) return;
  const int n = s.n, t = tile * kTrdTT + threadIdx.x;
  if (t >= n) return;
  const double* __restrict__ lamb = tv(s, TV_LAMB);
  const double lt = lamb[t];
  const long long kt = order_key(lt);
  int r = 0;
#pragma unroll 8
  for (int u = 0; u < n; ++u) {
    const long long ku = order_key(lamb[u]);
    r += (ku < kt) || (ku == kt && u < t);
  }
  ti(s, TI_RANK)[t] = r;
  tv(s, TV_LAMS)[r] = lt;
}

__global__ void __launch_bounds__(kTrdSortNT) k_trd_clusters(Search* S, int s0) {
  __shared__ int shi[kTrdSortNT];
  Search& s = S[s0 + blockIdx.x];
  if (!trd_due(s)) return;
  const double* lamb = tv(s, TV_LAMB);
  const int* b0 = ti(s, TI_B0);
  const double ctol = tv(s, TV_SCAL)[3];
  scan_last_start<kTrdSortNT>(
      s.n, [&](int u) { return u == b0[u] || !(lamb[u] - lamb[u - 1] <= ctol); }, ti(s, TI_CL0), shi);
}

// --------------------------------------------------------------------------
// 4b. Inverse iteration (thread t, eigenvalue lamb[t] of its block): three
// solves of (T - lambda I) x = x_prev with one Gaussian elimination with
// partial pivoting (its factors in scratch interleaved by thread), the
// iterate in column t of ET.
// --------------------------------------------------------------------------
__device__ __forceinline__ double start_value(int t, int j) {
  uint32_t h = static_cast<uint32_t>(t) * 0x9E3779B1u ^ (static_cast<uint32_t>(j) * 0x85EBCA77u);
  h ^= h >> 15;
  h *= 0x2C1B3C6Du;
  h ^= h >> 12;
  h *= 0x297A2D39u;
  h ^= h >> 15;
  return (static_cast<double>(h) + 0.5) * 0x1p-31 - 1.0;  // in (-1, 1)
}

constexpr long long kInvitSwap = 0x7ff8000000000000LL;  // a quiet NaN: the row-interchange flag
constexpr int kInvitU = 16;                              // rows whose loads are in flight together

// 1 / m: an FP32 seed of the mantissa, built and read back on the integer pipe,
// and one third-order Newton step (FP64 divides take ~560 clocks, this ~280);
// the division itself near the ends of the exponent range.
__device__ __forceinline__ double reciprocal(double m) {
  const int h = __double2hiint(m), ex = (h >> 20) & 0x7ff;
  if (ex < 8 || ex > 2038) return 1.0 / m;
  const float f = __int_as_float(0x3f800000 | ((h & 0xfffff) << 3) |
                                 static_cast<int>(static_cast<unsigned>(__double2loint(m)) >> 29));
  const int b = __float_as_int(__fdividef(1.0f, f));  // in (1/2, 1]
  double r = __hiloint2double(((b >> 3) + ((1023 - 127 + 1023 - ex) << 20)) | (h & static_cast<int>(0x80000000u)), b << 29);
  const double g = fma(-m, r, 1.0);
  r = fma(r, fma(g, g, g), r);
  return r;
}

// The rows are a chain (factorisation ~6 dependent FP64 operations, forward 1,
// back 2), so what is not on it is kept off it: the loads of kInvitU rows are
// issued together before their chain (one load a row behind each step of it was
// most of the time), and an iterate is scaled while the next solve reads it.
__global__ void __launch_bounds__(kTrdTT) k_trd_invit(Search* S, TileMap tm) {
  int tile;
  const int si = find_search(tm, tile);
  const Search& s = S[si];
  if (!trd_due(s)) return;
  const int n = s.n, t = tile * kTrdTT + threadIdx.x;
  if (t >= n) return;
  const long long L = s.ldn, nn = n;
  const double* __restrict__ d = tv(s, TV_D);
  const double* __restrict__ es = tv(s, TV_ES);
  const double lam = tv(s, TV_LAMB)[t];
  const double tiny = kTrdEps * tv(s, TV_SCAL)[0];
  const int b0 = ti(s, TI_B0)[t], b1 = ti(s, TI_B1)[t];
  double* v_out = s.ET + L * t;
  for (int i = 0; i < b0; ++i) v_out[i] = 0.0;
  for (int i = b1; i < n; ++i) v_out[i] = 0.0;
  if (b1 - b0 == 1) {
    v_out[t] = 1.0;
    return;
  }
  // the iterate and the factors interleaved by thread, so that a warp's access
  // to a row is one line (B is free until the back-transformation writes it)
  double* x = s.B + t;
  double* u0 = s.EA + t;
  double* u1 = s.EG + t;
  double* u2 = s.EH + t;
  // |a| as an ordered integer: comparing those keeps FP64 compares (~104 clocks) off the chain
  auto magnitude = [](double a) { return __double_as_longlong(a) & 0x7fffffffffffffffLL; };
  auto piv_of = [&](double a) { return magnitude(a) > magnitude(tiny) ? a : copysign(tiny, a); };
  // factorisation of T - lambda I, once for the three solves: row j keeps its
  // multiplier (u2), the reciprocal of its pivot (u0), and its superdiagonal or,
  // for an interchanged row, the flag kInvitSwap (u1; the rest of its U row,
  // d_{j+1} - lambda and e_{j+1}, is read from T again)
  double a = d[b0] - lam, b = es[b0];
  auto factor = [&](auto rows_c, int j0) {
    constexpr int R = decltype(rows_c)::value;
    double sub[R + 1], nd[R];
#pragma unroll
    for (int u = 0; u < R; ++u) {
      sub[u] = es[j0 + u];
      nd[u] = d[j0 + u + 1] - lam;
    }
    sub[R] = j0 + R + 1 < b1 ? es[j0 + R] : 0.0;
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const bool swap = magnitude(a) < magnitude(sub[u]);
      const double r = reciprocal(swap ? sub[u] : piv_of(a));
      const double l = (swap ? a : sub[u]) * r;
      const long long o = (j0 + u) * nn;
      u0[o] = r;
      u1[o] = swap ? __longlong_as_double(kInvitSwap) : b;
      u2[o] = l;
      a = swap ? fma(-l, nd[u], b) : fma(-l, b, nd[u]);
      b = swap ? -l * sub[u + 1] : sub[u + 1];
    }
  };
  double inv = 1.0, y = 0.0, xn1 = 0.0, xn2 = 0.0, ss = 0.0;
  int it = 0;
  // forward: the same row interchanges and multipliers on the iterate
  auto forward = [&](auto rows_c, int j0) {
    constexpr int R = decltype(rows_c)::value;
    double l[R], f[R], xr[R];
#pragma unroll
    for (int u = 0; u < R; ++u) {
      l[u] = u2[(j0 + u) * nn];
      f[u] = u1[(j0 + u) * nn];
      xr[u] = it == 0 ? start_value(t, j0 + u + 1) : x[(j0 + u + 1) * nn];
    }
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const bool swap = __double_as_longlong(f[u]) == kInvitSwap;
      const double xs = xr[u] * inv;
      x[(j0 + u) * nn] = swap ? xs : y;
      y = fma(-l[u], swap ? xs : y, swap ? y : xs);
    }
  };
  auto back = [&](auto rows_c, int j1) {  // rows j1, j1 - 1, ...
    constexpr int R = decltype(rows_c)::value;
    double r[R], c1[R], c2[R], xr[R];
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const int j = j1 - u;
      r[u] = u0[j * nn];
      c1[u] = u1[j * nn];
      xr[u] = x[j * nn];
      c2[u] = j + 2 < b1 ? es[j + 1] : 0.0;
      const double nd = d[j + 1] - lam;
      const bool swap = __double_as_longlong(c1[u]) == kInvitSwap;
      c1[u] = swap ? nd : c1[u];
      c2[u] = swap ? c2[u] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const double v = fma(-c1[u], xn1, fma(-c2[u], xn2, xr[u])) * r[u];
      x[(j1 - u) * nn] = v;
      xn2 = xn1;
      xn1 = v;
      ss = fma(v, v, ss);
    }
  };
  using Many = std::integral_constant<int, kInvitU>;
  using One = std::integral_constant<int, 1>;
  {
    int j = b0;
    for (; j + kInvitU < b1; j += kInvitU) factor(Many{}, j);
    for (; j + 1 < b1; ++j) factor(One{}, j);
  }
  const double rlast = reciprocal(piv_of(a));
  for (; it < 3; ++it) {
    y = it == 0 ? start_value(t, b0) : x[b0 * nn] * inv;
    int j = b0;
    for (; j + kInvitU < b1; j += kInvitU) forward(Many{}, j);
    for (; j + 1 < b1; ++j) forward(One{}, j);
    xn1 = y * rlast;
    xn2 = 0.0;
    x[(b1 - 1) * nn] = xn1;
    ss = xn1 * xn1;
    for (j = b1 - 2; j - kInvitU + 1 >= b0; j -= kInvitU) back(Many{}, j);
    for (; j >= b0; --j) back(One{}, j);
    inv = 1.0 / sqrt(ss);
  }
  auto scale = [&](auto rows_c, int j0) {
    constexpr int R = decltype(rows_c)::value;
    double xr[R];
#pragma unroll
    for (int u = 0; u < R; ++u) xr[u] = x[(j0 + u) * nn];
#pragma unroll
    for (int u = 0; u < R; ++u) v_out[j0 + u] = xr[u] * inv;
  };
  int j = b0;
  for (; j + kInvitU <= b1; j += kInvitU) scale(Many{}, j);
  for (; j < b1; ++j) scale(One{}, j);
}

// --------------------------------------------------------------------------
// 4c. Gram-Schmidt (twice) inside each cluster of close eigenvalues of one
// block, in chunks of at most kTrdClusMax consecutive vectors (independent of
// one another). A long chunk on a long block goes to a whole CTA as classical
// Gram-Schmidt applied twice (all projections of a vector at once: the dots
// spread over the warps, the update over the rows, the vector in shared
// memory); a short one to one warp as modified Gram-Schmidt, twice. Both keep
// the orthogonality that the later Newton-Schulz steps need (Giraud, Langou &
// Rozloznik 2005: two passes of either are enough for vectors that are not
// numerically dependent).
// --------------------------------------------------------------------------
// Modified Gram-Schmidt, twice, on vectors [c, ce) of rows [r0, r1) (one warp).
__device__ void cluster_mgs(double* V, long long L, int c, int ce, int r0, int r1, int lane) {
  double* vc = V + L * c;
  {
    double q = 0.0;
    for (int i = r0 + lane; i < r1; i += 32) q = fma(vc[i], vc[i], q);
    const double inv = 1.0 / sqrt(warp_sum_xor(q));
    for (int i = r0 + lane; i < r1; i += 32) vc[i] *= inv;
    __syncwarp();
  }
  for (int a = c + 1; a < ce; ++a) {
    double* va = V + L * a;
    for (int rep = 0; rep < 2; ++rep)
      for (int b = c; b < a; ++b) {
        const double* vb = V + L * b;
        double p = 0.0;
        for (int i = r0 + lane; i < r1; i += 32) p = fma(vb[i], va[i], p);
        p = warp_sum_xor(p);
        for (int i = r0 + lane; i < r1; i += 32) va[i] = fma(-p, vb[i], va[i]);
        __syncwarp();
      }
    double q = 0.0;
    for (int i = r0 + lane; i < r1; i += 32) q = fma(va[i], va[i], q);
    const double inv = 1.0 / sqrt(warp_sum_xor(q));
    for (int i = r0 + lane; i < r1; i += 32) va[i] *= inv;
    __syncwarp();
  }
}

// Classical Gram-Schmidt, twice, on vectors [c, ce) of rows [r0, r1) (the
// whole CTA; r1 - r0 <= kEigBigMaxN). Per vector a and pass: p = V_prev^T v_a
// (warp w takes the previous vectors w, w + 8, ...), then v_a -= V_prev p on
// every row (the terms in ascending order); then v_a / |v_a|.
__device__ void cluster_cgs2_cta(double* V, long long L, int c, int ce, int r0, int r1, double* va,
                                 double* pb, double* red) {
  constexpr int NW = kTrdNT / 32;
  const int R = r1 - r0, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int a = c; a < ce; ++a) {
    double* col = V + L * a + r0;
    for (int i = tid; i < R; i += kTrdNT) va[i] = col[i];
    __syncthreads();
    const int m = a - c;
    for (int rep = 0; rep < (m > 0 ? 2 : 0); ++rep) {
      for (int x = warp; x < m; x += NW) {
        const double* vb = V + L * (c + x) + r0;
        double p0 = 0.0, p1 = 0.0, p2 = 0.0, p3 = 0.0;
        int i = lane;
        for (; i + 96 < R; i += 128) {  // four rows per lane in flight
          p0 = fma(vb[i], va[i], p0);
          p1 = fma(vb[i + 32], va[i + 32], p1);
          p2 = fma(vb[i + 64], va[i + 64], p2);
          p3 = fma(vb[i + 96], va[i + 96], p3);
        }
        for (; i < R; i += 32) p0 = fma(vb[i], va[i], p0);
        const double p = warp_sum_xor((p0 + p1) + (p2 + p3));
        if (lane == 0) pb[x] = p;
      }
      __syncthreads();
      for (int i = tid; i < R; i += kTrdNT) {
        const double* vb = V + L * c + r0 + i;
        double acc = va[i];
        int x = 0;
        for (; x + 4 <= m; x += 4) {
          const double b0 = vb[L * x], b1 = vb[L * (x + 1)], b2 = vb[L * (x + 2)], b3 = vb[L * (x + 3)];
          acc = fma(-pb[x], b0, acc);
          acc = fma(-pb[x + 1], b1, acc);
          acc = fma(-pb[x + 2], b2, acc);
          acc = fma(-pb[x + 3], b3, acc);
        }
        for (; x < m; ++x) acc = fma(-pb[x], vb[L * x], acc);
        va[i] = acc;
      }
      __syncthreads();
    }
    double q = 0.0;
    for (int i = tid; i < R; i += kTrdNT) q = fma(va[i], va[i], q);
    q = warp_sum_xor(q);
    if (lane == 0) red[warp] = q;
    __syncthreads();
    double nq = 0.0;
    for (int w = 0; w < NW; ++w) nq += red[w];
    const double inv = 1.0 / sqrt(nq);
    for (int i = tid; i < R; i += kTrdNT) col[i] = va[i] * inv;
    __syncthreads();  // v_a complete before the next vector reads it (and red is reused)
  }
}

constexpr int kTrdMgsCtas = 32;    // CTAs per search of the Gram-Schmidt kernel
constexpr int kTrdCgsMinVec = 8;   // chunks of at least this many vectors
constexpr int kTrdCgsMinRows = 256;  // on blocks of at least this many rows go to a CTA

__global__ void __launch_bounds__(kTrdNT) k_trd_mgs(Search* S, int s0) {
  __shared__ double va[kEigBigMaxN];
  __shared__ double pb[kTrdClusMax];
  __shared__ double red[kTrdNT / 32];
  Search& s = S[s0 + blockIdx.x];
  if (!trd_due(s)) return;
  const int n = s.n, lane = threadIdx.x & 31;
  const int warp = blockIdx.y * (kTrdNT / 32) + (threadIdx.x >> 5);  // of the search's warps
  const long long L = s.ldn;
  const int* cl0 = ti(s, TI_CL0);
  const int* b0a = ti(s, TI_B0);
  const int* b1a = ti(s, TI_B1);
  double* V = s.ET;
  // work items: the chunks of every cluster of two or more; the long ones
  // dealt round-robin to the CTAs (pass 0), the others to the warps (pass 1)
  for (int pass = 0; pass < 2; ++pass) {
    int found = 0;
    for (int c = 0; c < n; ++c) {
      if (cl0[c] != c || c + 1 >= n || cl0[c + 1] != c) continue;
      int ce = c + 1;
      while (ce < n && cl0[ce] == c) ++ce;
      const int r0 = b0a[c], r1 = b1a[c];
      for (int cc = c; cc < ce; cc += kTrdClusMax) {
        const int cn = min(ce, cc + kTrdClusMax);
        const bool big = cn - cc >= kTrdCgsMinVec && r1 - r0 >= kTrdCgsMinRows;
        if (big != (pass == 0)) continue;
        if (big) {
          if ((found++ % kTrdMgsCtas) == static_cast<int>(blockIdx.y))
            cluster_cgs2_cta(V, L, cc, cn, r0, r1, va, pb, red);
        } else if ((found++ % (kTrdMgsCtas * kTrdNT / 32)) == warp) {
          cluster_mgs(V, L, cc, cn, r0, r1, lane);
        }
      }
    }
  }
}

// --------------------------------------------------------------------------
// 5. Newton-Schulz: M = (I - V^T V) / 2 in FP32 from an FP64-accurate
// product on the tensor cores (64 x 64 tiles, mirrored; tiles outside the
// eigenvalue band are zero and flagged so), then V' = V + V M with FP32
// products over the nonzero tiles.
// --------------------------------------------------------------------------
int tiles_trd_sq(int n) { const int T = ceil_div(n, kGBM); return T * T; }

int tiles_trd_ozp(int n) { return oz_rows_padded(n) / 64; }
int tiles_trd_ozg(int n) { return ceil_div(n, kOzBM) * ceil_div(n, kOzBN); }
size_t trd_oz_bytes(int n) { return trd_oz_layout(n).total; }
int trd_oz_exps(int n) { return trd_oz_layout(n).etotal; }

__device__ __forceinline__ bool trd_ns_skipped(const Search& s, int pass) {
  return pass > 0 && __ldcg(&tv(s, TV_SCAL)[3 + pass]) <= kTrdNsSkip;  // the previous step was enough
}

// The columns of this pass's V as the rows of a packed operand (K = n).
__global__ void __launch_bounds__(kOzNT) k_trd_oz_pack(Search* S, TileMap tm, int pass) {
  __shared__ int sh_e[64];
  int tile;
  const int si = find_search(tm, tile);
  const Search& s = S[si];
  if (!trd_due(s) || trd_ns_skipped(s, pass)) return;
  const double* V = (pass & 1) ? s.EA : s.ET;
  oz_pack_block(V, s.ldn, 1, s.n, s.n, tile, oz_nks(s.n), s.ozp, s.oze, sh_e);
}

// M = (I - V^T V) / 2 over the 64 x 64 tiles (fi, fj), fi <= fj, that hold a
// pair of one block with eigenvalues within kTrdNsBand ||T|| (mirrored,
// flagged; zero and unflagged elsewhere), from the FP64-accurate tensor-core
// product: CTA (bi, bj) owns the 128 x 64 tile of rows 128 bi.., columns
// 64 bj.., i.e. the 64 x 64 tiles (2 bi, bj) and (2 bi + 1, bj), and writes
// the elements i <= j of those it owns.
__global__ void __launch_bounds__(kOzNT, 1) k_trd_oz_gram(Search* S, TileMap tm, int pass) {
  extern __shared__ unsigned char dyn[];
  __shared__ uint64_t bar[5];
  __shared__ uint32_t tslot;
  __shared__ double trange[3][2];
  __shared__ int brange[3][2];
  int tile;
  const int si = find_search(tm, tile);
  const Search& s = S[si];
  if (!trd_due(s) || trd_ns_skipped(s, pass)) return;
  const int n = s.n, T = ceil_div(n, kGBM), TN = ceil_div(n, kOzBN);
  const int bi = tile / TN, bj = tile % TN;
  if (bj * kOzBN + kOzBN - 1 < bi * kOzBM) return;  // wholly below the diagonal
  const long long L = s.ldn;
  float* M = reinterpret_cast<float*>(s.EG);
  int* flags = ti(s, TI_TFLAG);
  double* sc = tv(s, TV_SCAL);
  // eigenvalue and block ranges of the column blocks 2 bi, 2 bi + 1 and bj
  if (threadIdx.x < 96) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int c0 = (w == 0 ? 2 * bi : (w == 1 ? 2 * bi + 1 : bj)) * kGBM;
    double lo = INFINITY, hi = -INFINITY;
    int blo = 0x7fffffff, bhi = -1;
    for (int u = l; u < kGBM; u += 32) {
      const int t = c0 + u;
      if (t < n) {
        const double lam = tv(s, TV_LAMB)[t];
        const int b = ti(s, TI_B0)[t];
        lo = fmin(lo, lam);
        hi = fmax(hi, lam);
        blo = min(blo, b);
        bhi = max(bhi, b);
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      blo = min(blo, __shfl_xor_sync(0xffffffffu, blo, o));
      bhi = max(bhi, __shfl_xor_sync(0xffffffffu, bhi, o));
    }
    if (l == 0) {
      trange[w][0] = lo;
      trange[w][1] = hi;
      brange[w][0] = blo;
      brange[w][1] = bhi;
    }
  }
  __syncthreads();
  bool owned[2], needed[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int fi = 2 * bi + h;
    owned[h] = fi <= bj && fi < T;
    const bool share = brange[h][0] <= brange[2][1] && brange[2][0] <= brange[h][1];
    const double dist = fmax(0.0, fmax(trange[2][0] - trange[h][1], trange[h][0] - trange[2][1]));
    needed[h] = owned[h] && share && !(dist > kTrdNsBand * sc[0]);
    if (owned[h] && threadIdx.x == 0) {
      flags[fi + T * bj] = needed[h];
      flags[bj + T * fi] = needed[h];
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = bi * kOzBM + 32 * (warp & 3) + lane;
  const int h = (warp & 3) >> 1;
  const int jb = bj * kOzBN + 32 * (warp >> 2);
  if (!needed[0] && !needed[1]) {  // M = 0 on the owned tiles and their mirrors
    if (owned[h] && i < n)
      for (int q = 0; q < 32; ++q) {
        const int j = jb + q;
        if (j < n && i <= j) {
          M[i + L * j] = 0.f;
          M[j + L * i] = 0.f;
        }
      }
    return;
  }
  OzCtx cx;
  oz_begin(cx, dyn, bar, &tslot);
  long long Wq[32];
  float Lq[32];
  const long long pitch = oz_pitch(oz_nks(n));
  const bool ok = oz_tile(cx, s.ozp, pitch, 2 * bi, s.ozp, pitch, bj, oz_nks(n), Wq, Lq);
  double dmax = 0.0;
  if (ok && owned[h] && i < n) {
    const int ei = s.oze[i];
#pragma unroll
    for (int q = 0; q < 32; ++q) {
      const int j = jb + q;
      if (j < n && i <= j) {
        double m = 0.0;
        if (needed[h]) {
          const int ej = s.oze[j];
          const double g = oz_value(Wq[q], Lq[q], ei, ej);
          m = 0.5 * ((i == j ? 1.0 : 0.0) - g);
          dmax = fmax(dmax, fabs(m));
        }
        M[i + L * j] = static_cast<float>(m);
        M[j + L * i] = static_cast<float>(m);
      }
    }
  }
  // the defect of this pass (non-negative doubles order like their bit
  // patterns); every lane of every warp takes part in the reduction
  for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
  if (lane == 0 && dmax > 0.0)
    atomicMax(reinterpret_cast<unsigned long long*>(&sc[4 + pass]),
              static_cast<unsigned long long>(__double_as_longlong(dmax)));
  if (!ok && threadIdx.x == 0) atomicOr(s.err, kDevErrTimeout);
  oz_end(cx);
}

struct GemmSmem32 {
  float As[kGBK][kGBM];
  float Bs[kGBK][kGBN];
};

// Step `pass` (0, 1, 2) maps ET -> EA, EA -> ET, ET -> EA: V' = V + V M, or a
// copy when the previous step started from a defect small enough (then no M
// was formed); the result is in EA after the three.
// V' = V + V M on one 64 x 64 tile of V': 256 threads, each a 4 x 4 block of
// consecutive rows and columns (float4 reads of the staged operands), k in
// steps of 32 over the k tiles whose 64 x 64 block of M is flagged nonzero,
// the next step's operands loaded into registers while the current one is
// multiplied (two shared-memory buffers, one barrier per step). The products
// are summed in ascending k, one FP32 FMA each.
constexpr int kNsBK = 32;

__global__ void __launch_bounds__(kGNT) k_trd_ns(Search* S, TileMap tm, int pass) {
  __shared__ __align__(16) float As[2][kNsBK][kGBM];      // V block, [k][i]
  __shared__ __align__(16) float Bs[2][kNsBK][kGBN + 4];  // M block, [k][j] (rows 16-byte aligned)
  int tile;
  const int si = find_search(tm, tile);
  const Search& s = S[si];
  if (!trd_due(s)) return;
  const int n = s.n, T = ceil_div(n, kGBM);
  const int i0 = (tile % T) * kGBM, j0 = (tile / T) * kGBN;
  const long long L = s.ldn;
  const double* V = (pass & 1) ? s.EA : s.ET;
  double* Vo = (pass & 1) ? s.ET : s.EA;
  const int tid = threadIdx.x, tr = tid & 15, tc = tid >> 4;
  if (pass > 0 && __ldcg(&tv(s, TV_SCAL)[3 + pass]) <= kTrdNsSkip) {
    for (int e = tid; e < kGBM * kGBN; e += kGNT) {
      const int i = i0 + (e & (kGBM - 1)), j = j0 + e / kGBM;
      if (i < n && j < n) Vo[i + L * j] = V[i + L * j];
    }
    return;
  }
  const float* M = reinterpret_cast<const float*>(s.EG);
  const int* flags = ti(s, TI_TFLAG);
  const int nkt = ceil_div(n, kNsBK);
  auto next_kt = [&](int kt) {  // the first k step at or after kt on a flagged block of M
    while (kt < nkt && !__ldcg(&flags[(kt * kNsBK) / kGBM + T * (j0 / kGBN)])) ++kt;
    return kt;
  };
  float ra[8], rb[8];
  auto load = [&](int kt) {
    const int k0 = kt * kNsBK;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = tid + q * kGNT;
      const int ii = e & (kGBM - 1), kk = e >> 6;  // V: consecutive threads, consecutive rows
      const int gi = i0 + ii, gk = k0 + kk;
      ra[q] = (gi < n && gk < n) ? static_cast<float>(V[gi + L * gk]) : 0.f;
      const int kk2 = e & (kNsBK - 1), jj = e >> 5;  // M: consecutive threads, consecutive k
      const int gk2 = k0 + kk2, gj = j0 + jj;
      rb[q] = (gk2 < n && gj < n) ? M[gk2 + L * gj] : 0.f;
    }
  };
  auto store = [&](int b) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = tid + q * kGNT;
      As[b][e >> 6][e & (kGBM - 1)] = ra[q];
      Bs[b][e & (kNsBK - 1)][e >> 5] = rb[q];
    }
  };
  float acc[4][4] = {};
  int kt = next_kt(0);
  if (kt < nkt) {
    load(kt);
    store(0);
  }
  __syncthreads();
  int b = 0;
  while (kt < nkt) {
    const int kn = next_kt(kt + 1);
    if (kn < nkt) load(kn);
#pragma unroll 8
    for (int kk = 0; kk < kNsBK; ++kk) {
      const float4 a4 = *reinterpret_cast<const float4*>(&As[b][kk][4 * tr]);
      const float4 b4 = *reinterpret_cast<const float4*>(&Bs[b][kk][4 * tc]);
      const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(av[r], bv[c], acc[r][c]);
    }
    if (kn < nkt) store(b ^ 1);
    __syncthreads();
    b ^= 1;
    kt = kn;
  }
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = i0 + 4 * tr + r, j = j0 + 4 * tc + c;
      if (i < n && j < n) Vo[i + L * j] = V[i + L * j] + static_cast<double>(acc[r][c]);
    }
}

// --------------------------------------------------------------------------
// 6. Back-transformation B = Q V' of the smaller sizes (reflectors applied in
// reverse order, one warp per column), canonical sign, and the column order of
// ascending eigenvalues; kernels_eig_trd_bt.cu takes n >= kBtBlockedMinN.
// --------------------------------------------------------------------------
__host__ __device__ inline int trd_bt_cols(int n) { return 8; }
int tiles_trd_bt(int n) { return trd_bt_blocked(n) ? 0 : ceil_div(n, trd_bt_cols(n)); }

// Each column held in registers (element lane + 32 r in x[r]; n <= 32 RMAX):
// the column never moves; each reflector is staged once
// per CTA in shared memory (double-buffered: the next one is loaded while the
// current one is applied) and rows at or above its first row are skipped 256
// at a time.
template <int RMAX>
__global__ void __launch_bounds__(kTrdNT) k_trd_backtf_reg(Search* S, TileMap tm) {
  __shared__ double vs[2][32 * RMAX];
  int tile;
  const int si = find_search(tm, tile);
  Search& s = S[si];
  if (!trd_due(s)) return;
  const int n = s.n;
  if (n > 32 * RMAX || trd_bt_blocked(n)) return;  // the blocked form takes these sizes
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t = tile * trd_bt_cols(n) + warp;
  const bool active = warp < trd_bt_cols(n) && t < n;  // idle warps still join the barriers
  const long long L = s.ldn;
  const double* Vs = s.EA + L * (active ? t : 0);
  double x[RMAX];
#pragma unroll
  for (int r = 0; r < RMAX; ++r) {
    const int i = lane + 32 * r;
    x[r] = (active && i < n) ? Vs[i] : 0.0;
  }
  const double* tau = tv(s, TV_TAU);
  const double* Hv = s.EX;
  constexpr int CH = 8;  // registers per chunk: 256 rows
  // stage reflector k - 1 while k is applied
  int cur = 0;
  if (n >= 2) {
    const double* v0 = Hv + L * (n - 2);
    for (int i = threadIdx.x; i < n; i += kTrdNT) vs[0][i] = i > n - 2 ? v0[i] : 0.0;
  }
  __syncthreads();
  for (int k = n - 2; k >= 0; --k) {
    // prefetch the next reflector into registers (stored after this one is applied)
    double pre[(32 * RMAX + kTrdNT - 1) / kTrdNT];
    if (k > 0) {
      const double* vn = Hv + L * (k - 1);
#pragma unroll
      for (int u = 0; u < (32 * RMAX + kTrdNT - 1) / kTrdNT; ++u) {
        const int i = threadIdx.x + kTrdNT * u;
        pre[u] = (i < n && i > k - 1) ? vn[i] : 0.0;
      }
    }
    const double tk = tau[k];
    const double* v = vs[cur];
    if (active && tk != 0.0) {
      double p0 = 0.0, p1 = 0.0;
#pragma unroll
      for (int c = 0; c < RMAX / CH; ++c) {
        if (256 * c + 255 <= k || 256 * c >= n) continue;
#pragma unroll
        for (int rr = 0; rr < CH; rr += 2) {
          const int i0 = lane + 32 * (CH * c + rr), i1 = i0 + 32;
          if (i0 > k && i0 < n) p0 = fma(v[i0], x[CH * c + rr], p0);
          if (i1 > k && i1 < n) p1 = fma(v[i1], x[CH * c + rr + 1], p1);
        }
      }
      const double p = tk * warp_sum_xor(p0 + p1);
#pragma unroll
      for (int c = 0; c < RMAX / CH; ++c) {
        if (256 * c + 255 <= k || 256 * c >= n) continue;
#pragma unroll
        for (int rr = 0; rr < CH; ++rr) {
          const int i = lane + 32 * (CH * c + rr);
          if (i > k && i < n) x[CH * c + rr] = fma(-p, v[i], x[CH * c + rr]);
        }
      }
    }
    if (k > 0) {
#pragma unroll
      for (int u = 0; u < (32 * RMAX + kTrdNT - 1) / kTrdNT; ++u) {
        const int i = threadIdx.x + kTrdNT * u;
        if (i < 32 * RMAX) vs[cur ^ 1][i] = pre[u];
      }
    }
    __syncthreads();
    cur ^= 1;
  }
  if (!active) return;
  // sign: the entry of largest magnitude (the first on ties) positive
  double best = -1.0, val = 0.0;
  int bi = 0x7fffffff;
#pragma unroll
  for (int r = 0; r < RMAX; ++r) {
    const int i = lane + 32 * r;
    const double a = fabs(x[r]);
    if (i < n && a > best) {
      best = a;
      val = x[r];
      bi = i;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const double ov = __shfl_xor_sync(0xffffffffu, val, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ob > best || (ob == best && oi < bi)) {
      best = ob;
      val = ov;
      bi = oi;
    }
  }
  const double sg = val < 0.0 ? -1.0 : 1.0;
  double* Bc = s.B + L * ti(s, TI_RANK)[t];
#pragma unroll
  for (int r = 0; r < RMAX; ++r) {
    const int i = lane + 32 * r;
    if (i < n) Bc[i] = sg * x[r];
  }
}

// --------------------------------------------------------------------------
// Eigenvalues with the PD guard (as in the Jacobi route), D, the work counter.
// --------------------------------------------------------------------------
constexpr double kTrdPdFloor = 1e-16;

__global__ void __launch_bounds__(kTrdNT) k_trd_finish(Search* S, int s0) {
  Search& s = S[s0 + blockIdx.x];
  if (!trd_due(s)) return;
  const int n = s.n;
  const long long L = s.ldn;
  const double* lams = tv(s, TV_LAMS);
  const double lo = lams[0], hi = lams[n - 1];
  const double add = (lo < hi * kTrdPdFloor) ? hi * kTrdPdFloor - lo : 0.0;
  for (int i = threadIdx.x; i < n; i += kTrdNT) {
    s.D[i] = sqrt(lams[i] + add);
    if (add != 0.0) s.C[i + L * i] += add;
  }
  if (threadIdx.x == 0) {
    s.eig_sweeps = 0;
    s.eig_count += 1;
  }
}

// --------------------------------------------------------------------------
// Host side
// --------------------------------------------------------------------------
void trd_set_attributes() {
  cudaFuncSetAttribute(k_trd_oz_gram, cudaFuncAttributeMaxDynamicSharedMemorySize, kOzSmem);
  bt_set_attributes();
}

// marks (optional, kTrdStages + 1 events): recorded before the reduction and
// after each stage (reduction, eigenvalues, inverse iteration, Gram-Schmidt in
// clusters, orthogonalisation, back-transformation), for the per-stage times
// of the profiling mode.
int launch_eig_trd(Search* S, const int4* grp, const TrdChunk* chunks, int nchunks, unsigned* bars, int s0, int s1,
                   const TrdReducePlan& plan, const TrdMaps& tm, int max_n, int bis_lanes, cudaStream_t st,
                   cudaEvent_t* marks) {
  if (nchunks <= 0 || s1 <= s0) return 0;
  int nl = 0;
  auto mark = [&](int k) {
    if (marks) cudaEventRecord(marks[k], st);
  };
  mark(0);
  nl += launch_trd_reduce(S, grp, chunks, nchunks, bars, s0, s1, plan, st);
  mark(1);
  k_trd_blocks<<<s1 - s0, kTrdNT, 0, st>>>(S, s0);
  const auto bisect = bis_lanes == 16 ? k_trd_bisect<16> : bis_lanes == 8 ? k_trd_bisect<8>
                      : bis_lanes == 4 ? k_trd_bisect<4> : k_trd_bisect<1>;
  bisect<<<tm.tbis.total, kTrdTT, 0, st>>>(S, tm.tbis);
  k_trd_rank<<<tm.tt.total, kTrdTT, 0, st>>>(S, tm.tt);
  k_trd_clusters<<<s1 - s0, kTrdSortNT, 0, st>>>(S, s0);
  mark(2);
  k_trd_invit<<<tm.tt.total, kTrdTT, 0, st>>>(S, tm.tt);
  mark(3);
  k_trd_mgs<<<dim3(s1 - s0, kTrdMgsCtas), kTrdNT, 0, st>>>(S, s0);
  mark(4);
  for (int pass = 0; pass < kTrdNsSteps; ++pass) {
    if (tm.ozp.total > 0) k_trd_oz_pack<<<tm.ozp.total, kOzNT, 0, st>>>(S, tm.ozp, pass);
    if (tm.ozg.total > 0) k_trd_oz_gram<<<tm.ozg.total, kOzNT, kOzSmem, st>>>(S, tm.ozg, pass);
    k_trd_ns<<<tm.tsq.total, kGNT, 0, st>>>(S, tm.tsq, pass);
  }
  mark(5);
  if (tm.tbt.total > 0) {  // n < kBtBlockedMinN
    k_trd_backtf_reg<16><<<tm.tbt.total, kTrdNT, 0, st>>>(S, tm.tbt);
    ++nl;
  }
  nl += launch_bt(S, tm, max_n, st);  // the larger ones
  k_trd_finish<<<s1 - s0, kTrdNT, 0, st>>>(S, s0);
  mark(6);
  return nl + 7 + 3 * kTrdNsSteps;
}

}  // namespace cmaes_gb300

// kernels_small.cu -- small searches: n <= kJacobiSmallN (32).
//
//   k_small_eig          C = B D^2 B^T of one search in one CTA, everything in
//                        shared memory (any precision).
//   k_small_generations  whole generations (Algorithm 1 lines 4-10 and the
//                        stop / restart of Algorithm 2) of FP64 searches whose
//                        population panel is small too, one CTA per search,
//                        any number of generations in one launch.
//
// What bounds them: at n = 10, lambda = 10 a generation is ~10^4 operations, so its time
// is chains and launches. As 18 launches of the phase kernels it took 277 us: 2 - 8 us
// each for a kernel's start and its loads, and 100 us for the Jacobi sweeps. Here the
// state stays in shared memory from generation to generation, the phases are one block
// barrier apart and work only the entries there are, and a Jacobi step's chain is ~1000
// clocks instead of ~2500: 49 us, of which 32 are the decomposition.
//
// A generation's sums have the operands and the order of the phase kernels': the
// products are those of gemm_tile_f64 on integers, the rest follows each kernel's
// partial sums. So a search has the same bits here and there -- beside a larger search,
// under profiling, between ask and tell -- and f is that of the allocation-free
// evaluation. (Plain FP64 sums of another order: 53 us.)
//
// A generation's code passes through the instruction cache every time: written out as
// the compiler does by itself it was 391 KB, and every phase began with ~3000 clocks of
// misses. The loops over a CTA's work and over a sum are therefore not unrolled (192 KB).
#include "descent.cuh"

namespace cmaes_gb300 {

namespace {

constexpr int kSmNT = 256;
constexpr int kSmNW = kSmNT / 32;
constexpr float kSmTol = 1e-14f;  // the cyclic Jacobi's relative threshold
constexpr int kSmMaxSweeps = 40;
constexpr double kSmPdFloor = 1e-16;

__device__ __forceinline__ int uniform(int x) { return __shfl_sync(0xffffffffu, x, 0); }

// e / d for 0 <= e < 2^20, rd = 1 / d in FP32: (e + 1/2) / d is at least 1/(2 d)
// away from an integer, far more than the rounding of two FP32 operations.
__device__ __forceinline__ int quotient(int e, float rd) {
  return __float2int_rz((static_cast<float>(e) + 0.5f) * rd);
}

// |x| in FP32, cut to 20 bits of mantissa, by the bits (a conversion takes the FP64
// pipe); below 2^-126 it is zero.
__device__ __forceinline__ unsigned sm_float_bits(double x) {
  const int hi = __double2hiint(x) & 0x7fffffff, e = hi - (896 << 20);
  return e < (1 << 20) ? 0u : static_cast<unsigned>(min(e, 0xff << 20)) << 3;
}

// sum_k x[sx k] y[k], k < n, in four chains
template <class Y>
__device__ __forceinline__ double sm_dot(int n, const double* x, int sx, const Y* y) {
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int k = 0;
#pragma unroll 1
  for (; k + 4 <= n; k += 4, x += 4 * sx, y += 4) {
    const double x0 = x[0], x1 = x[sx], x2 = x[2 * sx], x3 = x[3 * sx];
    a0 = fma(x0, static_cast<double>(y[0]), a0);
    a1 = fma(x1, static_cast<double>(y[1]), a1);
    a2 = fma(x2, static_cast<double>(y[2]), a2);
    a3 = fma(x3, static_cast<double>(y[3]), a3);
  }
  if (k < n) a0 = fma(x[0], static_cast<double>(y[0]), a0);
  if (k + 1 < n) a1 = fma(x[sx], static_cast<double>(y[1]), a1);
  if (k + 2 < n) a2 = fma(x[2 * sx], static_cast<double>(y[2]), a2);
  return (a0 + a1) + (a2 + a3);
}

// Shared memory of the eigensolver, N = n rounded up to even: the matrices (leading
// dimension N + 1: A, T, E, X, the FP32 pair), which nothing outlives, and a step's
// rotations with the index tables of the two triangles.
struct SmEig {
  double *A, *T, *E, *X, *c, *s, *t, *ev;
  float *A32, *V32;
  int *p, *q, *rk;
  unsigned char *bp, *bq;  // the pair-block grid's upper triangle
  unsigned char *ui, *uj;  // the upper triangle of an n x n matrix
};

__host__ __device__ inline int sm_even(int n) { return n + (n & 1); }
__host__ __device__ inline size_t sm_mat(int n) { return static_cast<size_t>(sm_even(n) + 1) * sm_even(n); }
__host__ __device__ inline size_t sm_eig_mats(int n) { return 5 * sm_mat(n); }
__host__ __device__ inline size_t sm_eig_rest(int n) {
  const size_t N = sm_even(n), P = N / 2;
  return 3 * P + N + (2 * P + N + 1) / 2 + (P * (P + 1) + N * (N + 1) + 7) / 8 + 2;
}

__device__ SmEig sm_eig_carve(double* mats, double* rest, int n) {
  const int N = sm_even(n), P = N / 2;
  SmEig w;
  w.A = mats;
  w.T = w.A + sm_mat(n);
  w.E = w.T + sm_mat(n);
  w.X = w.E + sm_mat(n);
  w.A32 = reinterpret_cast<float*>(w.X + sm_mat(n));
  w.V32 = w.A32 + sm_mat(n);
  w.c = rest;
  w.s = w.c + P;
  w.t = w.s + P;
  w.ev = w.t + P;
  w.p = reinterpret_cast<int*>(w.ev + N);
  w.q = w.p + P;
  w.rk = w.q + P;
  w.bp = reinterpret_cast<unsigned char*>(w.rk + N + (N & 1));
  w.bq = w.bp + P * (P + 1) / 2;
  w.ui = w.bq + P * (P + 1) / 2;
  w.uj = w.ui + N * (N + 1) / 2;
  return w;
}

// c = (1 + t^2)^(-1/2) for the FP32 value t: to FP64 accuracy from an FP32 seed
// by one third-order Newton-type step, so that (c, t c) is orthonormal to
// rounding; in FP32 the seed itself.
__device__ __forceinline__ void sm_cos(float tf, double& c) {
  const double t = static_cast<double>(tf), x = fma(t, t, 1.0);
  const double y = static_cast<double>(rsqrtf(fmaf(tf, tf, 1.f)));
  const double h = fma(-x * y, y, 1.0);
  c = fma(y * h, fma(0.375, h, 0.5), y);
}
__device__ __forceinline__ void sm_cos(float tf, float& c) { c = rsqrtf(fmaf(tf, tf, 1.f)); }

// Cyclic Jacobi on the symmetric A (N x N, leading dimension ld, a zero row and
// column beyond n), V <- V J over n rows. A pair turns when rotates(app, aqq,
// apq, p, q) says so (FP32 values). Round-robin steps of N / 2 disjoint pairs; a
// step's t = tan(phi) is an FP32 value in either type (its error leaves 2^-23
// of a_pq, which a later step takes). FP64 operations (66 clocks each, 19 of a
// whole SM's pipe a warp) stay where the result needs them: d = a_qq - a_pp, c,
// s and the updates. All kSmNT threads call it; returns the sweeps.
template <class T, class Test>
__device__ int sm_jacobi(int n, T* A, T* V, const SmEig& w, int max_sweeps, int* rot, const Test& rotates) {
  __shared__ unsigned sh_mask;
  const int N = sm_even(n), P = N / 2, ld = N + 1, M = N - 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = uniform(tid >> 5);
  T* rc = reinterpret_cast<T*>(w.c);
  T* rs = reinterpret_cast<T*>(w.s);
  T* rt = reinterpret_cast<T*>(w.t);
  const int nblk = P * (P + 1) / 2;
  const float rn = 1.0f / n;
  int sweeps = 0, quiet = 0;
  bool converged = false;
  for (; sweeps < max_sweeps && !converged; ++sweeps) {
    for (int r = 0; r < M; ++r) {
      if (warp == 0) {  // pair `lane` of round-robin step r (player N - 1 fixed)
        bool act = false;
        if (lane < P) {
          const int p = lane == 0 ? r : (r + lane >= M ? r + lane - M : r + lane);
          const int q = lane == 0 ? M : (r - lane < 0 ? r - lane + M : r - lane);
          T c = 1, s = 0, t = 0;
          if (p < n && q < n) {
            const T app = A[p + ld * p], aqq = A[q + ld * q], apq = A[p + ld * q];
            const T d = aqq - app;
            const float af = static_cast<float>(apq);
            if (rotates(static_cast<float>(app), static_cast<float>(aqq), af, p, q)) {
              act = true;
              const float df = static_cast<float>(d);
              float tf;
              if (fabsf(af) * 0x1p40f < fabsf(df)) {
                tf = __fdividef(af, df);
              } else {
                const float th = __fdividef(df, af + af);
                tf = __fdividef(th >= 0.f ? 1.f : -1.f, fabsf(th) + sqrtf(fmaf(th, th, 1.f)));
              }
              t = static_cast<T>(tf);
              sm_cos(tf, c);
              s = t * c;
            }
          }
          rc[lane] = c;
          rs[lane] = s;
          rt[lane] = t;
          w.p[lane] = p;
          w.q[lane] = q;
        }
        const unsigned mask = __ballot_sync(0xffffffffu, act);
        if (lane == 0) {
          sh_mask = mask;
          *rot += __popc(mask);
        }
      }
      __syncthreads();
      const unsigned mask = sh_mask;
      if (mask == 0u) {
        // a quiet step: every pair meets once in M consecutive steps; a check of
        // the whole matrix ends the window early
        ++quiet;
        if (quiet == 1 || quiet % 16 == 0) {
          int pend = 0;
#pragma unroll 1
          for (int e = tid; e < n * (n + 1) / 2; e += kSmNT) {
            const int i = w.ui[e], j = w.uj[e];
            if (i < j)
              pend |= rotates(static_cast<float>(A[i + ld * i]), static_cast<float>(A[j + ld * j]),
                              static_cast<float>(A[i + ld * j]), i, j);
          }
          if (!__syncthreads_or(pend)) quiet = M;
        } else {
          __syncthreads();  // sh_mask is read before the next step writes it
        }
        if (quiet >= M) {
          converged = true;
          break;
        }
        continue;
      }
      quiet = 0;
      // A <- J^T A J by 2 x 2 blocks of pairs (upper triangle, mirrored), and
      // V <- V J, an entry pair per thread
#pragma unroll 1
      for (int e = tid; e < nblk + P * n; e += kSmNT) {
        if (e >= nblk) {
          const int k = quotient(e - nblk, rn), row = (e - nblk) - k * n;
          if (!((mask >> k) & 1u)) continue;
          const int p = w.p[k], q = w.q[k];
          const T c = rc[k], s = rs[k], vp = V[row + ld * p], vq = V[row + ld * q];
          V[row + ld * p] = c * vp - s * vq;
          V[row + ld * q] = s * vp + c * vq;
          continue;
        }
        const int Pi = w.bp[e], Qi = w.bq[e];
        if (!(((mask >> Pi) | (mask >> Qi)) & 1u)) continue;
        const int p1 = w.p[Pi], q1 = w.q[Pi], p2 = w.p[Qi], q2 = w.q[Qi];
        if (Pi == Qi) {
          const T app = A[p1 + ld * p1], aqq = A[q1 + ld * q1], apq = A[p1 + ld * q1];
          const T t = rt[Pi], c = rc[Pi], c2 = c * c, tq = t * apq;
          const T x = c2 * (t * (t * aqq - 2 * apq) + app);
          const T y = c2 * (t * (t * app + 2 * apq) + aqq);
          const T z = c2 * (t * (app - aqq - tq) + apq);
          A[p1 + ld * p1] = x;
          A[q1 + ld * q1] = y;
          A[p1 + ld * q1] = z;
          A[q1 + ld * p1] = z;
          continue;
        }
        const T cP = rc[Pi], sP = rs[Pi], cQ = rc[Qi], sQ = rs[Qi];
        const T a = A[p1 + ld * p2], bb = A[p1 + ld * q2], c = A[q1 + ld * p2], d = A[q1 + ld * q2];
        const T y00 = a * cQ - bb * sQ, y01 = a * sQ + bb * cQ;
        const T y10 = c * cQ - d * sQ, y11 = c * sQ + d * cQ;
        const T x00 = cP * y00 - sP * y10, x01 = cP * y01 - sP * y11;
        const T x10 = sP * y00 + cP * y10, x11 = sP * y01 + cP * y11;
        A[p1 + ld * p2] = x00;
        A[p2 + ld * p1] = x00;
        A[p1 + ld * q2] = x01;
        A[q2 + ld * p1] = x01;
        A[q1 + ld * p2] = x10;
        A[p2 + ld * q1] = x10;
        A[q1 + ld * q2] = x11;
        A[q2 + ld * q1] = x11;
      }
      __syncthreads();
    }
  }
  return sweeps;
}

// out(i, j) = sum_k x(k, i) y(k, j) (TN) or sum_k x(i, k) y(k, j), n x n; SYM:
// the upper triangle, mirrored. epi(i, j, sum) gives the stored value.
template <bool TN, bool SYM, class Y, class Epi>
__device__ __forceinline__ void sm_product(int n, int ld, const SmEig& w, double* out, const double* x, const Y* y,
                                           const Epi& epi) {
  const int count = SYM ? n * (n + 1) / 2 : n * n;
  const int sx = TN ? 1 : ld;
  const float rn = 1.0f / n;
#pragma unroll 1
  for (int e = threadIdx.x; e < count; e += kSmNT) {
    const int j = SYM ? w.uj[e] : quotient(e, rn), i = SYM ? w.ui[e] : e - j * n;
    const double v = epi(i, j, sm_dot(n, x + (TN ? ld * i : i), sx, y + ld * j));
    out[i + ld * j] = v;
    if (SYM) out[j + ld * i] = v;
  }
}

// Eigendecomposition of C (leading dimension ld = N + 1) from the previous
// basis B (same layout), which it replaces by the new one in canonical form;
// ev: the eigenvalues with the PD guard in ascending order; C's diagonal takes
// the guard's shift. The refined route of kernels_eig_mixed.cu in one CTA:
//   A = B^T C B; FP32 Jacobi sweeps on it (~400 clocks a step against ~3800 in
//   FP64); two refinement steps (Ogita & Aishima 2018: S = X^T C X, G = X^T X,
//   lambda_i = s_ii / g_ii, e_ij = (s_ij - lambda_j g_ij) / (lambda_j -
//   lambda_i), X <- X + X E; pairs too close for first order get -g_ij / 2)
//   and a Newton-Schulz step; A = X^T C X; FP64 Jacobi on what is left above
//   the rounding level of that product's entries.
// A shift by tr(A) / n lets FP32 resolve a spectrum of nearly equal eigenvalues;
// a graded A is left as it is, so that its small eigenvalues keep their FP32
// relative accuracy. All kSmNT threads call it. Returns the sweeps of both; *rot the
// FP64 ones' rotations (thread 0).
constexpr double kSmSep = 0x1p-10, kSmDefect = 0x1p-28;
struct SmSweeps {
  int f64, f32;
};

// The index tables, once per launch.
__device__ void small_eig_tables(int n, const SmEig& w) {
  const int P = sm_even(n) / 2, tid = threadIdx.x;
#pragma unroll 1
  for (int b = tid; b < P * (P + 1) / 2; b += kSmNT) {
    int Q = 0;
    while ((Q + 1) * (Q + 2) / 2 <= b) ++Q;
    w.bq[b] = static_cast<unsigned char>(Q);
    w.bp[b] = static_cast<unsigned char>(b - Q * (Q + 1) / 2);
  }
#pragma unroll 1
  for (int b = tid; b < n * (n + 1) / 2; b += kSmNT) {
    int j = 0;
    while ((j + 1) * (j + 2) / 2 <= b) ++j;
    w.uj[b] = static_cast<unsigned char>(j);
    w.ui[b] = static_cast<unsigned char>(b - j * (j + 1) / 2);
  }
}

__device__ SmSweeps small_eig(int n, double* C, double* B, const SmEig& w, int* rot) {
  __shared__ int sh_big, sh_rot32;
  __shared__ float sh_shift;
  const int N = sm_even(n), ld = N + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = uniform(tid >> 5);
  double *A = w.A, *T = w.T, *E = w.E, *X = w.X;
#pragma unroll 1
  for (int e = tid; e < N * N; e += kSmNT) {  // (the dummy row and column of an odd n stay zero)
    A[e % N + ld * (e / N)] = 0.0;
    w.A32[e % N + ld * (e / N)] = 0.0f;
    w.V32[e % N + ld * (e / N)] = e % N == e / N ? 1.0f : 0.0f;
  }
  if (tid == 0) {
    *rot = sh_rot32 = 0;
    sh_big = 0;
  }
  __syncthreads();
  if (warp == 0 && lane < n) atomicMax(&sh_big, (__double2hiint(fabs(C[lane + ld * lane])) >> 20) & 0x7ff);
  sm_product<false, false>(n, ld, w, T, C, B, [](int, int, double v) { return v; });
  __syncthreads();
  const int big = min(max(sh_big, 1), 2045);
  const double up = __hiloint2double((2046 - big) << 20, 0);  // scales entries to at most ~1 (n for off-scale ones)
  const double down = __hiloint2double(big << 20, 0);
  sm_product<true, true>(n, ld, w, A, B, T, [&](int, int, double v) { return v * up; });
  __syncthreads();
  if (warp == 0) {
    const float d = lane < n ? static_cast<float>(A[lane + ld * lane]) : 0.0f;
    float hi = lane < n ? d : -INFINITY, lo = lane < n ? d : INFINITY, sum = d;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    if (lane == 0) sh_shift = lo * 64.0f >= hi ? sum / n : 0.0f;
  }
  __syncthreads();
  const float shift = sh_shift;
#pragma unroll 1
  for (int e = tid; e < n * n; e += kSmNT) {
    const int j = e / n, i = e - j * n;
    w.A32[i + ld * j] = static_cast<float>(A[i + ld * j] - (i == j ? static_cast<double>(shift) : 0.0));
  }
  __syncthreads();
  const float floor32 = shift != 0.0f ? 16.0f * 0x1p-24f * 2.0f : 0.0f;
  const int sweeps32 = sm_jacobi<float>(n, w.A32, w.V32, w, 12, &sh_rot32, [=](float app, float aqq, float apq, int, int) {
    return fabsf(apq) > floor32 && fabsf(apq) * rsqrtf(fabsf(app)) * rsqrtf(fabsf(aqq)) > 1e-6f;
  });
  __syncthreads();
  sm_product<false, false>(n, ld, w, X, B, w.V32, [](int, int, double v) { return v; });
  __syncthreads();
  for (int step = 0; step < 2; ++step) {
    sm_product<false, false>(n, ld, w, T, C, X, [&](int, int, double v) { return v * up; });
    sm_product<true, true>(n, ld, w, B, X, X, [](int, int, double v) { return v; });  // G
    __syncthreads();
    sm_product<true, true>(n, ld, w, A, X, T, [](int, int, double v) { return v; });  // S
    __syncthreads();
#pragma unroll 1
    for (int e = tid; e < n * (n + 1) / 2; e += kSmNT) {
      const int i = w.ui[e], j = w.uj[e];
      const double gij = B[i + ld * j];
      if (i == j) {
        E[i + ld * i] = 0.5 * (1.0 - gij);
        continue;
      }
      // s_ii / g_ii with g_ii = 1 + O(1e-6): 1 / g = 1 - d + d^2 to rounding
      auto ratio = [&](int l) {
        const double dl = B[l + ld * l] - 1.0;
        return A[l + ld * l] * fma(dl, dl - 1.0, 1.0);
      };
      const double sij = A[i + ld * j], li = ratio(i), lj = ratio(j);
      const double rg = 1.0 / (lj - li);
      double eij = fma(-lj, gij, sij) * rg, eji = -fma(-li, gij, sij) * rg;
      if (!(fabs(eij) < kSmSep && fabs(eji) < kSmSep)) eij = eji = -0.5 * gij;
      E[i + ld * j] = eij;
      E[j + ld * i] = eji;
    }
    __syncthreads();
    sm_product<false, false>(n, ld, w, T, X, E, [&](int i, int j, double v) { return X[i + ld * j] + v; });
    __syncthreads();
    double* q = X;
    X = T;
    T = q;
  }
  // Newton-Schulz: one step, or up to three from a defect whose square is above rounding
  // (pairs of repeated eigenvalues at the bound of the corrections); then A = X^T C X
#pragma unroll 1
  for (int ns = 0;; ++ns) {
    bool large = false;
    sm_product<true, true>(n, ld, w, E, X, X, [&](int i, int j, double v) {
      const double d = (i == j ? 1.0 : 0.0) - v;
      large |= fabs(d) > kSmDefect;
      return 0.5 * d;
    });
    const bool again = __syncthreads_or(large) && ns < 2;
    double* out = again ? T : B;
    sm_product<false, false>(n, ld, w, out, X, E, [&](int i, int j, double v) { return X[i + ld * j] + v; });
    __syncthreads();
    if (!again) break;
    T = X;
    X = out;
  }
  sm_product<false, false>(n, ld, w, T, C, B, [&](int, int, double v) { return v * up; });
  __syncthreads();
  sm_product<true, true>(n, ld, w, A, B, T, [](int, int, double v) { return v; });
  __syncthreads();
  if (tid == 0) sh_big = 0;
  __syncthreads();
  if (warp == 0 && lane < n) atomicMax(&sh_big, __float_as_int(fabsf(static_cast<float>(A[lane + ld * lane]))));
  __syncthreads();
  // The rounding of a_ij is within n eps of (|X|^T |C| |X|)_ij, and that of g_i g_j with
  // g_i = sum_k |x_ki| sqrt(c_kk), C being positive semi-definite: an entry below is not
  // turned. Where X mixes large and small c_kk this is the level of max a_ii; a graded
  // C whose X is near I keeps the relative test, and so its small eigenvalues.
  float *root = w.A32, *g = w.A32 + N;  // (the FP32 pair is done with)
  if (warp == 0 && lane < n) root[lane] = sqrtf(fabsf(static_cast<float>(C[lane + ld * lane] * up)));
  __syncwarp();
  if (warp == 0 && lane < n) {
    float sum = 0.0f;
#pragma unroll 1
    for (int k = 0; k < n; ++k)
      sum = fmaf(__uint_as_float(sm_float_bits(B[k + ld * lane])), root[k], sum);
    g[lane] = sum;
  }
  __syncthreads();
  const float noise = static_cast<float>(n) * 0x1p-53f, top = __int_as_float(sh_big);
  const int sweeps = sm_jacobi<double>(n, A, B, w, kSmMaxSweeps, rot, [=](float app, float aqq, float apq, int p, int q) {
    return fabsf(apq) > noise * fminf(top, g[p] * g[q]) &&
           fabsf(apq) * rsqrtf(fabsf(app)) * rsqrtf(fabsf(aqq)) > kSmTol;
  });
  // eigenvalues with the PD guard
  if (warp == 0) {
    const double e = lane < n ? A[lane + ld * lane] * down : 0.0;
    double lo = lane < n ? e : INFINITY, hi = lane < n ? e : -INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const double add = (lo < hi * kSmPdFloor) ? hi * kSmPdFloor - lo : 0.0;
    if (lane < n && add != 0.0) C[lane + ld * lane] += add;
    // ranks: ascending, ties by index
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      const double ej = __shfl_sync(0xffffffffu, e, j);
      rank += (ej < e) || (ej == e && j < lane);
    }
    if (lane < n) {
      w.rk[lane] = rank;
      w.ev[rank] = e + add;
    }
  }
  __syncthreads();
  // columns to their ranks (through T), the entry of largest magnitude (first
  // on ties) positive
  for (int j = warp; j < n; j += kSmNW) {
    const double v = lane < n ? B[lane + ld * j] : 0.0;
    const long long key = __double_as_longlong(fabs(v));
    const unsigned kh = static_cast<unsigned>(key >> 32);
    const unsigned mh = __reduce_max_sync(0xffffffffu, kh);
    const unsigned kl = kh == mh ? static_cast<unsigned>(key) : 0u;
    const unsigned ml = __reduce_max_sync(0xffffffffu, kl);
    const int first = __ffs(static_cast<int>(__ballot_sync(0xffffffffu, kh == mh && kl == ml))) - 1;
    const bool neg = __shfl_sync(0xffffffffu, v < 0.0 ? 1 : 0, first) != 0;
    if (lane < n) T[lane + ld * w.rk[j]] = neg ? -v : v;
  }
  __syncthreads();
#pragma unroll 1
  for (int e = tid; e < n * n; e += kSmNT) {
    const int j = e / n, i = e - j * n;
    B[i + ld * j] = T[i + ld * j];
  }
  __syncthreads();
  return SmSweeps{sweeps, sweeps32};
}

}  // namespace

// ---------------------------------------------------- eigendecomposition ----
__global__ void __launch_bounds__(kSmNT) k_small_eig(Search* S, int s0) {
  extern __shared__ double sdyn[];
  __shared__ int sh_rot;
  Search& s = S[s0 + blockIdx.x];
  if (s.done || !s.eig_due || s.n > kJacobiSmallN) return;
  const int n = s.n, ldn = s.ldn, N = sm_even(n), ld = N + 1, tid = threadIdx.x;
  double* C = sdyn;
  double* B = C + sm_mat(n);
  const SmEig w = sm_eig_carve(B + sm_mat(n), B + sm_mat(n) + sm_eig_mats(n), n);
  small_eig_tables(n, w);
#pragma unroll 1
  for (int e = tid; e < N * N; e += kSmNT) {
    const int i = e % N, j = e / N;
    const bool in = i < n && j < n;
    C[i + ld * j] = in ? 0.5 * (s.C[i + ldn * j] + s.C[j + ldn * i]) : 0.0;
    B[i + ld * j] = in ? s.B[i + ldn * j] : 0.0;
  }
  __syncthreads();
  const SmSweeps sweeps = small_eig(n, C, B, w, &sh_rot);
#pragma unroll 1
  for (int e = tid; e < n * n; e += kSmNT) s.B[e % n + ldn * (e / n)] = B[e % n + ld * (e / n)];
#pragma unroll 1
  for (int i = tid; i < n; i += kSmNT) {
    s.D[i] = sqrt(w.ev[i]);
    s.C[i + ldn * i] = C[i + ld * i];
  }
  if (tid == 0) {
    s.eig_sweeps = sweeps.f64;
    s.eig_count += 1;
    s.eig_sweeps_total += sweeps.f64;
    s.eig_sweeps32 += sweeps.f32;
    s.eig_rotations += sh_rot;
  }
}

static size_t small_eig_smem(int n) { return (2 * sm_mat(n) + sm_eig_mats(n) + sm_eig_rest(n)) * sizeof(double); }

void launch_small_eig(Search* S, int s0, int s1, int max_n, cudaStream_t st) {
  if (s1 > s0) k_small_eig<<<s1 - s0, kSmNT, small_eig_smem(max_n), st>>>(S, s0);
}

// ------------------------------------------------------ whole generations ----
namespace {

// Ordered integer key of a double (as in the counting rank), for maxima and
// minima off the FP64 pipe.
__device__ __forceinline__ long long order_bits(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}

struct SmGen {
  double *C, *B, *BD, *D, *m, *ps, *pc, *xs, *ld_, *yw, *zw, *w, *Z, *Y, *R, *U, *f;
  int2 *BDl, *Ql, *L;  // integer operands of the products: B D, Q, and the panel's
  int *eBD, *eQ, *eL;  // their scales: of a row, a row, a candidate
  unsigned long long* key;
  int* order;
  double *mats, *rest;  // of the eigensolver; the panels Z .. L lie where its matrices do
};

__host__ __device__ inline size_t sm_gen_panels(int n, int lam) {
  const size_t panels = 5 * static_cast<size_t>(n) * lam;
  return panels > sm_eig_mats(n) ? panels : sm_eig_mats(n);
}
__host__ __device__ inline size_t sm_gen_doubles(int n, int lam) {
  return 5 * sm_mat(n) + 9 * static_cast<size_t>(n) + lam / 2 + 1 + 2 * lam + 2 * ((lam + 1) / 2) + sm_eig_rest(n) +
         sm_gen_panels(n, lam);
}

__device__ SmGen sm_gen_carve(double* p, int n, int lam) {
  SmGen g;
  auto take = [&](size_t k) {
    double* q = p;
    p += k;
    return q;
  };
  g.C = take(sm_mat(n));
  g.B = take(sm_mat(n));
  g.BD = take(sm_mat(n));
  g.BDl = reinterpret_cast<int2*>(take(sm_mat(n)));
  g.Ql = reinterpret_cast<int2*>(take(sm_mat(n)));
  g.D = take(n);
  g.m = take(n);
  g.ps = take(n);
  g.pc = take(n);
  g.xs = take(n);
  g.ld_ = take(n);
  g.yw = take(n);
  g.zw = take(n);
  g.eBD = reinterpret_cast<int*>(take(n));
  g.eQ = g.eBD + n;
  g.w = take(lam / 2 + 1);
  g.f = take(lam);
  g.key = reinterpret_cast<unsigned long long*>(take(lam));
  g.order = reinterpret_cast<int*>(take((lam + 1) / 2));
  g.eL = reinterpret_cast<int*>(take((lam + 1) / 2));
  g.rest = take(sm_eig_rest(n));
  g.mats = p;
  g.Z = take(static_cast<size_t>(n) * lam);
  g.Y = take(static_cast<size_t>(n) * lam);
  g.R = take(static_cast<size_t>(n) * lam);
  g.U = take(static_cast<size_t>(n) * lam);
  g.L = reinterpret_cast<int2*>(take(static_cast<size_t>(n) * lam));
  return g;
}

// One K step of an output of gemm_tile_f64 added to acc: limbs a[sa k], b[sb k] with the
// scales ea, eb; the entries themselves A[sA k] and B[sB k], or B[sB order[k]]. (Not
// inlined, as the two below: a generation's code passes through the instruction cache
// each time, and these are called from three places.)
__device__ __noinline__ double sm_step(double acc, int kn, const int2* a, int sa, const int2* b, int sb, int ea,
                                       int eb, const double* A, int sA, const double* B, int sB, const int* order) {
  long long hh = 0, mid = 0;
  unsigned sum = 0;
#pragma unroll 2
  for (int k = 0; k < kn; ++k) {
    const int2 x = a[sa * k], y = b[sb * k];
    hh += static_cast<long long>(x.x) * y.x;
    mid += static_cast<long long>(x.x) * y.y;
    mid += static_cast<long long>(x.y) * y.x;
    sum += gemm_byte(x.x) * gemm_byte(y.x);
  }
  if (!gemm_in_f64(sum, ea, eb)) return acc + gemm_scaled<29>(hh, mid, ea + eb);
#pragma unroll 1
  for (int k = 0; k < kn; ++k) acc = fma(A[sA * k], B[sB * (order ? order[k] : k)], acc);
  return acc;
}

// The largest biased exponent of x[s k], k < n.
__device__ __forceinline__ int sm_scale(const double* x, int s, int n) {
  int e = 0;
  for (int k = 0; k < n; ++k) e = max(e, gemm_exponent(x[s * k]));
  return e;
}

// The n x n matrix x (entry (i, j) at x[i + lx j]) as integers by rows.
__device__ __noinline__ void sm_rows_as_integers(int n, int ld, const double* x, long long lx, int2* out, int* eo) {
#pragma unroll 1
  for (int e = threadIdx.x; e < n * n; e += kSmNT) {
    const int j = e / n, i = e - j * n;
    const int E = sm_scale(x + i, static_cast<int>(lx), n);
    out[i + ld * j] = gemm_limbs<29>(x[i + lx * j], E);
    if (j == 0) eo[i] = E;
  }
}

// The panel x (n x lam) as integers by columns.
__device__ __noinline__ void sm_panel_as_integers(int n, int lam, float rn, const double* x, int2* out, int* eo) {
#pragma unroll 1
  for (int e = threadIdx.x; e < n * lam; e += kSmNT) {
    const int k = quotient(e, rn), i = e - k * n;
    const int E = sm_scale(x + n * k, 1, n);
    out[e] = gemm_limbs<29>(x[e], E);
    if (i == 0) eo[k] = E;
  }
}

__device__ __forceinline__ double sm_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace

// PER_SM: the CTAs per SM that the registers are cut for. One search runs 15 % faster
// with a whole SM's; where more searches than SMs would wait, four side by side do more
// (20 generations of n = 10, lambda = 10: 965 and 1135 us; ten of 1000 such searches, two
// CTAs and four per SM: 2.08 and 1.56 ms; of 2000 with n = 20, lambda = 12: 9.6 and 7.8).
template <int PER_SM>
__global__ void __launch_bounds__(kSmNT, PER_SM) k_small_generations(Search* S, int s0, DevOptions o, int gens) {
  extern __shared__ double sdyn[];
  __shared__ double sh[32];
  __shared__ double sh_den, sh_psn, sh_hsig, sh_sigma, sh_best;
  __shared__ int sh_rot, sh_bits[2];
  Search& s = S[s0 + blockIdx.x];
  if (s.done) return;
  const int n = s.n, ldn = s.ldn, N = sm_even(n), ld = N + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = uniform(tid >> 5);
  const SmGen g = sm_gen_carve(sdyn, n, s.lam_cap);
  const SmEig we = sm_eig_carve(g.mats, g.rest, n);
  small_eig_tables(n, we);
  const int obj = s.obj, npairs = (n + 1) >> 1;
  const float rn = 1.0f / n, rp = 1.0f / npairs;
  const int tree_top = n > 16 ? 16 : n > 8 ? 8 : n > 4 ? 4 : n > 2 ? 2 : n - 1;  // f's first level with a pair

  for (int done_gens = 0; done_gens < gens;) {
    // ---- the state of this descent ----
    const int lam = s.lam, mu = s.mu, g_eig = s.g_eig, hist_len = s.hist_len, max_iter = s.max_iter;
    const double cs = s.cs, ds = s.ds, cc = s.cc, c1 = s.c1, cmu = s.cmu, chin = s.chin, mueff = s.mueff;
    int gen = s.gen, hist_count = s.hist_count;
#pragma unroll 1
    for (int e = tid; e < N * N; e += kSmNT) {
      const int i = e % N, j = e / N;
      const bool in = i < n && j < n;
      g.C[i + ld * j] = in ? s.C[i + ldn * j] : 0.0;
      g.B[i + ld * j] = in ? s.B[i + ldn * j] : 0.0;
      g.BD[i + ld * j] = in ? s.BD[i + ldn * j] : 0.0;
    }
    sm_rows_as_integers(n, ld, s.BD, ldn, g.BDl, g.eBD);
    if (obj != 3) sm_rows_as_integers(n, ld, s.Q, ldn, g.Ql, g.eQ);
#pragma unroll 1
    for (int i = tid; i < n; i += kSmNT) {
      g.D[i] = s.D[i];
      g.m[i] = s.m[i];
      g.ps[i] = s.ps[i];
      g.pc[i] = s.pc[i];
      g.xs[i] = s.xstar[i];
      g.ld_[i] = obj == 1 ? s.lamdiag[i] : 0.0;
    }
#pragma unroll 1
    for (int r = tid; r < mu; r += kSmNT) g.w[r] = s.w[r];
    if (tid == 0) {
      sh_sigma = s.sigma;
      sh_best = s.best_f;
    }
    __syncthreads();
    int flags = 0;
    bool due = false;
    // ---- generations until the block's count, a stop or a restart ----
    for (; done_gens < gens && !flags; ++done_gens) {
      // z; the denominator of the h_sigma test beside it
#pragma unroll 1
      for (int e = tid; e < npairs * lam; e += kSmNT) {
        const int k = quotient(e, rp), j = e - k * npairs;
        double z0, z1;
        normal_pair(static_cast<uint32_t>(j), static_cast<uint32_t>(k), static_cast<uint32_t>(gen),
                    stream_word(s.index, s.restart), o.key0, o.key1, z0, z1);
        g.Z[n * k + 2 * j] = z0;
        if (2 * j + 1 < n) g.Z[n * k + 2 * j + 1] = z1;
      }
      if (tid == kSmNT - 1) {
        sh_den = sqrt(1.0 - pow(1.0 - cs, 2.0 * (gen + 1)));
        sh_bits[0] = sh_bits[1] = 0;
      }
      __syncthreads();
      const double sigma = sh_sigma;
      sm_panel_as_integers(n, lam, rn, g.Z, g.L, g.eL);
      __syncthreads();
      // y = B D z, x = m + sigma y
#pragma unroll 1
      for (int e = tid; e < n * lam; e += kSmNT) {
        const int k = quotient(e, rn), i = e - k * n;
        const double y = sm_step(0.0, n, g.BDl + i, ld, g.L + n * k, 1, g.eBD[i], g.eL[k], g.BD + i, ld, g.Z + n * k, 1,
                                 nullptr);
        const double x = step_from(g.m[i], sigma, y);
        g.Y[n * k + i] = y;
        g.R[n * k + i] = x - g.xs[i];
        s.X[i + static_cast<long long>(ldn) * k] = x;
      }
      __syncthreads();
      if (obj != 3) {
        sm_panel_as_integers(n, lam, rn, g.R, g.L, g.eL);
        __syncthreads();
      }
      // the objective's terms
#pragma unroll 1
      for (int e = tid; e < n * lam; e += kSmNT) {
        const int k = quotient(e, rn), i = e - k * n;
        double term;
        if (obj == 3) {
          term = g.R[e] * g.R[e];
        } else {
          const double u = sm_step(0.0, n, g.Ql + i, ld, g.L + n * k, 1, g.eQ[i], g.eL[k], s.Q + i, ldn, g.R + n * k, 1,
                                   nullptr);
          term = objective_term(obj, g.ld_[i], u);
        }
        g.U[e] = term;
      }
      __syncthreads();
      // f: the shuffle tree of k_colreduce_f over 32 lanes
#pragma unroll 1
      for (int k = tid; k < lam; k += kSmNT) {
        double* u = g.U + n * k;
#pragma unroll 1
        for (int off = tree_top; off > 0; off >>= 1)
#pragma unroll 1
          for (int i = 0; i < min(off, n - off); i += 4) {  // four independent sums at a time
            double v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = i + q < min(off, n - off) ? u[i + q] + u[i + q + off] : 0.0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (i + q < min(off, n - off)) u[i + q] = v[q];
          }
        const double sum = n < 32 ? u[0] + 0.0 : u[0];
        const double f = (obj == 2) ? 10.0 * n + sum : sum;
        g.f[k] = f;
        g.key[k] = rank_key(f);
        s.f[k] = f;
      }
      __syncthreads();
      // rank: ascending f, ties by index
#pragma unroll 1
      for (int k = tid; k < lam; k += kSmNT) {
        const unsigned long long key = g.key[k];
        int r = 0;
        for (int j = 0; j < k; ++j) r += g.key[j] <= key;
        for (int j = k + 1; j < lam; ++j) r += g.key[j] < key;
        g.order[r] = k;
        s.order[r] = k;
      }
      __syncthreads();
      // <y>_w and <z>_w: eight threads per entry, for the eight warps of k_recomb_partial
#pragma unroll 1
      for (int e = tid; e < ((2 * n * 8 + 31) & ~31); e += kSmNT) {
        const int id = e >> 3, i = id % n;
        const double* src = id < n ? g.Y : g.Z;
        double total = 0.0;
        for (int r0 = 0; r0 < mu; r0 += 256) {
          double a = 0.0, v = 0.0;
          if (id < 2 * n)
            for (int r = r0 + (e & 7); r < min(mu, r0 + 256); r += 8) a = fma(g.w[r], src[n * g.order[r] + i], a);
#pragma unroll
          for (int q = 0; q < 8; ++q) v += __shfl_sync(0xffffffffu, a, (lane & 24) + q);
          total += v;
        }
        if ((e & 7) == 0 && id < 2 * n) (id < n ? g.yw : g.zw)[i] = total;
      }
      __syncthreads();
      // p_sigma, its norm, h_sigma (warp 0); the mean (warp 1); the best point (warp 2)
      if (warp == 0) {
        double ps = 0.0;
        if (lane < n) {
          double part[8] = {}, v = 0.0;  // the eight warps of k_psigma_partial
#pragma unroll 1
          for (int j0 = 0; j0 < n; j0 += 8)
#pragma unroll
            for (int q = 0; q < 8; ++q)
              if (j0 + q < n) part[q] = fma(g.B[lane + ld * (j0 + q)], g.zw[j0 + q], part[q]);
#pragma unroll
          for (int q = 0; q < 8; ++q) v += part[q];
          ps = path_step(cs, g.ps[lane], sqrt(cs * (2.0 - cs) * mueff), v);
          g.ps[lane] = ps;
        }
        const double psn = sqrt(sm_sum(ps * ps));
        if (lane == 0) {
          sh_psn = psn;
          sh_hsig = (psn / sh_den < (1.4 + 2.0 / (n + 1.0)) * chin) ? 1.0 : 0.0;
        }
      } else if (warp == 1) {
        if (lane < n) g.m[lane] = step_from(g.m[lane], sigma, g.yw[lane]);
      } else if (warp == 2) {
        const int i0 = g.order[0];
        const double f0 = g.f[i0];
        if (f0 < sh_best) {
          if (lane < n) s.best_x[lane] = s.X[lane + static_cast<long long>(ldn) * i0];
          __syncwarp();
          if (lane == 0) sh_best = f0;
        }
        if (lane == 0) {
          s.hist[hist_count % hist_len] = f0;
          s.hist[s.hist_cap + hist_count % hist_len] = 0.0;
        }
      }
      ++hist_count;
      __syncthreads();
      const double hsig = sh_hsig, psn = sh_psn;
      if (tid == kSmNT - 1) sh_sigma = sigma * exp((cs / ds) * (psn / chin - 1.0));
      if (warp == 0 && lane < n) g.pc[lane] = path_step(cc, g.pc[lane], hsig * sqrt(cc * (2.0 - cc) * mueff), g.yw[lane]);
      __syncthreads();
      // the rank-mu product's operands as integers, in the chunks of k_cov_partial and the
      // steps of its tile: w y at R and L, y at L + mu n, their scales at Z
      const int kc = s.cov_kc, chunk_steps = ceil_div(kc, gemm_step(kc));
      int *ea = reinterpret_cast<int*>(g.Z), *eb = ea + n * ceil_div(mu, kc) * chunk_steps;
      // rank r's step and that step's range
      auto step_of = [&](int r, int& r0, int& r1) {
        const int c = r / kc, last = min(mu, (c + 1) * kc), len = gemm_step(last - c * kc), q = (r - c * kc) / len;
        r0 = c * kc + q * len;
        r1 = min(last, r0 + len);
        return c * chunk_steps + q;
      };
#pragma unroll 1
      for (int e = tid; e < mu * n; e += kSmNT) {
        const int r = quotient(e, rn);
        g.R[e] = g.w[r] * g.Y[n * g.order[r] + (e - r * n)];
      }
      __syncthreads();
#pragma unroll 1
      for (int e = tid; e < mu * n; e += kSmNT) {
        const int r = quotient(e, rn), i = e - r * n;
        int r0, r1, a = 0, b = 0;
        const int st = step_of(r, r0, r1);
        for (int q = r0; q < r1; ++q) {
          a = max(a, gemm_exponent(g.R[n * q + i]));
          b = max(b, gemm_exponent(g.Y[n * g.order[q] + i]));
        }
        if (r == r0) {
          ea[n * st + i] = a;
          eb[n * st + i] = b;
        }
        g.L[e] = gemm_limbs<29>(g.R[e], a);
        g.L[mu * n + e] = gemm_limbs<29>(g.Y[n * g.order[r] + i], b);
      }
      __syncthreads();
      // C, upper triangle with its mirror
      {
        const double keep = cov_keep(c1, cmu, cc, hsig);
#pragma unroll 1
        for (int e = tid; e < n * (n + 1) / 2; e += kSmNT) {
          const int i = we.ui[e], j = we.uj[e];
          double acc = 0.0, chunk = 0.0;
          for (int r = 0; r < mu;) {
            int r0, r1;
            const int st = step_of(r, r0, r1);
            chunk = sm_step(chunk, r1 - r0, g.L + n * r0 + i, n, g.L + n * (mu + r0) + j, n, ea[n * st + i],
                            eb[n * st + j], g.R + n * r0 + i, n, g.Y + j, n, g.order + r0);
            r = r1;
            if (r % kc == 0 || r == mu) {
              acc += chunk;
              chunk = 0.0;
            }
          }
          const double v = cov_entry(keep, g.C[i + ld * j], c1, g.pc[i], g.pc[j], cmu, acc);
          g.C[i + ld * j] = v;
          g.C[j + ld * i] = v;
        }
      }
      ++gen;
      due = (gen % g_eig) == 0;
      __syncthreads();
      if (due) {
        const SmSweeps sweeps = small_eig(n, g.C, g.B, we, &sh_rot);
#pragma unroll 1
        for (int i = tid; i < n; i += kSmNT) g.D[i] = sqrt(we.ev[i]);
        if (tid == 0) {
          s.eig_sweeps = sweeps.f64;
          s.eig_count += 1;
          s.eig_sweeps_total += sweeps.f64;
          s.eig_sweeps32 += sweeps.f32;
          s.eig_rotations += sh_rot;
        }
        __syncthreads();
#pragma unroll 1
        for (int e = tid; e < n * n; e += kSmNT) {
          const int i = e % n, j = e / n;
          g.BD[i + ld * j] = g.B[i + ld * j] * g.D[j];
        }
        __syncthreads();
        sm_rows_as_integers(n, ld, g.BD, ld, g.BDl, g.eBD);
      }
      // ---- stop tests: the axis, coordinate, TolX and finiteness ones in warp
      // 0 (a lane per coordinate), the history in warp 1 ----
      const double sig = sh_sigma;
      if (warp == 0) {
        const int j = gen % n;
        const double axis = __dmul_rn(__dmul_rn(0.1, sig), g.D[j]);
        const double coord = __dmul_rn(0.2, sig), tolx = o.tol_x_factor * s.sigma0;
        bool tolx_fail = false, moves = false, stuck = false, bad = false;
        double dmax = 0.0, dmin = INFINITY;
        if (lane < n) {
          const double cii = g.C[lane + ld * lane], sd = sqrt(fmax(cii, 0.0)), mi = g.m[lane];
          tolx_fail = !(__dmul_rn(sig, fabs(g.pc[lane])) < tolx) || !(__dmul_rn(sig, sd) < tolx);
          moves = __dadd_rn(mi, __dmul_rn(axis, g.B[lane + ld * j])) != mi;
          stuck = __dadd_rn(mi, __dmul_rn(coord, sd)) == mi;
          bad = !isfinite(mi) || !isfinite(cii);
          dmax = fmax(dmax, g.D[lane]);
          dmin = fmin(dmin, g.D[lane]);
        }
        const bool any_fail = __any_sync(0xffffffffu, tolx_fail), any_moves = __any_sync(0xffffffffu, moves);
        const bool any_stuck = __any_sync(0xffffffffu, stuck), any_bad = __any_sync(0xffffffffu, bad);
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) {
          dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, q));
          dmin = fmin(dmin, __shfl_xor_sync(0xffffffffu, dmin, q));
        }
        if (lane == 0) {
          int fl = 0;
          if (sh_best < o.f_target) fl |= 1;
          if (gen >= max_iter) fl |= 2;
          if (!any_fail) fl |= 8;
          if (__dmul_rn(dmax, dmax) > __dmul_rn(__dmul_rn(o.cond_max, dmin), dmin)) fl |= 16;
          if (!any_moves) fl |= 32;
          if (any_stuck) fl |= 64;
          if (any_bad || !isfinite(sig)) {
            fl |= 128;
            atomicOr(s.err, kDevErrNonFinite);
          }
          sh_bits[0] = fl;
        }
      } else if (warp == 1 && hist_count >= hist_len) {
        // fmin / fmax ignore a NaN entry; the ordered keys are compared without it too
        long long hi = order_bits(-INFINITY), lo = order_bits(INFINITY);
        for (int q = lane; q < hist_len; q += 32) {
          const double v = s.hist[q];
          if (isnan(v)) continue;
          hi = max(hi, order_bits(v));
          lo = min(lo, order_bits(v));
        }
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) {
          hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, q));
          lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, q));
        }
        if (lane == 0) {
          const double a = __longlong_as_double(hi >= 0 ? hi : (hi ^ 0x7fffffffffffffffLL));
          const double b = __longlong_as_double(lo >= 0 ? lo : (lo ^ 0x7fffffffffffffffLL));
          if (a - b < o.tol_hist_fun) sh_bits[1] = 4;
        }
      }
      __syncthreads();
      flags = (sh_bits[0] | sh_bits[1]) & o.stop_mask;
      __syncthreads();  // sh_bits is cleared in the next generation
    }
    // ---- the state back to its place ----
#pragma unroll 1
    for (int e = tid; e < n * n; e += kSmNT) {
      const int i = e % n, j = e / n;
      s.C[i + ldn * j] = g.C[i + ld * j];
      s.B[i + ldn * j] = g.B[i + ld * j];
      s.BD[i + ldn * j] = g.BD[i + ld * j];
    }
#pragma unroll 1
    for (int i = tid; i < n; i += kSmNT) {
      s.D[i] = g.D[i];
      s.m[i] = g.m[i];
      s.ps[i] = g.ps[i];
      s.pc[i] = g.pc[i];
      s.yw[i] = g.yw[i];
      s.zw[i] = g.zw[i];
    }
    if (tid == 0) {
      s.psnorm = sh_psn;
      s.hsig = sh_hsig;
      s.sigma = sh_sigma;
      s.best_f = sh_best;
      s.gen = gen;
      s.hist_count = hist_count;
      s.eig_due = due;
      s.flags = flags;
    }
    __syncthreads();
    if (flags) {
      // a restart that would outgrow the panels allocated for lambda ends the search
      const bool ends = (flags & 1) || s.restart + 1 > o.max_restarts || (o.ipop_double && 2 * s.lam > s.lam_cap);
      if (ends || o.restart_hold) {
        __syncthreads();
        if (tid == 0) s.done = ends ? 1 : 2;
        return;
      }
      restart_descent<kSmNT>(s, o, sh);
    }
  }
}

bool small_generation(int n, int lam_cap) {
  return n <= kJacobiSmallN && lam_cap <= kSmallLambda && static_cast<long long>(n) * lam_cap <= kSmallPanel;
}

size_t small_generation_smem(int n, int lam_cap) { return sm_gen_doubles(n, lam_cap) * sizeof(double); }

static const void* small_fn(bool dense) {
  return dense ? reinterpret_cast<const void*>(k_small_generations<4>) : reinterpret_cast<const void*>(k_small_generations<1>);
}

cudaError_t small_smem_limits() {
  for (const void* k : {small_fn(false), small_fn(true), reinterpret_cast<const void*>(k_small_eig)})
    if (const cudaError_t e = smem_limit_max(k); e != cudaSuccess) return e;
  return cudaSuccess;
}

// Whether `count` searches overflow the CTAs of the kernel for few, and more fit of the other.
cudaError_t small_generations_dense(int count, size_t smem, bool* dense) {
  int dev = 0, sms = 0, few = 0, many = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&few, small_fn(false), kSmNT, smem)) != cudaSuccess ||
      (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&many, small_fn(true), kSmNT, smem)) != cudaSuccess)
    return e;
  *dense = many > few && count > static_cast<long long>(few) * sms;
  return cudaSuccess;
}

void launch_small_generations(Search* S, int count, DevOptions o, int gens, size_t smem, bool dense, cudaStream_t st) {
  if (dense) k_small_generations<4><<<count, kSmNT, smem, st>>>(S, 0, o, gens);
  else k_small_generations<1><<<count, kSmNT, smem, st>>>(S, 0, o, gens);
}

}  // namespace cmaes_gb300

// kernels_eig_refine.cu -- the dense FP64-accurate products of the refined
// eigendecomposition (kernels_eig_mixed.cu) for kJacobiSmallN < n <=
// kEigMixedMaxN, fused: one thread-block cluster per search runs the warm start
// A = B^T C B in one launch, and the basis X0 = B V32, both Ogita-Aishima steps,
// the Newton-Schulz step and A = X^T C X in another.
//
// As one launch per product the 13 products were bound by the FP64 pipe (n = 100,
// ten searches: 10^7 FMAs at 1.7 per clock and SM are 20 of the 25 us a launch
// took) and, for small n, by the latency of a launch whose every lane runs a chain
// of n FP64 FMAs (n = 40: 12.5 us). Here they run on integers and stay inside a
// cluster:
//   - Columns are dealt to the CTAs of the cluster in turn. Every product is
//     R(i, j) = sum_k M(k, i) Y(k, j) or sum_k M(i, k) Y(k, j) with Y the CTA's own
//     columns, which it keeps in shared memory, and M a whole matrix (C, the basis)
//     that the owners publish to global memory as integers; M passes through shared
//     memory in steps of 32 k. A cluster barrier follows each publication.
//   - Column j of an operand is scaled by the power of two above its largest entry
//     and rounded to 55 bits, (h 2^28 + l); h h and h l + l h are summed exactly over
//     the whole K (n <= 160: below 2^62 and 2^63), so an output costs 3 n integer
//     multiply-adds and one conversion. Rounding an entry (2^-56 of its column's
//     largest) and leaving l l out (2^-56 of the product of the scales, per term)
//     is less than the n roundings of an FP64 sum. Where M is used along its rows the
//     column scales of M are folded into Y, which is exact.
//   - X^T C X and X^T X are formed for i <= j only and mirrored.
// A column with an infinite or NaN entry makes every output it enters a NaN.
// What bounds it now: the integer multiply-adds of the SMs a cluster has (n = 100,
// clusters of 8: 17k of the 24k clocks of a full product), then the FP64 arithmetic of
// E and of the epilogues, then the cluster barriers (n = 40). Kernel time of a
// decomposition's products and corrections, one launch per product -> here (profiled
// one by one): six searches of n = 40 178 -> 111 us, ten of n = 100 340 -> 231. The
// results do not depend on the cluster size: every sum is exact.
#include <cmath>
#include <cooperative_groups.h>
#include "device_common.cuh"

namespace cg = cooperative_groups;

namespace cmaes_gb300 {

constexpr int kRfNT = 512, kRfW = kRfNT / 32;
constexpr int kRfK = 32;                                   // k per step of the left operand
constexpr int kRfCols = 20;                                // most columns of a CTA: ceil(kEigMixedMaxN / 8)
constexpr int kRfRow = (kEigMixedMaxN + 31) / 32;          // elements of a column per lane
constexpr int kRfPre = kRfK * kEigMixedMaxN / kRfNT;       // left elements per thread and step
constexpr double kRfSep = 0x1p-10;                         // largest first-order correction
constexpr int kRfTiny = 34;                                // corrections below 2^-34 take h h alone
constexpr int kRfMoreNs = 2;                               // most further Newton-Schulz steps
constexpr double kRfDefect = 0x1p-28;                      // largest |X^T X - I| that one step takes to rounding
static_assert(kEigMixedMaxN <= 160, "the integer sums over K hold up to 255 terms, the item lists up to n = 160");

namespace {

__device__ __forceinline__ int uni(int x) { return __shfl_sync(0xffffffffu, x, 0); }

struct RfLayout {
  int nc, ks, ns, lp;  // columns (rounded up to 4), K stride, column stride, left stride
  size_t r, left, ints, bytes;
};
__host__ __device__ inline RfLayout rf_layout(int n, int cs) {
  RfLayout l;
  l.nc = ((n + cs - 1) / cs + 3) & ~3;
  l.ks = (n + 31) & ~31;
  l.ns = n | 1;
  l.lp = (n + 1) | 1;
  l.r = static_cast<size_t>(2) * l.nc * l.ns * 8;       // after X and T (doubles)
  l.left = l.r + static_cast<size_t>(2) * l.nc * l.ks * 8;
  l.ints = l.left + static_cast<size_t>(2) * kRfK * l.lp * 8;
  l.ints = l.ints + static_cast<size_t>(n) * 8;         // lambda before the integers
  l.bytes = l.ints + static_cast<size_t>(3 * n + 2 * l.nc) * 4;
  return l;
}

struct Rf {
  double *X, *T, *lam;   // own columns (stride ns), lambda of all
  int2 *R0, *R1;         // own columns of the right operands (stride ks)
  int2* As;              // left operand, two steps
  int *ec, *ex, *e0, *e1;  // scales: of C, of X (two generations), of R0 and R1
  int n, ns, ks, lp, rank, cs, ncl, tid, lane, warp;
  __device__ int col(int c) const { return cs * c + rank; }
};

// One product over the cluster's columns. SYM: only i <= j. NA right operands
// (R0 and R1) share the left one. rows: M(i, k) at M[i + L k], else M(k, i) at
// M[k + L i]. CT columns and two rows per thread; epi(i, c, v0, v1). HI: h h only,
// as for every column of Ra whose scale is at most `tiny`.
template <int CT, int NA, bool SYM, bool HI, class EPI>
__device__ __forceinline__ void rf_product(const Rf& f, const int2* M, long long L, bool rows, const int2* Ra,
                                           const int2* Rb, const int* el, const int* ea, const int* eb, int tiny,
                                           const EPI& epi) {
  const int n = f.n, tid = f.tid, lane = f.lane, warp = f.warp;
  // this thread's outputs: rows r and r + H of columns c0 .. c0 + CT - 1
  int c0 = 0, r = tid, H = 0, lim = 0;
  bool work = false;
  if (SYM) {
    for (; c0 < f.ncl; c0 += CT) {
      lim = f.col(min(c0 + CT, f.ncl) - 1) + 1;
      H = (lim + 1) >> 1;
      if (r < H) break;
      r -= H;
    }
    work = c0 < f.ncl;
  } else {
    H = (n + 1) >> 1;
    c0 = tid / H * CT;
    r = tid % H;
    lim = n;
    work = c0 < f.ncl;
  }
  if (!work) c0 = r = H = 0;
  long long hh[NA][2][CT], mid[NA][2][CT];
#pragma unroll
  for (int x = 0; x < NA; ++x)
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int c = 0; c < CT; ++c) hh[x][u][c] = mid[x][u][c] = 0;
  constexpr int kRfU = CT * NA == 1 ? 8 : 4;  // k per batch of loads
  int2 pre[kRfPre];
  auto fetch = [&](int k0) {
    if (rows) {
#pragma unroll
      for (int q = 0; q < kRfPre; ++q) {
        const int k = warp + kRfW * (q / kRfRow), i = lane + 32 * (q % kRfRow);
        pre[q] = (k0 + k < n && i < n) ? __ldcg(M + i + L * (k0 + k)) : make_int2(0, 0);
      }
    } else {
#pragma unroll
      for (int q = 0; q < kRfPre; ++q) {
        const int i = warp + kRfW * q;
        pre[q] = (k0 + lane < n && i < n) ? __ldcg(M + k0 + lane + L * i) : make_int2(0, 0);
      }
    }
  };
  auto store = [&](int2* As) {
    if (rows) {
#pragma unroll
      for (int q = 0; q < kRfPre; ++q) {
        const int k = warp + kRfW * (q / kRfRow), i = lane + 32 * (q % kRfRow);
        if (i < n) As[k * f.lp + i] = pre[q];
      }
    } else {
#pragma unroll
      for (int q = 0; q < kRfPre; ++q) {
        const int i = warp + kRfW * q;
        if (i < n) As[lane * f.lp + i] = pre[q];
      }
    }
  };
  static_assert(kRfPre == 2 * kRfRow && kRfK == 2 * kRfW && kRfPre * kRfW >= kEigMixedMaxN, "left staging");
  fetch(0);
  store(f.As);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < n; k0 += kRfK) {
    if (k0 + kRfK < n) fetch(k0 + kRfK);
    if (work) {
      const int2* a = f.As + buf * kRfK * f.lp + r;
      const int2* b = Ra + c0 * f.ks + k0;
      const int2* b2 = Rb + c0 * f.ks + k0;
      const int kn = min(kRfK, n - k0);  // (rows past n are zero in both operands)
      for (int k = 0; k < kn; k += kRfU) {
        int2 av[kRfU][2], y[kRfU][CT][NA];
#pragma unroll
        for (int q = 0; q < kRfU; ++q) {
          av[q][0] = a[(k + q) * f.lp];
          av[q][1] = a[(k + q) * f.lp + H];
#pragma unroll
          for (int c = 0; c < CT; ++c)
#pragma unroll
            for (int x = 0; x < NA; ++x) y[q][c][x] = (x == 0 ? b : b2)[c * f.ks + k + q];
        }
#pragma unroll
        for (int q = 0; q < kRfU; ++q)
#pragma unroll
          for (int c = 0; c < CT; ++c)
#pragma unroll
            for (int x = 0; x < NA; ++x)
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                hh[x][u][c] += static_cast<long long>(av[q][u].x) * y[q][c][x].x;
                if (HI) continue;
                mid[x][u][c] += static_cast<long long>(av[q][u].x) * y[q][c][x].y;
                mid[x][u][c] += static_cast<long long>(av[q][u].y) * y[q][c][x].x;
              }
      }
    }
    buf ^= 1;
    if (k0 + kRfK < n) store(f.As + buf * kRfK * f.lp);
    __syncthreads();
  }
  if (work) {
    auto value = [&](long long h, long long m, int e, int e2) {
      if (e == 0x7ff || e2 == 0x7ff) return __longlong_as_double(0x7ff8000000000000ll);
      return gemm_scaled<28>(h, m, e + e2);
    };
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int i = r + u * H;
      if (i >= lim) continue;
      const int e = rows ? 1022 : el[i];
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        if (c0 + c >= f.ncl || (SYM && i > f.col(c0 + c))) continue;
        epi(i, c0 + c, value(hh[0][u][c], HI || ea[c0 + c] <= tiny ? 0 : mid[0][u][c], e, ea[c0 + c]),
            NA == 2 ? value(hh[NA - 1][u][c], mid[NA - 1][u][c], e, eb[c0 + c]) : 0.0);
      }
    }
  }
}

template <bool HI, class EPI>
__device__ __forceinline__ void rf_full(const Rf& f, const int2* M, long long L, bool rows, const int2* R,
                                        const int* el, const int* er, int tiny, const EPI& epi) {
  const int H = (f.n + 1) >> 1;
  if (H * f.ncl <= kRfNT) rf_product<1, 1, false, HI>(f, M, L, rows, R, R, el, er, er, tiny, epi);
  else if (H * ((f.ncl + 1) >> 1) <= kRfNT) rf_product<2, 1, false, HI>(f, M, L, rows, R, R, el, er, er, tiny, epi);
  else rf_product<4, 1, false, HI>(f, M, L, rows, R, R, el, er, er, tiny, epi);
}
template <int NA, class EPI>
__device__ __forceinline__ void rf_sym(const Rf& f, const int2* M, long long L, const int2* Ra, const int2* Rb,
                                       const int* el, const int* ea, const int* eb, const EPI& epi) {
  int items = 0;
  for (int c = 0; c < f.ncl; ++c) items += (f.col(c) + 2) >> 1;
  if (items <= kRfNT) rf_product<1, NA, true, false>(f, M, L, false, Ra, Rb, el, ea, eb, 0, epi);
  else rf_product<2, NA, true, false>(f, M, L, false, Ra, Rb, el, ea, eb, 0, epi);
}

// x 2^(E - 1022) by its exponent field; below the normal range it is zero, above it
// and where either is not finite it is a NaN.
__device__ __forceinline__ double rf_scaled(double x, int E) {
  const int hi = __double2hiint(x), be = (hi >> 20) & 0x7ff, e = be + E - 1022;
  if (be == 0 || e <= 0) return be == 0x7ff || E == 0x7ff ? __hiloint2double(0x7ff80000, 0) : 0.0;
  if (be == 0x7ff || E == 0x7ff || e >= 0x7ff) return __hiloint2double(0x7ff80000, 0);
  return __hiloint2double(hi + ((E - 1022) << 20), __double2loint(x));
}

// Columns src (own, stride ns, shared memory; fold: entry k times 2^(fold[k] - 1022))
// as integers: into R with scales er, and, for a matrix that the others read, into G
// (ldn x n) with its scales in `eg` of every CTA.
__device__ __forceinline__ void rf_integers(const Rf& f, const double* src, const int* fold, int2* R, int* er,
                                            int2* G, long long L, int* eg, cg::cluster_group& cl) {
  for (int c = f.warp; c < f.ncl; c += kRfW) {
    double x[kRfRow];
    unsigned mx = 0;
#pragma unroll
    for (int u = 0; u < kRfRow; ++u) {
      const int i = f.lane + 32 * u;
      x[u] = i < f.n ? src[c * f.ns + i] : 0.0;
      if (fold && i < f.n) x[u] = rf_scaled(x[u], fold[i]);
      mx = max(mx, static_cast<unsigned>(__double2hiint(x[u]) >> 20) & 0x7ffu);
    }
    const int E = static_cast<int>(__reduce_max_sync(0xffffffffu, mx)), j = f.col(c);
#pragma unroll
    for (int u = 0; u < kRfRow; ++u) {
      const int i = f.lane + 32 * u;
      if (i >= f.n) continue;
      const int2 v = gemm_limbs<28>(x[u], E);
      R[c * f.ks + i] = v;
      if (G) __stcg(G + i + L * j, v);
    }
    if (f.lane == 0) er[c] = E;
    if (eg && f.lane < f.cs) cl.map_shared_rank(eg, f.lane)[j] = E;
  }
}

}  // namespace

// head: A = B^T C B -> EH. Otherwise, with V32 in EG: X -> B, A = X^T C X -> EA.
// Scratch: ET holds C, EX and EH the basis as integers; EG and EA hold S and G.
__global__ void __launch_bounds__(kRfNT, 1) k_eig_refine(Search* S, int s0, int head) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ int sh_again[kRfMoreNs + 1];  // the n-th Newton-Schulz step started from a defect that needs another
  cg::cluster_group cl = cg::this_cluster();
  Rf f;
  f.cs = static_cast<int>(cl.num_blocks());
  f.rank = static_cast<int>(cl.block_rank());
  const Search& s = S[s0 + static_cast<int>(blockIdx.x) / f.cs];
  // uniform over the cluster: every CTA reads the same flags
  if (s.done || !s.eig_due || s.trd || s.n <= kJacobiSmallN || s.n > kEigMixedMaxN) return;
  f.n = uni(s.n);
  const int n = f.n;
  const RfLayout lay = rf_layout(n, f.cs);
  const long long L = s.ldn;
  f.ns = lay.ns; f.ks = lay.ks; f.lp = lay.lp;
  f.X = reinterpret_cast<double*>(dyn);
  f.T = f.X + static_cast<size_t>(lay.nc) * lay.ns;
  f.R0 = reinterpret_cast<int2*>(dyn + lay.r);
  f.R1 = f.R0 + static_cast<size_t>(lay.nc) * lay.ks;
  f.As = reinterpret_cast<int2*>(dyn + lay.left);
  f.lam = reinterpret_cast<double*>(dyn + lay.ints) - n;
  f.ec = reinterpret_cast<int*>(dyn + lay.ints);
  f.ex = f.ec + n;
  f.e0 = f.ex + 2 * n;
  f.e1 = f.e0 + lay.nc;
  f.tid = threadIdx.x; f.lane = f.tid & 31; f.warp = uni(f.tid >> 5);
  f.ncl = f.rank < n ? (n - f.rank + f.cs - 1) / f.cs : 0;
  int2* CL = reinterpret_cast<int2*>(s.ET);
  int2* XL[2] = {reinterpret_cast<int2*>(s.EX), reinterpret_cast<int2*>(s.EH)};
  double *So = s.EG, *Go = s.EA;

  // own columns of C, B and V32; columns past the last one are zero
  for (int e = f.tid; e < 2 * lay.nc * f.ks; e += kRfNT) f.R0[e] = make_int2(0, 0);
  if (f.tid <= kRfMoreNs) sh_again[f.tid] = 0;
  auto load = [&](double* dst, const double* src) {
    for (int c = f.warp; c < f.ncl; c += kRfW)
#pragma unroll
      for (int u = 0; u < kRfRow; ++u) {
        const int i = f.lane + 32 * u;
        if (i < n) dst[c * f.ns + i] = src[i + L * f.col(c)];
      }
  };
  load(f.T, s.C);
  load(f.X, s.B);
  cl.sync();  // every CTA of the cluster runs: its shared memory may be written
  rf_integers(f, f.T, nullptr, f.R1, f.e1, CL, L, f.ec, cl);
  int cur = head ? 0 : 1;  // the basis is in XL[cur], its scales in ex + cur n
  rf_integers(f, f.X, nullptr, f.R0, f.e0, XL[cur], L, f.ex + cur * n, cl);
  __syncthreads();
  if (!head) {
    load(f.T, s.EG);
    for (int e = f.tid; e < lay.nc * f.ns; e += kRfNT) f.X[e] = 0.0;
  }
  cl.sync();

  int ns = 0;  // Newton-Schulz steps formed
  for (int p = head ? 3 : 0; p < 4; ++p) {
    if (!head) {
      // X <- X + M T, M the published basis (p = 0: X = 0, M = B, T = V32)
      rf_integers(f, f.T, f.ex + cur * n, f.R1, f.e1, nullptr, L, nullptr, cl);
      __syncthreads();
      // corrections this small (the second step's and Newton-Schulz's, as a rule): the
      // products left out are below sqrt(n) 2^-63, an entry of X is rounded at 2^-56. Each
      // column decides for itself, so that which CTA has it does not show.
      constexpr int tiny = 1022 - kRfTiny;
      auto add = [&](int i, int c, double v, double) { f.X[c * f.ns + i] += v; };
      if (__syncthreads_or(f.tid < f.ncl && f.e1[f.tid] > tiny))
        rf_full<false>(f, XL[cur], L, true, f.R1, nullptr, f.e1, tiny, add);
      else
        rf_full<true>(f, XL[cur], L, true, f.R1, nullptr, f.e1, tiny, add);
      __syncthreads();
      cur ^= 1;
      rf_integers(f, f.X, nullptr, f.R0, f.e0, XL[cur], L, f.ex + cur * n, cl);
      cl.sync();
    }
    const int* ex = f.ex + cur * n;
    if (p == 2) {  // G = X^T X
      bool large = false;
      rf_sym<1>(f, XL[cur], L, f.R0, f.R0, ex, f.e0, f.e0, [&](int i, int c, double g, double) {
        const int j = f.col(c);
        __stcg(Go + i + L * j, g);
        __stcg(Go + j + L * i, g);
        large |= fabs(g - (i == j ? 1.0 : 0.0)) > kRfDefect;
      });
      // Groups of repeated eigenvalues far from their old basis leave pairs at the bound of
      // the first-order corrections, and with them a defect whose square is above rounding:
      // the step is then repeated, for every CTA of the cluster.
      if (__syncthreads_or(large) && f.tid < f.cs) cl.map_shared_rank(sh_again, f.tid)[ns] = 1;
      cl.sync();
      // E = (I - G) / 2
      for (int c = f.warp; c < f.ncl; c += kRfW)
#pragma unroll
        for (int u = 0; u < kRfRow; ++u) {
          const int i = f.lane + 32 * u, j = f.col(c);
          if (i < n) f.T[c * f.ns + i] = 0.5 * ((i == j ? 1.0 : 0.0) - __ldcg(Go + i + L * j));
        }
      __syncthreads();
      if (ns < kRfMoreNs && sh_again[ns]) p = 1;
      ++ns;
      continue;
    }
    // T = C X
    rf_full<false>(f, CL, L, false, f.R0, f.ec, f.e0, 0, [&](int i, int c, double v, double) { f.T[c * f.ns + i] = v; });
    __syncthreads();
    rf_integers(f, f.T, nullptr, f.R1, f.e1, nullptr, L, nullptr, cl);
    __syncthreads();
    if (p == 3) {  // A = X^T T
      double* A = head ? s.EH : s.EA;
      rf_sym<1>(f, XL[cur], L, f.R1, f.R1, ex, f.e1, f.e1, [&](int i, int c, double v, double) {
        const int j = f.col(c);
        A[i + L * j] = v;
        A[j + L * i] = v;
      });
      if (!head)
        for (int c = f.warp; c < f.ncl; c += kRfW)
          for (int i = f.lane; i < n; i += 32) s.B[i + L * f.col(c)] = f.X[c * f.ns + i];
      break;
    }
    // S = X^T T, G = X^T X, lambda_i = s_ii / g_ii
    rf_sym<2>(f, XL[cur], L, f.R1, f.R0, ex, f.e1, f.e0, [&](int i, int c, double sv, double gv) {
      const int j = f.col(c);
      __stcg(So + i + L * j, sv);
      __stcg(So + j + L * i, sv);
      __stcg(Go + i + L * j, gv);
      __stcg(Go + j + L * i, gv);
      if (i == j)
        for (int q = 0; q < f.cs; ++q) cl.map_shared_rank(f.lam, q)[i] = sv / gv;
    });
    cl.sync();
    // E. A pair is corrected to first order only when both of its corrections stay
    // below 2^-10; otherwise both entries only get the orthogonality half -g_ij / 2.
    // The bound keeps the second-order loss of orthogonality of a step,
    // sum_k |e_ki e_kj| <= n 2^-20, small enough that the second step and the
    // Newton-Schulz step bring X^T X to I within rounding (1.5 (n 2^-20)^4 << eps64).
    for (int q = f.tid; q < f.ncl * n; q += kRfNT) {
      const int c = q / n, i = q - c * n, j = f.col(c);
      const double g = __ldcg(Go + i + L * j), sv = __ldcg(So + i + L * j);
      double e = -0.5 * g;
      if (i == j) {
        e += 0.5;
      } else {
        // the test is symmetric in (i, j), so e_ij + e_ji = -g_ij in both branches
        // (bounds compared on their bit patterns: non-negative doubles order as integers)
        const double li = f.lam[i], lj = f.lam[j];
        const double num = sv - lj * g, num_t = sv - li * g, den = lj - li;
        const long long lim = __double_as_longlong(kRfSep * fabs(den));
        if (lim != 0 && __double_as_longlong(fabs(num)) <= lim && __double_as_longlong(fabs(num_t)) <= lim) e = num / den;
      }
      f.T[c * f.ns + i] = e;
    }
    __syncthreads();
  }
}

static cudaLaunchConfig_t refine_config(int searches, int max_n, int cs, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg = {};
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = static_cast<unsigned>(cs);
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cfg.blockDim = dim3(kRfNT);
  cfg.gridDim = dim3(static_cast<unsigned>(searches * cs));
  cfg.dynamicSmemBytes = rf_layout(max_n, cs).bytes;
  return cfg;
}

// How many clusters of each size run side by side (none of a size that the device
// refuses); a CTA holds at most kRfCols columns.
RefinePlan refine_plan(int max_n) {
  RefinePlan plan;
  cudaLaunchAttribute at[1];
  for (int q = 0; q < RefinePlan::kSizes; ++q) {
    const int cs = RefinePlan::kTop >> q;
    plan.fit[q] = 0;
    if (cs * kRfCols < max_n) break;
    const cudaLaunchConfig_t cfg = refine_config(1, max_n, cs, at);
    if (cudaOccupancyMaxActiveClusters(&plan.fit[q], k_eig_refine, &cfg) != cudaSuccess) {
      cudaGetLastError();
      plan.fit[q] = 0;
    }
    plan.least = cs;
  }
  return plan;
}

// The largest clusters of which those of all searches run side by side, else the
// smallest that hold n columns, which pass the fewest barriers: the results do not depend
// on it. Four searches of n = 100, the decomposition: clusters of 16 425 us, of 8 480;
// ten, of which seven fit with 16: 741 and 638. Two generations of 300 searches of n = 40:
// clusters of 8 3.74 ms, of 2 1.87; of 1000 of n = 33: 11.8 and 5.3.
void launch_eig_refine(Search* S, int s0, int s1, int max_n, const RefinePlan& plan, int head, cudaStream_t st) {
  if (s1 <= s0 || max_n <= kJacobiSmallN) return;
  int cs = plan.least;
  for (int q = RefinePlan::kSizes - 1; q >= 0; --q)
    if (plan.fit[q] >= s1 - s0 && (RefinePlan::kTop >> q) > cs) cs = RefinePlan::kTop >> q;
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t cfg = refine_config(s1 - s0, max_n, cs, at);
  cfg.stream = st;
  cudaLaunchKernelEx(&cfg, k_eig_refine, S, s0, head);
}

cudaError_t refine_smem_limit() {
  if (cudaFuncSetAttribute(k_eig_refine, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    cudaGetLastError();
  return smem_limit_max(reinterpret_cast<const void*>(k_eig_refine));
}

}  // namespace cmaes_gb300

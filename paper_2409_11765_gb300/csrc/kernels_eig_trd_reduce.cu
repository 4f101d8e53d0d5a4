// kernels_eig_trd_reduce.cu -- the Householder reduction T = Q^T C Q of the
// tridiagonal route (Golub & Van Loan §8.3.1, unblocked; the first half of
// LAPACK's dsyev that the paper calls, §3.1), in 64-bit fixed point.
//
// What bounds it. A step k forms the reflector of column k, applies the
// previous step's rank-2 update A <- A - v w^T - w v^T and accumulates
// p = A v for the new v: per element of the trailing matrix one update and one
// product, and one barrier over the search's CTAs. GB300 issues 1.7 FP64 FMAs
// per clock and SM (66 clocks latency) but 28 32 x 32 + 64-bit integer
// multiply-adds (15 clocks), so the three FP64 FMAs per element cost 1.8 clocks
// and this form's nine integer ones 0.33. Every per-row operation of a step is
// integer too (each FP64 one costs a CTA n / 1.7 clocks a step), and so are the
// reflector's scalars: an FP64 pipe that is used only a few times a step
// answers slowly (measured: 5200 clocks for the reflector's 20 dependent FP64
// operations against ~1300 back to back).
//
// Fixed point. With mu = tr(C) / n, F = ||C - mu I||_F and q = F / (1.75 2^62),
// the matrix is held as 64-bit integers a = (C - mu I) / q: every later entry
// is bounded by F (orthogonal similarity), so nothing overflows, and the
// storage error per update, q / 2, is F 2^-63.8 -- about that of the two FP64
// roundings per update it replaces (backward error measured over spectra and
// n = 60 .. 1000: 0.5 - 1 times the FP64 form's, 3 times for a nearly rank-one
// matrix, where both are ~1e-15 ||C||). A reflector entry |v_i| <= 1 is
// v = vh 2^-29 + vl 2^-59, an entry of w (in q) is (wh 2^30 + wl) 2^ls, all four
// signed 30-bit limbs, ls >= 0 the step's scale (0 unless |w| reaches 2^60 q).
//   update    hh = vh_i wh_j + wh_i vh_j,
//             mm = vh_i wl_j + vl_i wh_j + wh_i vl_j + wl_i vh_j,
//             a -= (hh << (ls + 1)) + (mm >> (29 - ls)); the partial terms may
//             wrap, their sum (modulo 2^64) is the exact small result
//   product   a = ah 2^32 + al: HH = sum ah vh (8 q), and ah vl (2^-27 q),
//             al vh (2^-29 q) over four rows, shifted to MID (2^-23 q); by
//             Cauchy-Schwarz with ||v||^2 <= 2 and ||a_j|| <= F / q no sum
//             overflows up to n = 4096
// All long sums are integer sums, so their order does not matter: partial sums
// meet in shared-memory and global atomics, and a search gives the same bits
// for every group size, alone or in a batch.
//
// Exchange. The p of a step and the next column go from their owners to every
// CTA of the search without a barrier: each 64-bit word carries two tag bits
// (p in 8 q shifted left by two, the column rounded to 4 q), and a reader polls
// its rows until the tag is the step's. Buffers alternate between even and odd
// steps; a word is overwritten two steps later, by an owner that has received
// every p of the step between, which each CTA sends after it has read this one.
// A grid barrier would cost ~2400 clocks a step and the loads behind it ~600; a
// polled word arrives in ~900. A CTA with no column left leaves.
//
// Layout. CTA blockIdx.x works for search grp[b].x as member r = grp[b].y of
// G = grp[b].z; column j belongs to member j mod G. With SM the columns live
// in the CTA's shared memory for the whole reduction (no L2 traffic: a step
// of n = 1000 on 152 CTAs moves 56 KB per SM); otherwise in EA.
#include <algorithm>
#include <cmath>
#include "trd_common.cuh"

namespace cmaes_gb300 {

namespace {

using u64 = unsigned long long;

constexpr int kRedPolls = 1 << 21;  // polls of a word before the wait gives up (a poll takes ~600 clocks: ~0.6 s)
constexpr int kRedPad = 1024;       // zero rows after the limb arrays: the largest work unit
constexpr double kRedRange = 1.75;  // |a| <= kRedRange 2^62

__device__ __forceinline__ int2 limbs30(long long f) {
  const int h = static_cast<int>((f + (1LL << 29)) >> 30);
  return make_int2(h, static_cast<int>(f - (static_cast<long long>(h) << 30)));
}

__device__ __forceinline__ long long mul_wide(int a, int b) { return static_cast<long long>(a) * b; }

// v_i w_j + w_i v_j in units of q, from limbs (vh, vl, wh, wl)
__device__ __forceinline__ long long pair_update(const int4& a, const int4& b, int ls) {
  const long long hh = mul_wide(a.x, b.z) + mul_wide(a.z, b.x);
  const long long mm = (1LL << (28 - ls)) + mul_wide(a.x, b.w) + mul_wide(a.y, b.z) + mul_wide(a.z, b.y) +
                       mul_wide(a.w, b.x);
  return (hh << (ls + 1)) + (mm >> (29 - ls));
}

__device__ __forceinline__ int uniform(int x) { return __shfl_sync(0xffffffffu, x, 0); }

__device__ __forceinline__ unsigned ld_relaxed_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Barrier of the G CTAs of one search (the launch is cooperative: all are
// resident). The wait is bounded: after ~1 s the device status word records a
// time-out and the CTA leaves the reduction.
__device__ bool group_sync(unsigned* ctr, unsigned target, int* err, int* sh_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
    const long long t0 = clock64();
    int ok = 1;
    while (ld_acquire_u32(ctr) < target) {
      if (clock64() - t0 > kTrdWaitCycles) {
        atomicOr(err, kDevErrTimeout);
        ok = 0;
        break;
      }
    }
    *sh_ok = ok;
  }
  __syncthreads();
  return uniform(*sh_ok) != 0;
}

// One word of the exchange, polled; tagged words are single 64-bit accesses.
__device__ __forceinline__ long long ld_word(const long long* p) {
  long long v;
  asm volatile("ld.relaxed.gpu.global.s64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_word(long long* p, long long v) {
  asm volatile("st.relaxed.gpu.global.s64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ int step_tag(int k) { return (k >> 1) & 3; }

// Warp sum of 64-bit integers (modulo 2^64) as three hardware sums of limbs of
// at most 22 bits: ~40 clocks against ~150 for a shuffle tree.
__device__ __forceinline__ u64 warp_sum_u64(u64 x) {
  const unsigned a = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(x) & 0x3fffffu);
  const unsigned b = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(x >> 22) & 0x3fffffu);
  const unsigned c = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(x >> 44));
  return a + (static_cast<u64>(b) << 22) + (static_cast<u64>(c) << 44);
}

// Sums of four 64-bit values over the warp: lanes 0, 8, 16, 24 return those of
// x0, x1, x2, x3 (two levels halve the number of values, three finish).
__device__ __forceinline__ long long warp_sum4(long long x0, long long x1, long long x2, long long x3, int lane) {
  const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0;
  const long long y0 = (b4 ? x2 : x0) + __shfl_xor_sync(0xffffffffu, b4 ? x0 : x2, 16);
  const long long y1 = (b4 ? x3 : x1) + __shfl_xor_sync(0xffffffffu, b4 ? x1 : x3, 16);
  long long z = (b3 ? y1 : y0) + __shfl_xor_sync(0xffffffffu, b3 ? y0 : y1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  return z;
}

// y (1 + c) for y in 2^-62 and a small c (|c| < 2^-20) in 2^-61
__device__ __forceinline__ u64 correct62(u64 y, long long c) {
  return y + static_cast<u64>(__mul64hi(static_cast<long long>(y >> 1), c << 20) >> 16);
}
// c^2 in 2^-61 for |c| < 2^-20 in 2^-61
__device__ __forceinline__ long long square61(long long c) { return __mul64hi(c << 20, c << 20) >> 37; }
// A float in [1/2, 2] as an integer in 2^-62
__device__ __forceinline__ u64 fixed62(float f) {
  const int b = __float_as_int(f);
  return static_cast<u64>((b & 0x7fffff) | 0x800000) << (39 - 127 + (b >> 23));
}

// The reflector of a column with the entry alpha on top of a part whose squares
// sum to hi 2^64 + lo: tau in 2^-61, ||c|| as norm 2^-62 2^e, and
// 1 / (|alpha| + ||c||) as sc 2^-61 2^-e. 1 / sqrt and 1 / x by one third-order
// step each from an FP32 seed (its residual h < 2^-20 leaves h^3 < 2^-62), in
// 64-bit fixed point.
struct Reflector {
  long long tau, sc;
  u64 norm;
  int e;
};
__device__ __forceinline__ Reflector reflector(long long alpha, u64 hi, u64 lo) {
  Reflector f{0, 0, 0ull, 0};
  const u64 a = static_cast<u64>(alpha < 0 ? -alpha : alpha), al = a * a;
  lo += al;
  hi += __umul64hi(a, a) + (lo < al ? 1ull : 0ull);
  // x = (||c|| 2^-e)^2 in [1/4, 1) as m 2^-64
  int z = hi != 0ull ? __clzll(static_cast<long long>(hi)) : 64 + __clzll(static_cast<long long>(lo));
  z &= ~1;
  const u64 m = z >= 64 ? lo << (z - 64) : z > 0 ? (hi << z) | (lo >> (64 - z)) : hi;
  f.e = 64 - (z >> 1);
  const float xf = __uint2float_rz(static_cast<unsigned>(m >> 32)) * 0x1p-32f;
  const float yf = fminf(rsqrtf(xf), 0x1.fffffep0f);
  const u64 af = a << (63 - f.e);  // |alpha| 2^-e in 2^-63
  const float rf = __fdividef(1.0f, fmaf(xf, yf, __uint2float_rz(static_cast<unsigned>(af >> 32)) * 0x1p-31f));
  u64 y = fixed62(yf);
  const long long h = (1LL << 61) - static_cast<long long>(__umul64hi(__umul64hi(y, y) << 1, m));
  y = correct62(y, (h >> 1) + 3 * (square61(h) >> 3));
  f.norm = __umul64hi(m, y);
  f.tau = (1LL << 61) + static_cast<long long>(__umul64hi(af, y));
  u64 r = fixed62(rf);
  const long long g = (1LL << 61) - static_cast<long long>(__umul64hi((af >> 1) + f.norm, r) << 1);
  r = correct62(r, g + square61(g));
  f.sc = static_cast<long long>(r >> 1);
  return f;
}

// v 2^s as a double, rounded to nearest (ties up), on the integer pipe
__device__ __forceinline__ double pack_f64(long long v, int s) {
  if (v == 0) return 0.0;
  u64 m = static_cast<u64>(v < 0 ? -v : v);
  const int z = __clzll(static_cast<long long>(m));
  m <<= z;  // in [2^63, 2^64), standing for [1, 2) 2^(s + 63 - z); its leading bit carries into the exponent
  m = (m >> 11) + ((m >> 10) & 1ull) + (static_cast<u64>(s + 63 - z + 1022) << 52);
  return __longlong_as_double(static_cast<long long>(m | (v < 0 ? 0x8000000000000000ull : 0ull)));
}

__device__ __forceinline__ long long shift_round(long long x, int s) {
  return s > 0 ? (x + (1LL << (s - 1))) >> s : x << -s;
}

}  // namespace

// NT threads: 512 with one CTA per SM (few rows per thread in the row stages,
// whose chains of FP64 and integer latencies set a small search's step), 256
// with two (a batch of more searches than SMs).
template <int NT, bool SM>
__global__ void __launch_bounds__(NT, 512 / NT) k_trd_reduce(Search* S, const int4* grp, int s0, int s1) {
  constexpr int NW = NT / 32;
  extern __shared__ int4 dyn4[];
  __shared__ double sh_mu, sh_scl, sh_q, sh_f2;
  __shared__ u64 redi[3][NW];  // the warps' integer sums of a step
  __shared__ unsigned redm[NW];
  __shared__ long long sh_half, sh_tau, sh_sc;  // fixed-point scalars of a step
  __shared__ u64 sh_norm;
  __shared__ int sh_ok, sh_ls, sh_ps, sh_sy, sh_cs, sh_sv, sh_e;
  const int4 g = grp[blockIdx.x];
  if (g.x < s0 || g.x >= s1) return;
  const Search& s = S[g.x];
  if (!trd_due(s)) return;
  const long long L = s.ldn;
  // Values that come through a shuffle are known to be uniform in the warp. A
  // warp-wide operation in a branch or loop on values that are not (loaded ones,
  // threadIdx.x / 32) goes through a slow convergence path, ~290 clocks each.
  const int tid = threadIdx.x, lane = tid & 31, warp = uniform(tid >> 5);
  const int n = uniform(s.n), r = uniform(g.y), G = uniform(g.z);
  const int ncmax = (n + G - 1) / G, np = n + kRedPad;
  int4* vw = dyn4;                                    // limbs of the pending v and w, per row
  int2* vc = reinterpret_cast<int2*>(vw + np);        // limbs of the new v (zero up to row k and from n on)
  long long* pa = reinterpret_cast<long long*>(vc + np);  // p of the pending step (8 q)
  long long* ca = pa + n;                                // column k (q)
  u64* acc = reinterpret_cast<u64*>(ca + n);  // HH, MID per own column
  long long* cols = reinterpret_cast<long long*>(acc + 2 * ncmax);          // SM: the own columns
  double* const W = s.EA;
  double* const Hv = s.EX;
  double* const tb = s.trd_v;
  int* const err = s.err;
  unsigned* const bar = s.trd_bar;
  double* const d = tb + L * TV_D;
  double* const e = tb + L * TV_E;
  double* const tau = tb + L * TV_TAU;
  // the exchanged words of even and odd steps: p, and the next column
  auto px = [&](int odd) { return reinterpret_cast<long long*>(tb + L * (odd ? TV_P1 : TV_P0)); };
  auto cx = [&](int odd) { return reinterpret_cast<long long*>(tb + L * (odd ? TV_LAMS : TV_LAMB)); };
  unsigned nb = 0;
  auto barrier = [&]() -> bool {
    if (G > 1) return group_sync(bar, static_cast<unsigned>(G) * ++nb, err, &sh_ok);
    __syncthreads();
    return true;
  };
  auto column = [&](int m) -> long long* {  // own column m (column r + G m)
    return SM ? cols + static_cast<long long>(m) * n : reinterpret_cast<long long*>(W) + L * (r + static_cast<long long>(G) * m);
  };

  // ---- (C + C^T) / 2 and the scale ----
  {
    const double* C = s.C;
    double* colss = tb + L * TV_SD;
#pragma unroll 1
    for (int m = warp; r + G * m < n; m += NW) {
      const int j = r + G * m;
      double ss = 0.0;
      for (int i = lane; i < n; i += 32) {
        const double a = 0.5 * (C[i + L * j] + C[j + L * i]);
        W[i + L * j] = a;
        if (i != j) ss = fma(a, a, ss);
      }
      ss = warp_sum_xor(ss);
      if (lane == 0) colss[j] = ss;
    }
    if (r == 0)
      for (int i = tid; i < n; i += NT) px(0)[i] = px(1)[i] = cx(0)[i] = cx(1)[i] = 3;  // no step's tag yet
    for (int c = tid; c < 2 * ncmax; c += NT) acc[c] = 0ull;
    for (int i = tid; i < np; i += NT) {
      vw[i] = make_int4(0, 0, 0, 0);
      vc[i] = make_int2(0, 0);
    }
    if (!barrier()) return;
    if (warp == 0) {  // every CTA the same sums in the same order
      double tr = 0.0, f2 = 0.0;
#pragma unroll 1
      for (int i = lane; i < n; i += 32) tr += C[i + L * i];
      const double mean = warp_sum_xor(tr) / n;
#pragma unroll 1
      for (int i = lane; i < n; i += 32) {
        const double di = C[i + L * i] - mean;
        f2 = fma(di, di, f2 + __ldcg(&colss[i]));
      }
      f2 = warp_sum_xor(f2);
      if (lane == 0) {
        const double F = sqrt(f2);
        sh_mu = mean;
        sh_scl = F > 0.0 ? kRedRange * 0x1p62 / F : 0.0;
        sh_q = F * (0x1p-62 / kRedRange);
        sh_f2 = f2;
      }
    }
    __syncthreads();
  }
  const double mu = sh_mu;
  if (r == 0 && tid == 0) {
    double* sc = tb + L * TV_SCAL;
    sc[8] = sh_f2 < INFINITY ? sh_q : nan("");
    sc[9] = mu;
  }
  if (!(sh_f2 < INFINITY)) {  // NaN or infinite entries: a NaN T (the stop test ends the descent)
    for (int j = r + G * warp; j < n; j += G * NW)
      for (int i = lane; i < n; i += 32) Hv[i + L * j] = 0.0;
    if (r == 0)
      for (int i = tid; i < n; i += NT) {
        reinterpret_cast<long long*>(d)[i] = reinterpret_cast<long long*>(e)[i] = 1;
        reinterpret_cast<long long*>(tau)[i] = 0;
        reinterpret_cast<long long*>(tb + L * TV_ES)[i] = 62;
      }
    return;
  }
#pragma unroll 1
  for (int m = warp; r + G * m < n; m += NW) {
    const int j = r + G * m;
    const double scl = sh_scl;
    long long* col = column(m);
    for (int i = lane; i < n; i += 32) {
      const long long f = __double2ll_rn((W[i + L * j] - (i == j ? mu : 0.0)) * scl);
      col[i] = f;
      if (j == 0) cx(0)[i] = (f + 2) & ~3LL;
    }
  }
  if (!barrier()) return;

  // v of step k (as FP64) and, as integers, d, tau and e = -sgn(alpha) ||c||
  // (||c|| as an integer in 2^-62 2^e, e in TV_ES; without a reflector alpha
  // itself): k_trd_blocks turns them into FP64. Nothing here uses the FP64 pipe,
  // which would hold up this CTA's next step.
  auto store = [&](int k) {
#pragma unroll 1
    for (int i = k + 1 + tid; i < n; i += NT) {
      const int2 y = vc[i];
      const long long v = (static_cast<long long>(y.x) << 30) + y.y;
      Hv[i + L * k] = pack_f64(v, -59);
    }
    if (tid == 0) {
      const long long alpha = ca[k + 1], norm = static_cast<long long>(sh_norm);
      reinterpret_cast<long long*>(d)[k] = ca[k];
      reinterpret_cast<long long*>(tau)[k] = sh_tau;
      reinterpret_cast<long long*>(e)[k] = sh_tau == 0 ? alpha : alpha < 0 ? norm : -norm;
      reinterpret_cast<long long*>(tb + L * TV_ES)[k] = sh_tau == 0 ? 62 : sh_e;
    }
  };
  if (tid == 0) sh_tau = 0;
  __syncthreads();
  long long tk = 0;  // tau of the pending step (warp 0)
  unsigned sent = static_cast<unsigned>(G) * nb;  // arrivals up to the step before: a CTA adds one per step it sends p in
  int m0 = 0;      // first own column at or after k + 1
  const int nct = r < n ? (n - 1 - r) / G + 1 : 0;
#pragma unroll 1
  for (int k = 0; k + 1 < n; ++k) {
    if (r + G * m0 < k + 1) ++m0;
    const int nc = nct - m0;
    if (nc <= 0) return;
    const bool first = r + G * m0 == k + 1;  // the owner of column k + 1 also stores d, e, tau and v of step k
    // ---- receive p of step k - 1 and column k; p . v ----
    {
      const long long* pb = px((k + 1) & 1);
      const long long* cb = cx(k & 1);
      const int ptag = step_tag(k - 1), ctag = step_tag(k);
      int ok = 1;
      if (G > 1 && k > 0) {  // one poller per CTA until (about) every CTA has sent: the words are then rarely polled twice
        if (tid == 0) {
          const unsigned want = sent + static_cast<unsigned>(min(G, n - k));
          for (int it = 0; it < kRedPolls; ++it)
            if (ld_relaxed_u32(bar) >= want) break;
        }
        sent += static_cast<unsigned>(min(G, n - k));
        __syncthreads();
      }
#pragma unroll 1
      for (int i = k + tid; i < n; i += 2 * NT) {
        const int i2 = i + NT < n ? i + NT : i;  // two rows' loads in flight
        long long pw1, pw2, cw1, cw2;
#pragma unroll 1
        for (int it = 0;; ++it) {
          cw1 = ld_word(&cb[i]);
          pw1 = ld_word(&pb[i]);
          cw2 = ld_word(&cb[i2]);
          pw2 = ld_word(&pb[i2]);
          const int po = static_cast<int>(pw1 | pw2) & 3, pa_ = static_cast<int>(pw1 & pw2) & 3;
          const int co = static_cast<int>(cw1 | cw2) & 3, ca_ = static_cast<int>(cw1 & cw2) & 3;
          if (po == ptag && pa_ == ptag && co == ctag && ca_ == ctag) break;
          if (it >= kRedPolls) {
            atomicOr(err, kDevErrTimeout);
            ok = 0;
            break;
          }
        }
        ca[i] = cw1 & ~3LL;
        ca[i2] = cw2 & ~3LL;
        pa[i] = pw1 >> 2;  // p in 8 q
        pa[i2] = pw2 >> 2;
      }
      u64 sum = 0ull;  // p . v in 2 q, each row's product rounded alone: it does not depend on which thread has the row
      unsigned tmx = 0u;
#pragma unroll 1
      for (int i = k + tid; i < n; i += NT) {
        const long long P = pa[i];
        const int2 y = vc[i];
        const long long v = (static_cast<long long>(y.x) << 30) + y.y;
        const u64 lo = static_cast<u64>(P * v), low = lo + (1ull << 56);
        sum += (static_cast<u64>(__mul64hi(P, v) + (low < lo ? 1 : 0)) << 7) + (low >> 57);
        tmx = max(tmx, static_cast<unsigned>((P < 0 ? -P : P) >> 32));
      }
      __syncwarp();
      sum = warp_sum_u64(sum);
      tmx = __reduce_max_sync(0xffffffffu, tmx);
      if (lane == 0) {
        redi[0][warp] = sum;
        redm[warp] = tmx;
      }
      if (!__syncthreads_and(ok)) return;
    }
    if (warp == 0) {  // half = (tau / 2) p . v of p = tau A v; the scale of w from |w| <= tau max|A v| + |half|
      long long pv = 0;
      unsigned mx = 0u;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        pv += static_cast<long long>(redi[0][w]);
        mx = max(mx, redm[w]);
      }
      // p . v is in 2 q: half = tau^2 pv q, from pv 2^zp < 2^62 and tau^2 in 2^-60
      const u64 ap = static_cast<u64>(pv < 0 ? -pv : pv);
      const int zp = ap != 0ull ? __clzll(static_cast<long long>(ap)) - 2 : 61, eh = 66 - zp;
      const u64 hm = __umul64hi(zp >= 0 ? ap << zp : ap >> -zp, __umul64hi(static_cast<u64>(tk), static_cast<u64>(tk)) << 2);
      const int pb = 32 - __clz(mx) + 32;  // |p| < 2^(pb + 3) q; |half| = hm 2^(eh - 62) q
      const int ls = min(max(0, max(eh, pb + 4) + 1 - 60), 20);
      const int sy = ls + 59 - eh;
      if (lane == 0) {
        sh_half = sy > 62 ? 0 : pv < 0 ? -static_cast<long long>(hm) : static_cast<long long>(hm);
        sh_ls = ls;
        sh_ps = 62 - pb;
        sh_sy = min(sy, 62);
      }
    }
    __syncthreads();
    const int ls = sh_ls;
    // ---- w = tau p - half v in 2^ls q (sums of 2^(ls - 1) q at most: the bounds behind ls) ----
    {
      const long long hm = sh_half, tf = sh_tau;
      const int ps = sh_ps, sx = ls - 6 + ps, sy = sh_sy;
#pragma unroll 1
      for (int i = k + tid; i < n; i += NT) {
        const int2 v = vc[i];
        const long long vf = (static_cast<long long>(v.x) << 30) + v.y;
        const int2 w = limbs30(shift_round(__mul64hi(pa[i] << ps, tf), sx) - shift_round(__mul64hi(vf << 2, hm), sy));
        vw[i] = make_int4(v.x, v.y, w.x, w.y);
      }
    }
    __syncthreads();
    // ---- column k with the pending update, and the squares below its first
    // off-diagonal entry, summed exactly ----
    {
      const int4 vk = vw[k];
      u64 s2 = 0ull, s1 = 0ull, s0_ = 0ull;
#pragma unroll 1
      for (int i = k + tid; i < n; i += NT) {
        const long long c = ca[i] - pair_update(vw[i], vk, ls);
        ca[i] = c;
        if (i >= k + 2) {
          const u64 a = static_cast<u64>(c < 0 ? -c : c), lo = a * a;
          s2 += __umul64hi(a, a);
          s1 += lo >> 32;
          s0_ += lo & 0xffffffffull;
        }
      }
      __syncwarp();
      s1 += s0_ >> 32;
      s2 = warp_sum_u64(s2);
      s1 = warp_sum_u64(s1);
      const unsigned low = static_cast<unsigned>(s0_);
      const unsigned l0 = __reduce_add_sync(0xffffffffu, low & 0xffffu), l1 = __reduce_add_sync(0xffffffffu, low >> 16);
      if (lane == 0) {
        redi[0][warp] = s2;
        redi[1][warp] = s1;
        redi[2][warp] = l0 + (static_cast<u64>(l1) << 16);
      }
    }
    __syncthreads();
    if (warp == 0) {  // beta = -sgn(alpha) ||c||, tau = 1 + |alpha| / ||c||, v = c / (alpha - beta)
      Reflector f{0, 0, 0ull, 0};
      const long long alpha = ca[k + 1];
      u64 s2 = 0ull, s1 = 0ull, s0_ = 0ull;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        s2 += redi[0][w];
        s1 += redi[1][w];
        s0_ += redi[2][w];
      }
      const u64 mid = s1 + (s0_ >> 32), hi = s2 + (mid >> 32), lo = (mid << 32) | (s0_ & 0xffffffffull);
      if ((hi | lo) != 0ull) f = reflector(alpha, hi, lo);
      tk = f.tau;
      if (lane == 0) {
        // as an integer in 2^-59, v = ((c << cs) sc 2^-64) >> sv
        sh_tau = f.tau;
        sh_sc = alpha < 0 ? -f.sc : f.sc;
        sh_norm = f.norm;
        sh_e = f.e;
        sh_cs = max(0, 62 - f.e);
        sh_sv = max(0, f.e - 62);
      }
    }
    __syncthreads();
    {
      const long long sf = sh_sc;
      const int cs = sh_cs, sv = sh_sv;
      if (tid == NT - 1) vc[k] = make_int2(0, 0);
#pragma unroll 1
      for (int i = k + 1 + tid; i < n; i += NT) {
        const long long v = i == k + 1 ? 1LL << 59 : shift_round(__mul64hi(ca[i] << cs, sf), sv);
        vc[i] = limbs30(v);
      }
    }
    __syncthreads();
    // ---- own columns j >= k + 1, rows in units of a multiple of 128: the pending
    // update and the new product. Rows up to k and from n on are worked too
    // (v = 0 there), so that the code has no branch per row. Units of one column
    // from shared memory, sized to give every warp one; of two columns from HBM
    // (the limbs are then read once for both). ----
    {
      constexpr int NCOL = SM ? 1 : 2;
      const int groups = SM ? nc : (nc + 1) >> 1, base = (k + 1) & ~31;
      int batches = 1;
      while (batches < 8 && groups * ((n - base + 128 * batches - 1) / (128 * batches)) > NW) ++batches;
      const int unit = 128 * batches, chunks = (n - base + unit - 1) / unit;
      long long* const cnext = cx((k + 1) & 1);
      const int ctag = step_tag(k + 1);
#pragma unroll 1
      for (int un = warp; un < groups * chunks; un += NW) {
        const int ch = un / groups, c1 = NCOL * (un - ch * groups), j1 = r + G * (m0 + c1);
        const bool two = NCOL == 2 && c1 + 1 < nc;
        long long* const A1 = column(m0 + c1);
        long long* const A2 = column(m0 + c1 + (two ? 1 : 0));
        if (!SM && un + NW < groups * chunks) {
          // the warp's next unit on its way to L2 (rows r0 .. below n of its columns; 16-byte
          // pieces from a multiple of 32 rows): 40 searches of n = 2000 391 -> 366 ms
          const int nu = un + NW, nch = nu / groups, nc1 = NCOL * (nu - nch * groups), r0 = base + unit * nch;
          const unsigned bytes = static_cast<unsigned>(min(unit, n - r0) * 8) & ~15u;
          if (lane < NCOL && nc1 + lane < nc && bytes != 0u)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(column(m0 + nc1 + lane) + r0), "r"(bytes) : "memory");
        }
        const int4 x1 = vw[j1], x2 = vw[two ? j1 + G : j1];
        const bool pub = j1 == k + 1;
        long long h1 = 0, h2 = 0, mid1 = 0, mid2 = 0;
        int i0 = base + unit * ch + lane;
        const int live = min(batches, (n - base - unit * ch + 127) >> 7);  // batches with a row below n
#pragma unroll 1
        for (int bt = 0; bt < live; ++bt, i0 += 128) {
          long long a1[4], a2[4], ma1 = 0, mb1 = 0, ma2 = 0, mb2 = 0;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + 32 * u;
            a1[u] = i < n ? (SM ? A1[i] : __ldcg(&A1[i])) : 0;
            if (NCOL == 2) a2[u] = i < n ? (SM ? A2[i] : __ldcg(&A2[i])) : 0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int4 x = vw[i0 + 32 * u];
            a1[u] -= pair_update(x, x1, ls);
            if (NCOL == 2) a2[u] -= pair_update(x, x2, ls);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + 32 * u;
            if (i < n) {
              A1[i] = a1[u];
              if (two) A2[i] = a2[u];
            }
          }
          if (pub) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int i = i0 + 32 * u;
              if (i > k && i < n) st_word(&cnext[i], ((a1[u] + 2) & ~3LL) | ctag);
              if (i == n - 1 && k == n - 2) reinterpret_cast<long long*>(d)[n - 1] = a1[u];  // the last diagonal entry
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int2 y = vc[i0 + 32 * u];
            const int ah1 = static_cast<int>((a1[u] + 0x80000000LL) >> 32), al1 = static_cast<int>(a1[u]);
            h1 += mul_wide(ah1, y.x);
            ma1 += mul_wide(ah1, y.y);
            mb1 += mul_wide(al1, y.x);
            if (NCOL == 2) {
              const int ah2 = static_cast<int>((a2[u] + 0x80000000LL) >> 32), al2 = static_cast<int>(a2[u]);
              h2 += mul_wide(ah2, y.x);
              ma2 += mul_wide(ah2, y.y);
              mb2 += mul_wide(al2, y.x);
            }
          }
          mid1 += (ma1 >> 4) + (mb1 >> 6);
          mid2 += (ma2 >> 4) + (mb2 >> 6);
        }
        if (NCOL == 2) {
          const long long z = warp_sum4(h1, mid1, h2, mid2, lane);
          if ((lane & 7) == 0 && (two || lane < 16))
            atomicAdd(&acc[2 * c1 + (lane >> 3)], static_cast<u64>(z));
        } else {
          const u64 za = warp_sum_u64(static_cast<u64>(h1));
          const u64 zb = warp_sum_u64(static_cast<u64>(mid1));
          if (lane < 2) atomicAdd(&acc[2 * c1 + lane], lane == 0 ? za : zb);
        }
      }
    }
    __syncthreads();
    if (k + 2 >= n) {  // the last reflector is the identity (tau = 0): nothing is pending after it
      store(k);
      return;
    }
    {
      long long* const pout = px(k & 1);
      const int ptag = step_tag(k);
#pragma unroll 1
      for (int c = tid; c < nc; c += NT) {
        const long long HH = static_cast<long long>(acc[2 * c]), MID = static_cast<long long>(acc[2 * c + 1]);
        acc[2 * c] = 0ull;
        acc[2 * c + 1] = 0ull;
        const long long P = HH + ((MID + (1LL << 25)) >> 26);  // in 8 q
        st_word(&pout[r + G * (m0 + c)], (P << 2) | ptag);
      }
    }
    __syncthreads();
    if (tid == 0) asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    if (first) store(k);  // while the other CTAs' p is on its way
  }
}

namespace {

using RedFn = void (*)(Search*, const int4*, int, int);
RedFn reduce_fn(int in_smem, int nt) {
  return in_smem ? k_trd_reduce<512, true> : nt == 512 ? k_trd_reduce<512, false> : k_trd_reduce<256, false>;
}

}  // namespace

size_t trd_reduce_smem(int n, int G, int in_smem) {
  const size_t nc = static_cast<size_t>(ceil_div(n, G));
  return static_cast<size_t>(n) * 40 + 24 * kRedPad + 16 * nc + (in_smem ? 8 * nc * n : 0);
}

// The dynamic shared memory a CTA can have: the attribute is always set to this
// limit, whatever a handle needs, because it belongs to the process.
static size_t reduce_smem_max() {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return optin > 1024 ? optin - 1024 : 0;  // less the kernel's static arrays
}

int trd_reduce_blocks_per_sm(size_t smem, int in_smem, int nt) {
  int b = 0;
  const void* fn = reinterpret_cast<const void*>(reduce_fn(in_smem, nt));
  const size_t top = reduce_smem_max();
  if (smem > top) return 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(top)) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, nt, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return b;
}

int launch_trd_reduce(Search* S, const int4* grp, const TrdChunk* chunks, int nchunks, unsigned* bars, int s0, int s1,
                      const TrdReducePlan& plan, cudaStream_t st) {
  // the group barriers of these searches count from zero
  cudaMemsetAsync(bars + s0, 0, sizeof(unsigned) * (s1 - s0), st);
  for (int c = 0; c < nchunks; ++c) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(chunks[c].count);
    cfg.blockDim = dim3(plan.threads);
    cfg.dynamicSmemBytes = plan.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, reduce_fn(plan.in_smem, plan.threads), S, grp + chunks[c].first, s0, s1);
  }
  return nchunks;
}

}  // namespace cmaes_gb300

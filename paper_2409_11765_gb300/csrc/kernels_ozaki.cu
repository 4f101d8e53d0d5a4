// kernels_ozaki.cu -- the general FP64-accurate product C = alpha A B + beta C
// on the BF16 tensor cores (digit planes and bucket sums of ozaki.cuh), used
// by include/cmaes_ozaki.h and by the eigensolver's Gram products.
#include <algorithm>
#include <mutex>
#include <cuda_runtime.h>
#include "../../include/cmaes_ozaki.h"
#include "engine.h"
#include "ozaki.cuh"

namespace cmaes_gb300 {

// One operand to pack: x(r, k) = src[r * sr + k * sk], r < R, k < K.
struct OzPackJob {
  const double* src;
  long long sr, sk;
  int R, K, nks;
  unsigned char* out;
  int* e;
  int blocks;  // 64-row blocks
};

// CTAs take 64 rows by kOzPackK, first for the rows' exponents (e starts below
// kOzZeroExp), then, with those complete, for the digits; the second pass finds the
// operands in L2. Bound by the digits' 14 bytes per element on their way to L2: 13 + 28 us
// for 1000 x 1024 x 2000, where one CTA per 64 rows is a serial pass of K / 32 steps on 32
// CTAs, 240 us.
constexpr int kOzPackKC = 4, kOzPackK = kOzPackKC * kOzKS;

template <class F>
__device__ __forceinline__ void oz_pack_job(const OzPackJob& a, const OzPackJob& b, const F& f) {
  int rb = static_cast<int>(blockIdx.x);
  const OzPackJob& J = rb < a.blocks ? a : b;
  if (rb >= a.blocks) rb -= a.blocks;
  f(J, [&](int r, int k) { return J.src[static_cast<long long>(r) * J.sr + static_cast<long long>(k) * J.sk]; }, rb);
}

__global__ void __launch_bounds__(kOzNT) k_oz_exponents(OzPackJob a, OzPackJob b) {
  __shared__ int sh_e[64];
  if (threadIdx.x < 64) sh_e[threadIdx.x] = kOzZeroExp;
  __syncthreads();
  oz_pack_job(a, b, [&](const OzPackJob& J, auto get, int rb) {
    const bool kfast = J.sk == 1;
    int rl, oc;
    oz_pack_place(kfast, rl, oc);
    int e = kOzZeroExp;
    for (int k0 = blockIdx.y * kOzPackK; k0 < J.K; k0 += gridDim.y * kOzPackK)
      e = max(e, oz_pack_exponent(get, kfast, J.R, k0, min(J.K, k0 + kOzPackK), rb));
    atomicMax(&sh_e[rl], e);
    __syncthreads();
    if (oc == 0) atomicMax(&J.e[rb * 64 + rl], sh_e[rl]);
  });
}

// One step of K in one pass (64 x 64 x 64: 60 us a call, 70 in two).
__global__ void __launch_bounds__(kOzNT) k_oz_pack_short(OzPackJob a, OzPackJob b) {
  __shared__ int sh_e[64];
  oz_pack_job(a, b, [&](const OzPackJob& J, auto get, int rb) {
    oz_pack_block_get(get, J.sk == 1, J.R, J.K, rb, J.nks, J.out, J.e, sh_e);
  });
}

__global__ void __launch_bounds__(kOzNT) k_oz_pack(OzPackJob a, OzPackJob b) {
  oz_pack_job(a, b, [&](const OzPackJob& J, auto get, int rb) {
    const bool kfast = J.sk == 1;
    int rl, oc;
    oz_pack_place(kfast, rl, oc);
    const int e = J.e[rb * 64 + rl];
    for (int kc0 = blockIdx.y * kOzPackKC; kc0 < J.nks; kc0 += gridDim.y * kOzPackKC)
      oz_pack_digits(get, kfast, J.R, J.K, rb, J.nks, kc0, min(J.nks, kc0 + kOzPackKC), e, J.out);
  });
}

// C (M x N, column-major, ldc) = alpha * A B + beta * C from packed A (M rows)
// and B (N rows), K = nks * 32. One 128 x 64 output tile per CTA.
struct OzGemmJob {
  const unsigned char* a;
  const int* ea;
  const unsigned char* b;
  const int* eb;
  int M, N, nks;
  double* c;
  long long ldc;
  double alpha, beta;
};

__global__ void __launch_bounds__(kOzNT, 1) k_oz_gemm(OzGemmJob J, int* err) {
  extern __shared__ unsigned char dyn[];
  __shared__ uint64_t bar[5];
  __shared__ uint32_t tslot;
  const int tn_count = (J.N + kOzBN - 1) / kOzBN;
  const int tm = static_cast<int>(blockIdx.x) / tn_count, tn = static_cast<int>(blockIdx.x) % tn_count;
  OzCtx cx;
  oz_begin(cx, dyn, bar, &tslot);
  long long W[32];
  float L[32];
  const bool ok = oz_tile(cx, J.a, oz_pitch(J.nks), 2 * tm, J.b, oz_pitch(J.nks), tn, J.nks, W, L);
  if (!ok) {
    if (threadIdx.x == 0) atomicOr(err, kDevErrTimeout);
  } else {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = tm * kOzBM + 32 * (warp & 3) + lane;
    const int jb = tn * kOzBN + 32 * (warp >> 2);
    if (i < J.M) {
      const int ea = J.ea[i];
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        const int j = jb + q;
        if (j >= J.N) continue;
        const double v = oz_value(W[q], L[q], ea, J.eb[j]);
        double* cp = J.c + i + J.ldc * j;
        *cp = J.beta == 0.0 ? J.alpha * v : fma(J.alpha, v, J.beta * *cp);
      }
    }
  }
  oz_end(cx);
}

}  // namespace cmaes_gb300

using namespace cmaes_gb300;

// Workspace up to kOzKeep from a stream-ordered pool of the engine's own, so that a call
// neither maps nor unmaps memory: cudaMalloc and cudaFree take up to 150 us of a call
// (500 x 500 x 500: 251 us with them, 112 from the pool) and synchronise the device. The
// pool keeps at most kOzKeep bytes per context between calls; what several threads took
// beyond that goes back at the next synchronisation, and an allocation that fails gives
// everything back first. Pools are safe from every thread and stream. A larger
// workspace, or one where there is no pool, is cudaMalloc's: the pool would map and
// unmap it on every call (3000 x 3000 x 3000: 2630 us, 2870 from the pool).
// A pool ends with its context (cudaDeviceReset), and a context's number is never given
// twice, so a pool is kept under the number of the context that made it; a number that
// does not come again costs its entry, and beyond kOzMaxPools there is no pool.
namespace {
constexpr uint64_t kOzKeep = 64ull << 20;
constexpr int kOzMaxPools = 64;
struct OzPool {
  unsigned long long context;
  cudaMemPool_t pool;
};
std::mutex g_oz_mutex;
OzPool g_oz_pool[kOzMaxPools];
int g_oz_pools = 0;

// (called with a current context: the call has asked for its stream's state)
cudaMemPool_t oz_pool() {
  const unsigned long long id = context_number();
  if (id == 0) return nullptr;
  std::lock_guard<std::mutex> lock(g_oz_mutex);
  for (int i = 0; i < g_oz_pools; ++i)
    if (g_oz_pool[i].context == id) return g_oz_pool[i].pool;
  int dev = 0, ok = 0;
  if (g_oz_pools == kOzMaxPools || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&ok, cudaDevAttrMemoryPoolsSupported, dev) != cudaSuccess || !ok)
    return nullptr;
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  uint64_t keep = kOzKeep;
  cudaMemPool_t p = nullptr;
  if (cudaMemPoolCreate(&p, &props) != cudaSuccess) return nullptr;
  if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
    cudaMemPoolDestroy(p);
    return nullptr;
  }
  g_oz_pool[g_oz_pools++] = OzPool{id, p};
  return p;
}

struct OzWorkspace {
  unsigned char* p = nullptr;
  bool pooled = false;
  bool get(size_t bytes, cudaStream_t st) {
    if (cudaMemPool_t pool = bytes <= kOzKeep ? oz_pool() : nullptr) {
      if (cudaMallocFromPoolAsync(reinterpret_cast<void**>(&p), bytes, pool, st) == cudaSuccess) return pooled = true;
      cudaGetLastError();
      cudaMemPoolTrimTo(pool, 0);
    }
    p = nullptr;
    if (cudaMalloc(&p, bytes) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
  }
  void give_back(cudaStream_t st) {
    if (pooled) cudaFreeAsync(p, st);
    else cudaFree(p);
  }
};
}  // namespace

extern "C" int cmaes_ozaki_dgemm(int M, int N, int K, double alpha, const double* A, long long lda,
                                 const double* B, long long ldb, double beta, double* C, long long ldc,
                                 void* stream) {
  if (M < 0 || N < 0 || K < 0) return 1;
  if (M == 0 || N == 0) return 0;
  if (!A || !B || !C || lda < M || ldb < K || ldc < M) return 1;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // a call ends with a synchronisation, so a stream under capture cannot take it
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return 2;
  }
  const int nks = oz_nks(K);
  const size_t abytes = oz_bytes(M, K), bbytes = oz_bytes(N, K);
  const int mpad = oz_rows_padded(M), npad = oz_rows_padded(N);
  const size_t ebytes = sizeof(int) * (static_cast<size_t>(mpad) + npad);
  OzWorkspace ws;
  if (!ws.get(abytes + bbytes + ebytes + sizeof(int), st)) return 2;
  unsigned char* pa = ws.p;
  unsigned char* pb = pa + abytes;
  int* ea = reinterpret_cast<int*>(pb + bbytes);
  int* eb = ea + mpad;
  int* d_err = eb + npad;
  // A: row i, K index k at A[i + lda k]; B: row j (a column of B), k at B[k + ldb j]
  const OzPackJob ja{A, 1, lda, M, K, nks, pa, ea, mpad / 64};
  const OzPackJob jb{B, ldb, 1, N, K, nks, pb, eb, npad / 64};
  const OzGemmJob gj{pa, ea, pb, eb, M, N, nks, C, ldc, alpha, beta};
  int rc = 0;
  int herr = 0;
  // one fill for the exponents (0x80808080 is below kOzZeroExp) and the status word
  // (whose timeout bit it leaves clear)
  if (cudaMemsetAsync(ea, 0x80, ebytes + sizeof(int), st) != cudaSuccess) {
    rc = 3;
  } else {
    const dim3 grid(mpad / 64 + npad / 64, std::min(65535, (nks + kOzPackKC - 1) / kOzPackKC));
    if (nks > 0 && nks <= kOzPackKC) {
      k_oz_pack_short<<<grid.x, kOzNT, 0, st>>>(ja, jb);
    } else if (nks > 0) {
      k_oz_exponents<<<grid, kOzNT, 0, st>>>(ja, jb);
      k_oz_pack<<<grid, kOzNT, 0, st>>>(ja, jb);
    }
    cudaFuncSetAttribute(k_oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, kOzSmem);
    const int tiles = (mpad / kOzBM) * ((N + kOzBN - 1) / kOzBN);
    k_oz_gemm<<<tiles, kOzNT, kOzSmem, st>>>(gj, d_err);
    if (cudaMemcpyAsync(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) rc = 3;
  }
  ws.give_back(st);
  if (cudaStreamSynchronize(st) != cudaSuccess) rc = 3;
  else if (rc == 0 && (herr & kDevErrTimeout)) rc = 4;
  if (cudaGetLastError() != cudaSuccess) rc = 3;
  return rc;
}

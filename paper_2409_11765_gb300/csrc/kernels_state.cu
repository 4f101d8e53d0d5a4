// kernels_state.cu -- a search's state to and from host memory in one launch.
//
// One kernel moves every vector, matrix and scalar of cmaes_get_state and cmaes_set_state
// between the arena and a pinned host buffer of the handle, and the host copies between
// that buffer and the caller's memory: a copy of its own for each (10 to 14 blocking ones,
// and for set three kernels) is latency. Larger matrices (n > kStateMaxN) go by copies of
// their own, which reach the caller's memory without the host's pass. With a copy for each
// -> here, to restore and to read: n = 40 127 -> 39 and 80 -> 14 us, n = 100 137 -> 47 and
// 83 -> 17, n = 1000 282 -> 242 and 166 -> 122. What is left is the launch, the
// synchronisation and, to restore, the logarithms of the weights in one CTA.
#include <cmath>
#include "descent.cuh"
#include "device_common.cuh"
#include "tc_common.cuh"

namespace cmaes_gb300 {

namespace {
constexpr int kStT = 32;  // matrix tile
}

// Offsets in the buffer, in doubles.
StateLayout state_layout(int n, int hist_cap, bool matrices) {
  StateLayout l;
  l.m = sizeof(StateHead) / 8;
  l.ps = l.m + n;
  l.pc = l.ps + n;
  l.D = l.pc + n;
  l.best_x = l.D + n;
  l.hist = l.best_x + n;
  l.C = l.hist + hist_cap;
  l.B = l.C + (matrices ? static_cast<size_t>(n) * n : 0);
  l.total = l.B + (matrices ? static_cast<size_t>(n) * n : 0);
  l.matrices = matrices;
  return l;
}

// CTA 0: scalars, vectors and the history ring as it lies; the others one tile of C
// and of B each.
__global__ void __launch_bounds__(256) k_state_get(const Search* S, int si, double* buf, StateLayout l) {
  const Search& s = S[si];
  const int n = s.n, tid = threadIdx.x;
  if (blockIdx.x == 0) {
    if (tid == 0) {
      StateHead h{};
      h.sigma = s.sigma;
      h.best_f = s.best_f;
      h.lam = s.lam;
      h.gen = s.gen;
      h.restart = s.restart;
      h.done = s.done;
      h.flags = s.flags;
      h.hist_count = s.hist_count;
      h.hist_len = s.hist_len;
      h.err = *s.err;
      *reinterpret_cast<StateHead*>(buf) = h;
    }
    for (int i = tid; i < n; i += 256) {
      buf[l.m + i] = s.m[i];
      buf[l.ps + i] = s.ps[i];
      buf[l.pc + i] = s.pc[i];
      buf[l.D + i] = s.D[i];
      buf[l.best_x + i] = s.best_x[i];
    }
    for (int i = tid; i < s.hist_len; i += 256) buf[l.hist + i] = s.hist[i];
    return;
  }
  const long long L = s.ldn;
  const int T = ceil_div(n, kStT), t = blockIdx.x - 1, i = (t % T) * kStT + (tid & 31), j0 = (t / T) * kStT;
  if (i >= n) return;
  double c[kStT / 8], b[kStT / 8];
#pragma unroll
  for (int u = 0; u < kStT / 8; ++u) {
    const int j = j0 + (tid >> 5) + 8 * u;
    if (j >= n) break;
    c[u] = s.C[i + L * j];
    b[u] = s.B[i + L * j];
  }
#pragma unroll
  for (int u = 0; u < kStT / 8; ++u) {
    const int j = j0 + (tid >> 5) + 8 * u;
    if (j >= n) break;
    buf[l.C + i + static_cast<long long>(n) * j] = c[u];
    buf[l.B + i + static_cast<long long>(n) * j] = b[u];
  }
}

// The reverse, with what follows from the state: CTA 0 also forms the strategy
// parameters, the others B diag(D) and its operand copy. Nothing is written when the
// handle's status word reports a timeout or a non-finite state: head.err returns it.
// `has` bit k: field k is given (StateField); the others keep their values.
__global__ void __launch_bounds__(256) k_state_put(Search* S, int si, DevOptions o, double* buf, StateLayout l,
                                                   StateHead h, int has) {
  __shared__ double sh[32];
  __shared__ double tile[kStT][kStT + 1];
  Search& s = S[si];
  const int n = s.n, tid = threadIdx.x;
  const int err = *s.err & (kDevErrTimeout | kDevErrNonFinite);
  if (blockIdx.x == 0) {
    if (tid == 0) reinterpret_cast<StateHead*>(buf)->err = err;
    if (err) return;
    for (int i = tid; i < n; i += 256) {
      if (has & 1 << kStM) s.m[i] = buf[l.m + i];
      if (has & 1 << kStPs) s.ps[i] = buf[l.ps + i];
      if (has & 1 << kStPc) s.pc[i] = buf[l.pc + i];
      if (has & 1 << kStD) s.D[i] = buf[l.D + i];
      if (has & 1 << kStBest) s.best_x[i] = buf[l.best_x + i];
    }
    for (int i = tid; i < s.hist_cap; i += 256) {
      if (i < h.hist_count) s.hist[i] = buf[l.hist + i];
      s.hist[s.hist_cap + i] = 0.0;  // the snapshot holds no evaluation errors
    }
    if (tid == 0) {
      s.lam = h.lam;
      s.gen = h.gen;
      s.restart = h.restart;
      s.done = h.done;
      s.flags = h.flags;
      s.sigma = h.sigma;
      s.best_f = h.best_f;
      s.eig_due = 0;
      s.hist_count = h.hist_count;
    }
    __syncthreads();
    compute_params<256>(s, o, sh);
    return;
  }
  if (err) return;
  const long long L = s.ldn;
  const int T = ceil_div(n, kStT), t = blockIdx.x - 1, i0 = (t % T) * kStT, j0 = (t / T) * kStT;
  const int i = i0 + (tid & 31);
  double c[kStT / 8], b[kStT / 8], d[kStT / 8];
#pragma unroll
  for (int u = 0; u < kStT / 8; ++u) {
    const int j = j0 + (tid >> 5) + 8 * u;
    c[u] = b[u] = d[u] = 0.0;
    if (i >= n || j >= n) continue;
    if (has & 1 << kStC) c[u] = buf[l.C + i + static_cast<long long>(n) * j];
    b[u] = has & 1 << kStB ? buf[l.B + i + static_cast<long long>(n) * j] : s.B[i + L * j];
    d[u] = has & 1 << kStD ? buf[l.D + j] : s.D[j];
  }
#pragma unroll
  for (int u = 0; u < kStT / 8; ++u) {
    const int j = j0 + (tid >> 5) + 8 * u;
    const double v = b[u] * d[u];
    tile[(tid >> 5) + 8 * u][tid & 31] = v;
    if (i >= n || j >= n) continue;
    if (has & 1 << kStC) s.C[i + L * j] = c[u];
    if (has & 1 << kStB) s.B[i + L * j] = b[u];
    if (!h.done) s.BD[i + L * j] = v;
  }
  if (!s.mixed || h.done) return;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kStT / 8; ++u) {
    const int ii = (tid >> 5) + 8 * u, kk = tid & 31;
    if (i0 + ii >= n || j0 + kk >= n) continue;
    const long long e = static_cast<long long>(i0 + ii) * s.kp + j0 + kk;
    const float v = static_cast<float>(tile[kk][ii]);
    if (s.mixed == 2) static_cast<__nv_bfloat16*>(s.BDT)[e] = TcElem<1>::from(v);
    else static_cast<float*>(s.BDT)[e] = TcElem<0>::from(v);
  }
}

static int state_blocks(int n, bool matrices) {
  const int T = ceil_div(n, kStT);
  return 1 + (matrices ? T * T : 0);
}
void launch_state_get(const Search* S, int s, int n, double* buf, const StateLayout& l, cudaStream_t st) {
  k_state_get<<<state_blocks(n, l.matrices), 256, 0, st>>>(S, s, buf, l);
}
void launch_state_put(Search* S, int s, int n, DevOptions o, double* buf, const StateLayout& l, const StateHead& h,
                      int has, cudaStream_t st) {
  k_state_put<<<state_blocks(n, l.matrices), 256, 0, st>>>(S, s, o, buf, l, h, has);
}

}  // namespace cmaes_gb300

// The chain: many steps of the update rule per pass over HBM, the sites of a warp in registers.
//
// A lane holds K consecutive sites and a warp 32 K; a step moves psi_0 one site up and psi_1 one
// site down, so only one value of each crosses a lane (two shuffles), and the mass step is the four
// FP32 operations per number of `finish`: at K = 16 a warp issues 256 FP32 operations and 4 shuffles
// per step.  The outermost `steps` sites of a warp's window go stale, one per step and side, and are
// not written: windows overlap by 2 steps.  Bound by the FP32 pipe: 16 operations a site-step.
// Measured on one GB300, complex64: N = 20 000 003, 150 steps: 1.93 ms against 13.1 ms of the
// shared-memory tiles (four steps a pass), 1.56 T site-steps/s; complex128: N = 1024, 512 steps (the
// FP64 pipe, half a lane a clock per quarter of an SM, and the start of a launch): 0.21 ms against
// 2.10 ms of one launch a step (0.36 ms without overlapped launches).
#include <cuda_runtime.h>

#include <algorithm>

#include "qw_internal.cuh"
#include "qw_stencil_dev.cuh"

namespace qw {
namespace {

constexpr int kWarps1 = 4;  // most warps per CTA (independent of one another)

__device__ __forceinline__ float2 shfl_c(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ double2 shfl_c(double2 v, int src) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// steps <= 16 K - 1.  Global accesses are element wise and coalesced; the window is turned between
// that order and the lanes' K consecutive sites in shared memory (rows of K padded to K + 1).
// Plain loads: the launch before may still be writing `in` while this grid starts (launch_overlapped).
template <typename R, int K>
__global__ void __launch_bounds__(32 * kWarps1)
    march1d_kernel(const typename CplxOf<R>::T* in, typename CplxOf<R>::T* out, int64_t N,
                   int steps, int64_t windows, typename CoefOf<R>::T cf) {
  using C = typename CplxOf<R>::T;
  constexpr int W = 32 * K;
  __shared__ C turn[kWarps1][32 * (K + 1)];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t win = (int64_t)blockIdx.x * (blockDim.x >> 5) + w;
  grid_wait();
  if (win >= windows) return;  // whole warps: nothing below synchronises more than a warp
  C* t = turn[w];
  const int valid = W - 2 * steps;
  int64_t s0 = win * valid - steps;  // first site of the window
  C p[2][K];
  if (s0 >= 0 && s0 + W <= N) {  // inside the chain: every load in flight at once
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int i = 0; i < K; ++i) p[q][i] = in[q * N + s0 + i * 32 + lane];
  } else {  // around the chain's end, for a window longer than the chain more than once
    if (s0 < 0) s0 += N;
    if (s0 < 0) s0 = N - 1 - (-s0 - 1) % N;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      int64_t s = s0 + i * 32 + lane;
      if (s >= N) s = N >= W ? s - N : s % N;
      p[0][i] = in[s];
      p[1][i] = in[N + s];
    }
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
#pragma unroll
    for (int i = 0; i < K; ++i) t[i * 32 + lane + (i * 32 + lane) / K] = p[q][i];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < K; ++j) p[q][j] = t[lane * (K + 1) + j];
    __syncwarp();
  }
  const int up = max(lane - 1, 0), dn = min(lane + 1, 31);
  for (int n = 0; n < steps; ++n) {
    C last = shfl_c(p[0][K - 1], up);
    const C next = shfl_c(p[1][0], dn);
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const C o0 = p[0][j], o1 = p[1][j];
      p[0][j] = finish(cf, last, o1);
      p[1][j] = finish(cf, j + 1 < K ? p[1][j + 1 < K ? j + 1 : 0] : next, o0);
      last = o0;
    }
  }
  const int64_t first = win * valid;
  const int count = (int)min((int64_t)valid, N - first);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
#pragma unroll
    for (int j = 0; j < K; ++j) t[lane * (K + 1) + j] = p[q][j];
    __syncwarp();
    for (int e = lane; e < count; e += 32) out[q * N + first + e] = t[e + steps + (e + steps) / K];
    __syncwarp();
  }
}

// Few windows: a warp per CTA, so that they spread over the SMs.
int cta_warps(int64_t windows, int sms) { return windows < (int64_t)kWarps1 * sms ? 1 : kWarps1; }

// us of one launch of `steps` steps with K sites per lane.
template <typename R> double cost1(int64_t N, int K, int steps, int sms) {
  constexpr bool f32 = sizeof(R) == 4;
  const int64_t windows = (N + 32 * K - 2 * steps - 1) / (32 * K - 2 * steps);
  // warps of the fullest SM; its CTAs come and go whole, which the FP64 pipe feels (in FP32 they hide in the waits)
  const int warps = f32 ? 1 : cta_warps(windows, sms);
  const int64_t ctas = (windows + warps - 1) / warps;
  const double per_sm = (double)((ctas + sms - 1) / sms * warps);
  // clocks of a step: a warp on its own (issue and the shuffle's latency; FP64: 8 instructions a
  // site of 64 clocks each, half a lane a clock on its quarter of the SM), or all warps of an SM
  // (FP32: 16 instructions a site on four schedulers; FP64: 8 of 16 clocks each, measured 141 with many steps a
  // launch and 149 with one)
  const double own = f32 ? 16.0 * K + 45.0 : 512.0 * K + 60.0;
  const double all = per_sm * K * (f32 ? 4.4 : 140.0 + 9.0 / steps);
  const double compute = steps * std::max(own, all) / 1900.0;
  const double bytes = 2.0 * 2.0 * (f32 ? 8.0 : 16.0) * (double)N / 5.5e6;
  return 2.5 + std::max(compute, bytes);
}

template <typename R, int K>
qw_status launch1(const void* in, void* out, int64_t N, int steps, typename CoefOf<R>::T cf, int sms,
                  bool overlap, cudaStream_t st) {
  using C = typename CplxOf<R>::T;
  const int64_t windows = (N + 32 * K - 2 * steps - 1) / (32 * K - 2 * steps);
  const int warps = cta_warps(windows, sms);
  return launch_overlapped(march1d_kernel<R, K>, (unsigned)((windows + warps - 1) / warps), 32 * warps, 0, overlap,
                           st, static_cast<const C*>(in), static_cast<C*>(out), N, steps, windows, cf);
}

}  // namespace

// The launches that make nsteps: sites per lane and the number of launches, whose steps differ by
// at most one.  Long chains take the widest window (least overlap); short ones narrower windows on
// more SMs, and as many steps a launch as pay for its start.  K = 0: a launch of a thread per site for
// every step, for complex128 chains that fill the SMs (bound by the same FP64 instructions, and none in a
// halo: N = 20 000 003 310 us a step against 317) and single steps of the shorter ones.
March1 march1_schedule(int64_t N, qw_dtype dt, int64_t nsteps, int sms) {
  const bool f32 = dt == QW_C64;
  const double bytes = 2.0 * (f32 ? 8.0 : 16.0) * (double)N;
  const double copy = f32 ? 3.0 + 2.0 * bytes / 6.0e6 : 4.6 + 2.0 * bytes / (bytes < 33e6 ? 16.0e6 : 6.8e6);
  March1 best{1, nsteps};
  double bc = -1.0;
  if (!f32) {
    bc = (double)nsteps * std::max(4.1, 3.5 + (double)N / 65.4e3) + (nsteps % 2 ? copy : 0.0);
    best.K = 0;
  }
  for (int K : {1, 2, 4, 8, 16}) {
    if (K == 16 && !f32) continue;
    for (int t : {1, 2, 3, 4, 6, 8, 10, 12, 14, 16, 18, 20, 24, 28, 32, 40, 48, 64, 80, 96}) {
      if (t > 12 * K || t > nsteps) continue;
      for (int odd = 0; odd < 2; ++odd) {
        const int64_t k = (nsteps + t - 1) / t + odd;
        if (k > nsteps) continue;
        const int steps = (int)((nsteps + k - 1) / k);
        double c = k % 2 ? copy : 0.0;
        if (f32) {
          c += (double)k * cost1<float>(N, K, steps, sms);
        } else {
          const int64_t full = nsteps - k * (steps - 1);  // launches of `steps`; the others take one step less
          c += kFirstMarch + (double)full * cost1<double>(N, K, steps, sms);
          if (full < k) c += (double)(k - full) * cost1<double>(N, K, steps - 1, sms);
        }
        if (bc < 0 || c < bc) {
          bc = c;
          best = March1{K, k};
        }
      }
    }
  }
  return best;
}

qw_status launch_march1(int64_t N, qw_dtype dt, int K, int steps, double n, double m, const void* in, void* out,
                        int sms, bool overlap, cudaStream_t st) {
  if (dt == QW_C64) {
    const Coef32 cf = make_coef32(1, n, m);
    switch (K) {
      case 1: return launch1<float, 1>(in, out, N, steps, cf, sms, overlap, st);
      case 2: return launch1<float, 2>(in, out, N, steps, cf, sms, overlap, st);
      case 4: return launch1<float, 4>(in, out, N, steps, cf, sms, overlap, st);
      case 8: return launch1<float, 8>(in, out, N, steps, cf, sms, overlap, st);
      default: return launch1<float, 16>(in, out, N, steps, cf, sms, overlap, st);
    }
  }
  const Coef64 cf = make_coef64(1, n, m);
  switch (K) {
    case 1: return launch1<double, 1>(in, out, N, steps, cf, sms, overlap, st);
    case 2: return launch1<double, 2>(in, out, N, steps, cf, sms, overlap, st);
    case 4: return launch1<double, 4>(in, out, N, steps, cf, sms, overlap, st);
    default: return launch1<double, 8>(in, out, N, steps, cf, sms, overlap, st);
  }
}

}  // namespace qw

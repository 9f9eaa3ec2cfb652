// BCC boxes: several steps of the update rule per pass over HBM with the marching kernel of
// qw_march.cuh (any M, complex64 and complex128), and the choice of its tile per box.
//
// complex64, one GB300, G site-steps/s against the kernels it replaced (the two-step
// TMA kernel for M % 64 = 0, one thread per site and step otherwise): M = 256: 206 against 121;
// M = 125: 166 against 68; M = 64: 90 against 36.  It is bound by issue slots and dependent
// latencies (2 warps per scheduler at ~250 registers; IPC 0.55, FP32 pipe 40%), no longer by
// shared memory (43% of the wavefront peak) or HBM (43% at M = 192, 48% at M = 256), so what a tile recomputes in its halo
// costs directly: the tile and the number of steps are chosen by the estimate below.
// complex128: bound by the FP64 pipe (2 lanes a clock and SM): 48 FP64 instructions a site-step
// instead of 104, one step a launch (every recomputed site costs): M = 64: 7.9 against 5.1.
#include <cuda_runtime.h>

#include <algorithm>

#include "qw_march.cuh"

namespace qw {
namespace {

// Instantiated tiles: KX cells per lane, KY rows per warp, T steps, NW warps, CTAs per SM; us per
// half-layer of a CTA with the SM full and of one on its own (measured, which the estimate multiplies
// with the half-layers of the longest CTA).
struct Tile3 {
  int kx, ky, t, nw, ctas;
  double us, alone;
};
template <typename R, int KX, int KY, int T, int NW, int CTAS>
qw_status launch_tile(const March3<typename CplxOf<R>::T>& p, int grid, typename CoefOf<R>::T cf, bool overlap,
                      cudaStream_t st) {
  auto* k = march3d_kernel<R, KX, KY, T, NW, CTAS>;
  constexpr int smem = march3_smem<R, KX, KY, NW>();
  const qw_status s = smem_attr(k, smem);
  if (s != QW_OK) return s;
  return launch_overlapped(k, (unsigned)grid, 32 * NW, smem, overlap, st, p, cf);
}

#define QW_TILES3_C64(X)                                                                            \
  X(1, 3, 4, 8, 1, 1.40, 1.07) X(1, 2, 4, 8, 1, 1.05, 0.80) X(1, 3, 3, 4, 2, 1.04, 0.48)            \
  X(1, 4, 3, 4, 2, 1.42, 0.65) X(1, 4, 2, 4, 2, 1.10, 0.50) X(1, 2, 1, 8, 2, 0.72, 0.33)
#define QW_TILES3_C128(X) X(2, 1, 1, 4, 2, 6.1, 6.1) X(1, 1, 1, 8, 2, 6.5, 6.5)

const Tile3 kTiles64[] = {
#define X(kx, ky, t, nw, ctas, us, alone) {kx, ky, t, nw, ctas, us, alone},
    QW_TILES3_C64(X)};
const Tile3 kTiles128[] = {QW_TILES3_C128(X)
#undef X
};

template <typename C> March3<C> geometry3(const Geometry& g, const Tile3& s, int sms, int* grid) {
  March3<C> p{};
  const int M = (int)g.nx;
  p.g = tile3_geo(M, s.kx, s.ky, s.t, s.nw);
  p.ntx = (M + p.g.tx - 1) / p.g.tx;
  p.nty = (M + p.g.ty - 1) / p.g.ty;
  *grid = march3_split(p, s.t, sms * s.ctas);
  return p;
}

// us of a launch.  Each figure with what was measured beside it, one GB300.
double estimate3(const Geometry& g, const Tile3& s, bool f32, int sms) {
  int grid;
  const March3<float2> p = geometry3<float2>(g, s, sms, &grid);
  const int P = 2 * p.g.M;
  int iters = p.rounds * (P + 2 * s.t);
  if (p.rest) iters += (p.planes < P ? p.planes : P) + 2 * s.t;
  // complex128: us of a half-layer on the FP64 pipe, less the ends of a launch, where nothing is computed
  // (N = 80 29.9 us, 192 242 us, 300 725 us)
  if (!f32) return std::max(10.8, iters * s.us - 7.0);
  // start and end of a launch, and the half-layers of the longest CTA.  One tile across (M <= 32): CTAs on SMs of
  // their own; fewer cells than lanes load the same addresses and take turns (M = 1: twice as long)
  if (g.nx <= 32) return 2.5 + iters * s.alone * (1.0 + 1.2 / ((double)g.nx * g.nx));
  const double us = 2.5 + iters * s.us;
  const double field = (double)g.elems * 8;
  if (field < 64e6) return us;
  // Fields beyond L2: the boxes read with their halos and the field written, at 5.2 TB/s.  Tiles find
  // their neighbours' rows in L2 only while the CTAs keep to one height, which the larger boxes do not:
  // three steps a launch took 545-645 us at N = 512 and 5062 at N = 1024 (450 and 3480 without this
  // bound), four 638 and 4651, so N = 512 went from 156 to 206 G site-steps/s; at N = 450 three stay
  // the better choice (322 against 498 us).  Planes that lie at multiples of large powers of two (M a
  // multiple of 256) reach 4.4 (N = 512: 583 us for two steps, 638 for three).  Fewer steps a launch have more
  // traffic in flight: two steps 5.7 up to 800 MB (N = 400 211 us, 450 306 us), 4.8 beyond (N = 600 863 us, 800
  // 1969 us); one step 5.8 up to 600 MB (N = 320 107 us), 4.2 beyond (N = 600 932 us, 768 1850 us).
  const double box = (double)p.ntx * p.nty * 32 * s.kx * s.ky * s.nw / ((double)p.g.M * p.g.M);
  const double rate = s.t == 1                          ? (field > 600e6 ? 4.2e6 : 5.8e6)
                      : s.t < 4 && g.nx % 256 == 0 ? 4.4e6
                      : s.t == 2                   ? (field > 800e6 ? 4.8e6 : 5.7e6)
                                                   : 5.2e6;
  return std::max(us, field * (box + 1.0) / rate);
}

}  // namespace

// One step: a thread per site (step3d_kernel) where the marching kernel does not fill the SMs or, on large
// boxes, reads its tiles' halos from HBM (N = 600: 708 against 880 us; complex128, where a halo's arithmetic
// costs too, N = 48: 8.2 against 18.1 us, 192: 235 against 242 us); with the TMA kernels allowed, their boxes of
// more than L2 (N = 512: 378 us, against 413 with a thread per site and 608 marching; two steps at N = 1024:
// 4284 against 4800 us marching).
void march3_table(const Geometry& g, qw_dtype dt, int sms, bool tma, StepTable* t) {
  const bool f32 = dt == QW_C64;
  const Tile3* tiles = f32 ? kTiles64 : kTiles128;
  const int n = f32 ? (int)(sizeof(kTiles64) / sizeof(Tile3)) : (int)(sizeof(kTiles128) / sizeof(Tile3));
  for (int i = 0; i <= 4; ++i) t->kernel[i] = kNoStep;
  auto offer = [t](int steps, int kernel, double us) {
    if (t->kernel[steps] != kNoStep && t->us[steps] <= us) return;
    t->us[steps] = us;
    t->kernel[steps] = kernel;
  };
  for (int i = 0; i < n; ++i) offer(tiles[i].t, i, estimate3(g, tiles[i], f32, sms));
  // the threads of whole warps along x: FP64 pipe at 7.75 G, or L2 and HBM at 78 G threads/s
  const double threads = 2.0 * (double)g.nx * g.nx * (double)((g.nx + 31) / 32 * 32);
  const double site = f32 ? std::max(g.nx == 1 ? 3.1 : 4.1, 3.3 + threads / 78e3)
                          : std::max(7.0, 5.8 + threads / 7.75e3);
  // a run has few single steps in complex64, and the first launch of a marching kernel does not overlap
  if (t->us[1] + (f32 ? kFirstMarch : 0.0) >= site) {
    t->us[1] = site;
    t->kernel[1] = kSiteStep;
  }
  const double field = (double)g.elems * 8;
  if (tma && f32 && tma_step_supported(g)) offer(1, kTmaStep, 15.0 + 2.0 * field / 5.9e6);
  if (tma && f32 && tma2_step_supported(g)) offer(2, kTma2Step, 15.0 + 2.0 * field / 4.0e6);
}

qw_status launch_march3(const Geometry& g, qw_dtype dt, int kernel, double n, double m, const void* in, void* out,
                        int sms, bool overlap, cudaStream_t st) {
  int grid, i = 0;
  auto planes = [&](auto& p) {
    using C = std::remove_const_t<std::remove_pointer_t<std::remove_reference_t<decltype(p.out[0][0])>>>;
    for (int c = 0; c < 2; ++c)
      for (int q = 0; q < 4; ++q) {
        p.in[c][q] = static_cast<const C*>(in) + (int64_t)(c * 4 + q) * g.vol;
        p.out[c][q] = static_cast<C*>(out) + (int64_t)(c * 4 + q) * g.vol;
      }
  };
  if (dt == QW_C64) {
    March3<float2> p = geometry3<float2>(g, kTiles64[kernel], sms, &grid);
    planes(p);
    const Coef32 cf = make_coef32(3, n, m);
#define X(kx, ky, T, nw, ctas, us, alone) \
  if (i++ == kernel) return launch_tile<float, kx, ky, T, nw, ctas>(p, grid, cf, overlap, st);
    QW_TILES3_C64(X)
  } else {
    March3<double2> p = geometry3<double2>(g, kTiles128[kernel], sms, &grid);
    planes(p);
    const Coef64 cf = make_coef64(3, n, m);
#undef X
#define X(kx, ky, T, nw, ctas, us, alone) \
  if (i++ == kernel) return launch_tile<double, kx, ky, T, nw, ctas>(p, grid, cf, overlap, st);
    QW_TILES3_C128(X)
#undef X
  }
  return QW_EINVAL;
}

}  // namespace qw

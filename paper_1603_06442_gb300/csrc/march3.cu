// BCC boxes: several steps of the update rule per pass over HBM with the marching kernel of
// qw_march.cuh (any M, complex64 and complex128), and the choice of its tile per box.
//
// complex64, one GB300, G site-steps/s against the kernels it replaced (the two-step
// TMA kernel for M % 64 = 0, one thread per site and step otherwise): M = 256: 206 against 121;
// M = 125: 166 against 68; M = 64: 90 against 36.  It is bound by issue slots and dependent
// latencies (2 warps per scheduler at ~250 registers; IPC 0.55, FP32 pipe 40%), no longer by
// shared memory (40% of the wavefront peak) or HBM (31%), so what a tile recomputes in its halo
// costs directly: the tile and the number of steps are chosen by the estimate below.
// complex128: bound by the FP64 pipe (2 lanes a clock and SM): 48 FP64 instructions a site-step
// instead of 104, one step a launch (every recomputed site costs): M = 64: 7.9 against 5.1.
#include <cuda_runtime.h>

#include "qw_march.cuh"

namespace qw {
namespace {

// Instantiated tiles: KX cells per lane, KY rows per warp, T steps, NW warps, CTAs per SM; us per
// half-layer of a CTA with the SM full (measured, which the estimate multiplies with the half-layers
// of the longest CTA).
struct Tile3 {
  int kx, ky, t, nw, ctas;
  double us;
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
  X(1, 3, 4, 8, 1, 1.40) X(1, 2, 4, 8, 1, 1.05) X(1, 3, 3, 4, 2, 1.04) X(1, 4, 3, 4, 2, 1.42)       \
  X(1, 4, 2, 4, 2, 1.25) X(1, 2, 1, 8, 2, 0.85)
#define QW_TILES3_C128(X) X(2, 1, 1, 4, 2, 4.9) X(1, 1, 1, 8, 2, 5.0)

const Tile3 kTiles64[] = {
#define X(kx, ky, t, nw, ctas, us) {kx, ky, t, nw, ctas, us},
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

double estimate3(const Geometry& g, const Tile3& s, int elem, int sms) {
  int grid;
  const March3<float2> p = geometry3<float2>(g, s, sms, &grid);
  const int P = 2 * p.g.M;
  int iters = p.rounds * (P + 2 * s.t);
  if (p.rest) iters += (p.planes < P ? p.planes : P) + 2 * s.t;
  const double us = 2.5 + iters * s.us;  // a launch: start and end, and the half-layers of the longest CTA
  const double field = (double)g.elems * elem;
  if (field < 64e6) return us;
  // Fields beyond L2: the boxes read with their halos and the field written, at 5.2 TB/s.  Tiles find
  // their neighbours' rows in L2 only while the CTAs keep to one height, which the larger boxes do not:
  // three steps a launch took 545-645 us at N = 512 and 5062 at N = 1024 (450 and 3480 without this
  // bound), four 638 and 4651, so N = 512 went from 156 to 206 G site-steps/s; at N = 450 three stay
  // the better choice (322 against 498 us).
  const double box = (double)p.ntx * p.nty * 32 * s.kx * s.ky * s.nw / ((double)p.g.M * p.g.M);
  const double hbm = field * (box + 1.0) / 5.2e6;
  return us > hbm ? us : hbm;
}

}  // namespace

double march3_cost(const Geometry& g, qw_dtype dt, int steps, int sms) {
  double best = -1.0;
  const Tile3* t = dt == QW_C64 ? kTiles64 : kTiles128;
  const int n = dt == QW_C64 ? (int)(sizeof(kTiles64) / sizeof(Tile3)) : (int)(sizeof(kTiles128) / sizeof(Tile3));
  for (int i = 0; i < n; ++i)
    if (t[i].t == steps) {
      const double c = estimate3(g, t[i], dt == QW_C64 ? 8 : 16, sms);
      if (best < 0 || c < best) best = c;
    }
  return best;
}

qw_status launch_march3(const Geometry& g, qw_dtype dt, int steps, double n, double m, const void* in, void* out,
                        int sms, bool overlap, cudaStream_t st) {
  const Tile3* t = dt == QW_C64 ? kTiles64 : kTiles128;
  const int cnt = dt == QW_C64 ? (int)(sizeof(kTiles64) / sizeof(Tile3)) : (int)(sizeof(kTiles128) / sizeof(Tile3));
  int best = -1;
  double bc = 0.0;
  for (int i = 0; i < cnt; ++i) {
    if (t[i].t != steps) continue;
    const double c = estimate3(g, t[i], dt == QW_C64 ? 8 : 16, sms);
    if (best < 0 || c < bc) {
      best = i;
      bc = c;
    }
  }
  if (best < 0) {
    set_error("marching stencil: no kernel for %d steps", steps);
    return QW_EINVAL;
  }
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
    March3<float2> p = geometry3<float2>(g, t[best], sms, &grid);
    planes(p);
    const Coef32 cf = make_coef32(3, n, m);
#define X(kx, ky, T, nw, ctas, us) \
  if (i++ == best) return launch_tile<float, kx, ky, T, nw, ctas>(p, grid, cf, overlap, st);
    QW_TILES3_C64(X)
  } else {
    March3<double2> p = geometry3<double2>(g, t[best], sms, &grid);
    planes(p);
    const Coef64 cf = make_coef64(3, n, m);
#undef X
#define X(kx, ky, T, nw, ctas, us) \
  if (i++ == best) return launch_tile<double, kx, ky, T, nw, ctas>(p, grid, cf, overlap, st);
    QW_TILES3_C128(X)
#undef X
  }
  return QW_EINVAL;
}

}  // namespace qw

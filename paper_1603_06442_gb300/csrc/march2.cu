// The square lattice: several steps of the update rule per pass over HBM with the marching kernel of
// qw_march2.cuh, the split of a field over its warps, and (for the BCC boxes too) the mix of launches
// that makes a number of steps.
//
// complex64, one GB300: N = 2998, 150 steps: 5.8 ms against 15.3 ms of one thread per site and one
// pass per step; G site-steps/s: N = 8192: 245 (four steps a pass) against 94.  It is bound by issue and
// latency at two warps per scheduler (0.58 a cycle at N = 2998, FP32 pipe 44%; 41 additions, 16 packed mass
// operations and 4 shuffles a site-step), then by the halo of 8 in 64 columns; HBM is at 43%.  Measured slower (the kernel alone makes 263 at
// N = 8192): rows handed from level to level one row late, so that the levels are independent (253),
// and the sums in packed additions (244: fewer instructions, the same pipe).
// One step, and complex128 (64 FP64 instructions a site-step on the FP64 pipe, where a recomputed
// halo costs as much as shared sums save: 523 against 539 us at N = 2048), stay with one thread per
// site (stencil.cu).
#include <cuda_runtime.h>

#include <algorithm>

#include "qw_march2.cuh"

namespace qw {
namespace {

// Instantiated kernels: KX columns per lane, T steps, warps per CTA, CTAs per SM; us of one row with
// the SM full, and of one row of a warp on its own (measured).
struct Strip2 {
  int kx, t, nw, ctas;
  double full, own;
};
#define QW_STRIPS2(X) X(2, 4, 4, 2, 1.00, 0.45) X(2, 3, 4, 3, 1.25, 0.36) X(2, 2, 4, 4, 1.66, 0.27)
#define X(kx, t, nw, ctas, full, own) {kx, t, nw, ctas, full, own},
const Strip2 kStrips[] = {QW_STRIPS2(X)};
#undef X

// The chunks of rows per strip: enough warps for every SM, but no more rows recomputed at the chunks'
// ends (2 T each) than the waves saved; *us receives the estimate of the launch.
March2 geometry2(int64_t N, const Strip2& s, int sms, double* us) {
  March2 p{};
  p.N = (int)N;
  const int tx = 32 * s.kx - 2 * s.t;
  p.ntx = (p.N + tx - 1) / tx;
  const int full = sms * s.ctas * s.nw;  // resident warps
  const int base = std::max(1, full / p.ntx);
  double best = -1.0;
  for (int c : {1, base / 8, base / 4, base / 2, base, 2 * base, 3 * base, 4 * base, p.N}) {
    if (c < 1 || c > p.N) continue;
    const int rows = (p.N + c - 1) / c, chunks = (p.N + rows - 1) / rows;
    const int64_t items = (int64_t)p.ntx * chunks;
    const int64_t waves = (items + full - 1) / full;
    // time a row of the SM with most warps: of full waves, or of a part of one.  Half the warps take two
    // thirds of the time, not half: with one warp a scheduler nothing fills its waits (a proportional
    // share left N = 2998 and 8192 half empty: 192 and 198 against 232 and 245 G site-steps/s)
    const double share = waves > 1 ? 1.0 : (double)((items + sms - 1) / sms) / (s.ctas * s.nw);
    const double t = waves * (rows + 2 * s.t) * std::max(s.own, s.full * (0.33 + 0.67 * share));
    if (best < 0 || t < best) {
      best = t;
      p.rows = rows;
      p.chunks = chunks;
    }
  }
  *us = 2.5 + best;
  return p;
}

template <int KX, int T, int NW, int CTAS>
qw_status launch_strips(const March2& p, const Coef32& cf, bool overlap, cudaStream_t st) {
  auto* k = march2d_kernel<KX, T, NW, CTAS>;
  constexpr int smem = march2_smem<KX, NW>();
  const qw_status s = smem_attr(k, smem);
  if (s != QW_OK) return s;
  const int64_t items = (int64_t)p.ntx * p.chunks;
  return launch_overlapped(k, (unsigned)((items + NW - 1) / NW), 32 * NW, smem, overlap, st, p, cf);
}

}  // namespace

void march2_table(const Geometry& g, qw_dtype dt, int sms, StepTable* t) {
  for (int i = 0; i <= 4; ++i) t->kernel[i] = kNoStep;
  // one thread per site: launches and HBM at 90 G site-steps/s (complex64: N = 2998 101 us; two steps a launch
  // 114 us, with a copy of the field where the run has no second one), or the FP64 pipe
  t->us[1] = std::max(4.1, 2.0 + (double)g.sites / (dt == QW_C64 ? 90.0e3 : 7.8e3));
  t->kernel[1] = kSiteStep;
  if (dt != QW_C64) return;
  for (int i = 0; i < (int)(sizeof(kStrips) / sizeof(Strip2)); ++i) {
    const Strip2& s = kStrips[i];
    geometry2(g.nx, s, sms, &t->us[s.t]);
    t->kernel[s.t] = i;
  }
}

qw_status launch_march2(const Geometry& g, int kernel, double n, double m, const void* in, void* out, int sms,
                        bool overlap, cudaStream_t st) {
  const Strip2& s = kStrips[kernel];
  double us;
  March2 p = geometry2(g.nx, s, sms, &us);
  for (int q = 0; q < 4; ++q) {
    p.in[q] = static_cast<const float2*>(in) + q * g.vol;
    p.out[q] = static_cast<float2*>(out) + q * g.vol;
  }
  const Coef32 cf = make_coef32(2, n, m);
#define X(kx, T, nw, ctas, full, own) \
  if (s.t == T) return launch_strips<kx, T, nw, ctas>(p, cf, overlap, st);
  QW_STRIPS2(X)
#undef X
  return QW_EINVAL;
}

// The kernels index a component plane (of a coset) in 32 bits.
bool march_supported(const Geometry& g, qw_dtype) { return g.dim >= 2 && g.vol < (int64_t)1 << 32; }

// The cheapest mix by the estimates; an odd number of launches ends in the scratch field and costs a
// copy of the field.
void march_schedule(const Geometry& g, qw_dtype dt, int64_t nsteps, const StepTable& table, int64_t (&count)[5]) {
  const double bytes = (double)g.elems * (dt == QW_C64 ? 8 : 16);
  const double copy = 4.6 + 2.0 * bytes / (bytes < 33e6 ? 16.0e6 : 6.8e6);  // 4.6 after a kernel; L2 or HBM
  double best = -1.0;
  for (int64_t& c : count) c = 0;
  // small counts of three of the sizes, the rest in launches of the fourth
  for (int main = 1; main <= 4 && main <= nsteps; ++main) {
    if (table.kernel[main] == kNoStep) continue;
    int64_t k[5] = {0, 0, 0, 0, 0};
    const int a = main == 1 ? 2 : 1, b = main <= 2 ? 3 : 2, c = main <= 3 ? 4 : 3;
    auto most = [&](int t, int64_t left) { return table.kernel[t] == kNoStep ? 0 : std::min<int64_t>(4, left / t); };
    const int64_t ma = most(a, nsteps);
    for (k[a] = 0; k[a] <= ma; ++k[a]) {
      const int64_t la = nsteps - a * k[a], mb = most(b, la);
      for (k[b] = 0; k[b] <= mb; ++k[b]) {
        const int64_t lb = la - b * k[b], mc = most(c, lb);
        for (k[c] = 0; k[c] <= mc; ++k[c]) {
          const int64_t left = lb - c * k[c];
          if (left % main) continue;
          k[main] = left / main;
          const int64_t launches = k[1] + k[2] + k[3] + k[4];
          double total = launches % 2 ? copy : 0.0;
          for (int t = 1; t <= 4; ++t)
            // the first of a marching kernel's launches does not overlap the launch before it
            if (k[t]) total += (double)k[t] * table.us[t] + (table.kernel[t] >= 0 ? kFirstMarch : 0.0);
          if (best < 0 || total < best) {
            best = total;
            for (int t = 1; t <= 4; ++t) count[t] = k[t];
          }
        }
      }
    }
  }
}

}  // namespace qw

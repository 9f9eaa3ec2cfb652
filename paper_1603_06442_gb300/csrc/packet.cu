// Synthetic initial states on the device: a Gaussian packet times a plane wave
// times a fixed spinor, the shape of the particle states of Sec. 5 (Definition 1,
// Figs. 2, 5, 6) written in position space.  The served path builds its
// inputs here so that no field crosses the host link.
#include <cuda_runtime.h>

#include <cmath>

#include "qw_internal.cuh"

namespace qw {

struct PacketArgs {
  double x0[3], k0[3], chi[8];
  double inv4s2;  // 1 / (4 sigma^2)
};

constexpr int kPacketRows = 8;  // y rows per CTA (2D and BCC): the x factor is reused across them

// One axis of the separable packet: exp(-d^2 / (4 sigma^2)) exp(i k0 d) at the
// lattice coordinate pos, d the minimum-image displacement from x0 in [-N/2, N/2).
// d and the phase k0 d (reduced modulo 2 pi) are formed in FP64, since d can
// exceed 2^24 on long chains; complex64 then takes expf / sincosf of the small
// reduced arguments, complex128 stays in FP64.
template <typename T>
__device__ __forceinline__ typename CplxOf2<T>::t axis_factor(double pos, double x0, double N, double invN, double k0,
                                                              double inv4s2) {
  double d = pos - x0 + 0.5 * N;
  d = fma(-N, floor(d * invN), d);
  d = d < 0.0 ? d + N : (d >= N ? d - N : d);  // guard the rounding of d * invN
  d -= 0.5 * N;
  const double arg = d * d * inv4s2;
  const double ph = k0 * d;
  const double r = fma(-6.283185307179586232, rint(ph * 0.15915494309189533577), ph);
  typename CplxOf2<T>::t v;
  if (sizeof(T) == 8) {
    double sn, cs;
    sincos(r, &sn, &cs);
    const double e = exp(-arg);
    v.x = (T)(e * cs);
    v.y = (T)(e * sn);
  } else {
    float sn, cs;
    sincosf((float)r, &sn, &cs);
    const float e = arg < 104.0 ? expf(-(float)arg) : 0.0f;
    v.x = (T)(e * cs);
    v.y = (T)(e * sn);
  }
  return v;
}

template <typename V>
__device__ __forceinline__ V cx_mul(V a, V b) {
  V r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}

// grid (ceil(nx / 256), ceil(ny / kPacketRows), nz * ncoset); each CTA fills
// kPacketRows rows of one (z, coset) plane.
template <typename T>
__global__ void __launch_bounds__(256) packet_kernel(Geometry g, PacketArgs pa, typename CplxOf2<T>::t* psi) {
  using V = typename CplxOf2<T>::t;
  __shared__ V fyz[kPacketRows];
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t y0 = (int64_t)blockIdx.y * kPacketRows, zc = blockIdx.z;
  const int c = g.dim == 3 ? (int)(zc & 1) : 0;
  const int64_t z = g.dim == 3 ? (zc >> 1) : 0;
  const double N = (double)g.N, invN = 1.0 / N;
  const double scale = g.dim == 3 ? 2.0 : 1.0;
  const int rows = g.dim == 1 ? 1 : (int)((g.ny - y0) < kPacketRows ? (g.ny - y0) : kPacketRows);
  if (threadIdx.x < rows) {  // the y (and z) factors of this CTA's rows
    V f;
    f.x = (T)1;
    f.y = (T)0;
    if (g.dim >= 2)
      f = axis_factor<T>(scale * (double)(y0 + threadIdx.x) + c, pa.x0[1], N, invN, pa.k0[1], pa.inv4s2);
    if (g.dim == 3) f = cx_mul(f, axis_factor<T>(scale * (double)z + c, pa.x0[2], N, invN, pa.k0[2], pa.inv4s2));
    fyz[threadIdx.x] = f;
  }
  __syncthreads();
  if (x >= g.nx) return;
  const V fx = axis_factor<T>(scale * (double)x + c, pa.x0[0], N, invN, pa.k0[0], pa.inv4s2);
  V chi[4];
  for (int q = 0; q < g.s; ++q) {
    chi[q].x = (T)pa.chi[2 * q];
    chi[q].y = (T)pa.chi[2 * q + 1];
  }
  for (int r = 0; r < rows; ++r) {
    const V f = cx_mul(fx, fyz[r]);
    const int64_t cell = (z * g.ny + (y0 + r)) * g.nx + x;
    for (int q = 0; q < g.s; ++q) psi[((int64_t)c * g.s + q) * g.vol + cell] = cx_mul(f, chi[q]);
  }
}

// ---- complex64 without FP64: an FP64 instruction costs ~64 FP32 ones here, and a chain has an axis
// factor per site.  Positions are whole numbers: with x0 = X + delta, d = di - delta for the whole
// number di = minimum image of pos - X.  The phase k0 d / 2 pi is taken in 64-bit fixed point (turns,
// modulo 1: exact up to the rounding of k0 / 2 pi), d and d^2 / (4 sigma^2) in two FP32 pieces.
// Measured against the FP64 form: chain N = 20 000 003 127 against 1266 us (320 MB written), square
// lattice N = 2187 38 against 61 us, BCC N = 324 55 against 125 us (16 rows a group, several groups a
// CTA, instead of 8 rows); rms error against 64 bits 7.4e-8 against 7.8e-8 of the norm on the chain,
// 1.2e-7 against 1.3e-7 on the BCC lattice.
struct AxisF {
  long long X, N, wrap;     // floor(x0) mod N, the side, the first image (pos - X) mod N that is taken as - N
  unsigned long long k, k0; // k0 / 2 pi and delta k0 / 2 pi, in units of 2^-64 turns
  float dh, dl, ch, cl;     // delta = dh + dl; 1 / (4 sigma^2) = ch + cl
};
struct PacketF {
  AxisF ax[3];
  float2 chi[4];
};

static unsigned long long turns64(double t) {
  t -= floor(t);
  return t >= 1.0 ? 0ull : (unsigned long long)(t * 18446744073709551616.0);
}

static AxisF axis_f(double x0, double N, double k0, double inv4s2) {
  AxisF a;
  double X = floor(x0);
  const double delta = x0 - X;
  X -= N * floor(X / N);
  a.N = (long long)N;
  a.X = (long long)X % a.N;
  if (a.X < 0) a.X += a.N;  // the quotient was rounded up
  a.wrap = (long long)ceil(0.5 * N + delta);
  const double kt = k0 / 6.283185307179586232;
  a.k = turns64(kt);
  a.k0 = turns64(kt * delta);
  a.dh = (float)delta;
  a.dl = (float)(delta - (double)a.dh);
  a.ch = (float)inv4s2;
  a.cl = (float)(inv4s2 - (double)a.ch);
  return a;
}

__device__ __forceinline__ float2 axis_factor_f(const AxisF& a, long long pos) {
  long long e = pos - a.X;
  if (e < 0) e += a.N;
  const long long di = e >= a.wrap ? e - a.N : e;
  const unsigned long long turns = (unsigned long long)di * a.k - a.k0;
  const float t = (float)(int)(turns >> 32) * 2.3283064365386963e-10f;  // in [-1/2, 1/2)
  float sn, cs;
  sincospif(2.0f * t, &sn, &cs);
  const float h = (float)di, l = (float)(di - (long long)h) - a.dh;
  const float d = h + l, r = (l - (d - h)) - a.dl;  // di - delta = d + r, |r| below an ulp of d
  const float p = d * d, pe = fmaf(2.0f * d, r, fmaf(d, d, -p));
  const float arg = fmaf(p, a.ch, fmaf(p, a.cl, pe * a.ch));
  const float ex = arg < 104.0f ? expf(-arg) : 0.0f;
  return make_float2(ex * cs, ex * sn);
}

// Rows of 256 sites (chain) or kPacketGroup rows of the box per unit; a CTA takes units in turn and
// leaves sum |psi|^2 of what it wrote in partials (four doubles, the last three 0).  The densities of at
// most 8 sites are summed in FP32, as the moments kernel does, and those sums in FP64.
constexpr int kPacketGroup = 16, kPacketChain = 8;
__global__ void __launch_bounds__(256) packet_f_kernel(Geometry g, PacketF pa, int bx, int64_t units,
                                                       float2* __restrict__ psi, double* __restrict__ partials) {
  __shared__ float2 fyz[kPacketGroup];
  double acc[1] = {0.0};
  const int tid = threadIdx.x;
  if (g.dim == 1) {
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
      float sum = 0.f;
#pragma unroll 2
      for (int j = 0; j < kPacketChain; ++j) {
        const int64_t x = (u * kPacketChain + j) * 256 + tid;
        if (x >= g.nx) break;
        const float2 f = axis_factor_f(pa.ax[0], x);
        float d = 0.f;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const float2 v = cx_mul(f, pa.chi[q]);
          psi[q * g.vol + x] = v;
          d = fmaf(v.x, v.x, fmaf(v.y, v.y, d));
        }
        sum += d;
      }
      acc[0] += (double)sum;
    }
  } else {
    const int tx = tid % bx, ty = tid / bx, by = 256 / bx;
    const int xt = (int)((g.nx + bx - 1) / bx);
    const int64_t rows = (int64_t)g.ncoset * g.nz * g.ny;
    const int scale = g.dim == 3 ? 2 : 1;
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
      const int64_t row0 = u / xt * kPacketGroup;
      const int x = (int)(u % xt) * bx + tx;
      __syncthreads();  // fyz of the unit before has been read
      if (tid < kPacketGroup && row0 + tid < rows) {
        const int64_t row = row0 + tid, zc = row / g.ny, y = row - zc * g.ny;
        const int c = (int)(zc / g.nz);
        float2 f = axis_factor_f(pa.ax[1], scale * y + c);
        if (g.dim == 3) f = cx_mul(f, axis_factor_f(pa.ax[2], scale * (zc - c * g.nz) + c));
        fyz[tid] = f;
      }
      __syncthreads();
      if (ty < by && x < g.nx) {
        float sum = 0.f;
        int cx = -1, sites = 0;
        float2 fx = make_float2(0.f, 0.f);
        for (int r = ty; r < kPacketGroup && row0 + r < rows; r += by) {
          const int64_t row = row0 + r;
          const int c = g.ncoset == 2 && row >= g.nz * g.ny ? 1 : 0;
          if (c != cx) {  // the x factor of the row's coset
            fx = axis_factor_f(pa.ax[0], (long long)scale * x + c);
            cx = c;
          }
          const float2 f = cx_mul(fx, fyz[r]);
          float2* dst = psi + (int64_t)c * 3 * g.vol + row * g.nx + x;  // row counts through both cosets
          float d = 0.f;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float2 v = cx_mul(f, pa.chi[q]);
            dst[q * g.vol] = v;
            d = fmaf(v.x, v.x, fmaf(v.y, v.y, d));
          }
          sum += d;
          if (++sites == 8) {
            acc[0] += (double)sum;
            sum = 0.f;
            sites = 0;
          }
        }
        acc[0] += (double)sum;
      }
    }
  }
  if (!partials) return;
  block_sum<1, 256>(acc);
  if (tid == 0) {
    partials[4 * blockIdx.x] = acc[0];
    partials[4 * blockIdx.x + 1] = partials[4 * blockIdx.x + 2] = partials[4 * blockIdx.x + 3] = 0.0;
  }
}

static qw_status launch_packet_f(const Geometry& g, const double* x0, double sigma, const double* k0,
                                 const double* chi, void* psi, double* partials, cudaStream_t st) {
  PacketF pa;
  const double inv4s2 = 1.0 / (4.0 * sigma * sigma);
  for (int j = 0; j < 3; ++j) pa.ax[j] = axis_f(j < g.dim ? x0[j] : 0.0, (double)g.N, j < g.dim ? k0[j] : 0.0, inv4s2);
  for (int q = 0; q < 4; ++q) pa.chi[q] = make_float2((float)chi[2 * q], (float)chi[2 * q + 1]);
  const int bx = (int)(g.nx < 256 ? (g.nx + 31) / 32 * 32 : 256);
  int64_t units;
  if (g.dim == 1)
    units = (g.nx + 256 * kPacketChain - 1) / (256 * kPacketChain);
  else
    units = ((int64_t)g.ncoset * g.nz * g.ny + kPacketGroup - 1) / kPacketGroup * ((g.nx + bx - 1) / bx);
  packet_f_kernel<<<kObsBlocks, 256, 0, st>>>(g, pa, bx, units, static_cast<float2*>(psi), partials);
  QW_CHECK_LAUNCH("packet launch");
  return QW_OK;
}

// Finite parameters in the range of the fixed-point form: a whole number floor(x0) in 64 bits, k0 / 2 pi
// with 30 bits or more after the point, d^2 / (4 sigma^2) within FP32.  The rest (and complex128) keeps
// the FP64 form, which is the slower one at every size.
bool packet_sums(const Geometry& g, qw_dtype dt, const double* x0, double sigma, const double* k0) {
  bool ok = dt == QW_C64 && sigma > 1e-6;
  for (int j = 0; j < g.dim; ++j) ok = ok && fabs(x0[j]) < 9.0e15 && fabs(k0[j]) < 1.0e6;
  return ok;
}

qw_status launch_packet(const Geometry& g, qw_dtype dt, const double* x0, double sigma, const double* k0,
                        const double* chi, void* psi, cudaStream_t st, double* partials) {
  if (!(sigma > 0.0)) {
    set_error("packet: sigma must be > 0");
    return QW_EINVAL;
  }
  if (packet_sums(g, dt, x0, sigma, k0)) return launch_packet_f(g, x0, sigma, k0, chi, psi, partials, st);
  if (partials) {
    set_error("packet: no norm for these parameters");
    return QW_EINVAL;
  }
  PacketArgs pa;
  for (int j = 0; j < 3; ++j) {
    pa.x0[j] = x0[j];
    pa.k0[j] = k0[j];
  }
  for (int j = 0; j < 8; ++j) pa.chi[j] = chi[j];
  pa.inv4s2 = 1.0 / (4.0 * sigma * sigma);
  dim3 grid((unsigned)((g.nx + 255) / 256), (unsigned)((g.ny + kPacketRows - 1) / kPacketRows),
            (unsigned)(g.nz * g.ncoset));
  if (dt == QW_C64)
    packet_kernel<float><<<grid, 256, 0, st>>>(g, pa, static_cast<float2*>(psi));
  else
    packet_kernel<double><<<grid, 256, 0, st>>>(g, pa, static_cast<double2*>(psi));
  QW_CHECK_LAUNCH("packet launch");
  return QW_OK;
}

}  // namespace qw

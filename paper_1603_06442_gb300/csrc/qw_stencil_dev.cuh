// Per-site update of the Dirac walk shared by the plain and batched stencil
// kernels (derivation of the transition matrices at the top of stencil.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "qw_internal.cuh"

namespace qw {

template <typename R> struct CplxOf;
template <> struct CplxOf<float> { using T = float2; };
template <> struct CplxOf<double> { using T = double2; };

// Loads of the field.  The read-only path (__ldg, ld.global.nc) is only valid
// while nothing in the same launch writes the field; the batched kernel, whose
// CTAs read what other CTAs wrote earlier in the launch, passes NC = false and
// uses ordinary loads, which the PTX memory model orders after the CTA's
// acquire (thread 0's ld.acquire.gpu, then bar.sync).
template <bool NC = true, typename C>
__device__ __forceinline__ C ldg(const C* p) {
  if constexpr (NC) return __ldg(p);
  else return *p;  // ordinary load: ordered after the CTA's acquire by the memory model
}

// acc += (A + i B) * v  for A, B in {-1, 0, 1}: additions only.
template <int A, int B, typename C>
__device__ __forceinline__ void cmac(C& acc, const C& v) {
  if constexpr (A == 1) { acc.x += v.x; acc.y += v.y; }
  if constexpr (A == -1) { acc.x -= v.x; acc.y -= v.y; }
  if constexpr (B == 1) { acc.x -= v.y; acc.y += v.x; }
  if constexpr (B == -1) { acc.x += v.y; acc.y -= v.x; }
}

// nq * S + i m * o  (FP32: hi/lo split coefficients through FMA chains).
__device__ __forceinline__ float2 finish(const Coef32& c, float2 S, float2 o) {
  float rx = -c.m_lo * o.y;
  rx = fmaf(c.nq_lo, S.x, rx);
  rx = fmaf(-c.m_hi, o.y, rx);
  rx = fmaf(c.nq_hi, S.x, rx);
  float ry = c.m_lo * o.x;
  ry = fmaf(c.nq_lo, S.y, ry);
  ry = fmaf(c.m_hi, o.x, ry);
  ry = fmaf(c.nq_hi, S.y, ry);
  return make_float2(rx, ry);
}
__device__ __forceinline__ double2 finish(const Coef64& c, double2 S, double2 o) {
  return make_double2(fma(c.nq, S.x, -c.m * o.y), fma(c.nq, S.y, c.m * o.x));
}

template <typename R> struct CoefOf;
template <> struct CoefOf<float> { using T = Coef32; };
template <> struct CoefOf<double> { using T = Coef64; };

template <typename I>
__device__ __forceinline__ I wrapm(I v, I M) { return v < 0 ? v + M : (v >= M ? v - M : v); }


// ------------------------------------------------------------ per-site updates
// Each update has a core that takes pointers to component 0 of the cells it reads and a
// component stride, so that fields in global memory and tiles in shared memory (other
// pitches) run the same arithmetic in the same order.

// chain, s = 2: psi'_0(x) = n psi_0(x-1) + i m psi_1(x), psi'_1(x) = i m psi_0(x) + n psi_1(x+1)
template <bool NC, typename C, typename CF, typename I>
__device__ __forceinline__ void core_1d(const C* xm, const C* xp, const C* own, I cs, C (&r)[2], const CF& cf) {
  C a = ldg<NC>(xm);        // psi_0(x - 1)
  C b = ldg<NC>(xp + cs);   // psi_1(x + 1)
  C o0 = ldg<NC>(own), o1 = ldg<NC>(own + cs);
  r[0] = finish(cf, a, o1);
  r[1] = finish(cf, b, o0);
}

// (I: index type; the batched kernel's walks fit 32-bit indices)
template <typename R, bool NC = true, typename I = int64_t>
__device__ __forceinline__ void site_update_1d(const typename CplxOf<R>::T* __restrict__ in,
                                               typename CplxOf<R>::T* __restrict__ out, I N, I x,
                                               const typename CoefOf<R>::T& cf) {
  typename CplxOf<R>::T r[2];
  core_1d<NC>(in + wrapm<I>(x - 1, N), in + wrapm<I>(x + 1, N), in + x, N, r, cf);
  out[x] = r[0];
  out[N + x] = r[1];
}

// Complex helpers of the factored updates: rho = 1 + i, rhob = 1 - i.
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
template <typename C> __device__ __forceinline__ C rho(C z) { return C{z.x - z.y, z.x + z.y}; }
template <typename C> __device__ __forceinline__ C rhob(C z) { return C{z.x + z.y, z.y - z.x}; }
template <typename C> __device__ __forceinline__ C addi(C a, C b) { return C{a.x - b.y, a.y + b.x}; }  // a + i b
template <typename C> __device__ __forceinline__ C subi(C a, C b) { return C{a.x + b.y, a.y - b.x}; }  // a - i b

// square lattice, s = 4: the four outputs from the cells A = x-1, B = x+1, C = y-1, D = y+1
// (sources of h = +e1, -e1, +e2, -e2) and the own cell.  Every transition matrix is a column times
// a row (tables in stencil.cu), so a source enters through one number per spinor.  From its
// components a, b, c, d, with rho = 1 + i, rhob = 1 - i:
//   K1 = (a - i b)(A), K2 = (a + i b)(B), K3 = (a + i b)(C), K4 = (a - i b)(D),
//   L1 = (c - d)(A),   L2 = (c + d)(B),   L3 = (c - d)(C),   L4 = (c + d)(D),
//   S0 = rho [(K1 + K2) - i (K3 + K4)],  S1 = rho [(K1 - K2) - i (K3 - K4)],
//   S2 = rhob [(L1 + L2) + i (L3 + L4)], S3 = rho [(L2 - L1) - i (L4 - L3)]
// (48 real additions instead of 128 term by term, 40 where neighbours share the sources' numbers),
// then the mass step (finish).
template <typename C>
__device__ __forceinline__ void sums_2d(C K1, C K2, C K3, C K4, C L1, C L2, C L3, C L4, C (&S)[4]) {
  S[0] = rho(subi(cadd(K1, K2), cadd(K3, K4)));
  S[1] = rho(subi(csub(K1, K2), csub(K3, K4)));
  S[2] = rhob(addi(cadd(L1, L2), cadd(L3, L4)));
  S[3] = rho(subi(csub(L2, L1), csub(L4, L3)));
}

template <bool NC, typename C, typename CF, typename I>
__device__ __forceinline__ void core_2d(const C* sxm, const C* sxp, const C* sym, const C* syp, const C* own, I cs,
                                        C (&r)[4], const CF& cf) {
  const C A0 = ldg<NC>(sxm), A1 = ldg<NC>(sxm + cs), A2 = ldg<NC>(sxm + 2 * cs), A3 = ldg<NC>(sxm + 3 * cs);
  const C B0 = ldg<NC>(sxp), B1 = ldg<NC>(sxp + cs), B2 = ldg<NC>(sxp + 2 * cs), B3 = ldg<NC>(sxp + 3 * cs);
  const C C0 = ldg<NC>(sym), C1 = ldg<NC>(sym + cs), C2 = ldg<NC>(sym + 2 * cs), C3 = ldg<NC>(sym + 3 * cs);
  const C D0 = ldg<NC>(syp), D1 = ldg<NC>(syp + cs), D2 = ldg<NC>(syp + 2 * cs), D3 = ldg<NC>(syp + 3 * cs);
  C S[4];
  sums_2d(subi(A0, A1), addi(B0, B1), addi(C0, C1), subi(D0, D1), csub(A2, A3), cadd(B2, B3), csub(C2, C3),
          cadd(D2, D3), S);
  const C o0 = ldg<NC>(own), o1 = ldg<NC>(own + cs), o2 = ldg<NC>(own + 2 * cs), o3 = ldg<NC>(own + 3 * cs);
  r[0] = finish(cf, S[0], o2);
  r[1] = finish(cf, S[1], o3);
  r[2] = finish(cf, S[2], o0);
  r[3] = finish(cf, S[3], o1);
}

// site (x, y) of the N x N box
template <typename R, bool NC = true, typename I = int64_t>
__device__ __forceinline__ void site_update_2d(const typename CplxOf<R>::T* __restrict__ in,
                                               typename CplxOf<R>::T* __restrict__ out, I N, I x, I y,
                                               const typename CoefOf<R>::T& cf) {
  const I vol = N * N;
  const I xm = wrapm<I>(x - 1, N), xp = wrapm<I>(x + 1, N);
  const I ym = wrapm<I>(y - 1, N), yp = wrapm<I>(y + 1, N);
  const I i = y * N + x;
  typename CplxOf<R>::T r[4];
  core_2d<NC>(in + y * N + xm, in + y * N + xp, in + ym * N + x, in + yp * N + x, in + i, vol, r, cf);
#pragma unroll
  for (int q = 0; q < 4; ++q) out[i + q * vol] = r[q];
}

// BCC, s = 4: output coset c at cell (x, y, z) reads coset 1-c at (per axis) m - 1 + c for
// h = +1 and m + c for h = -1 (the site x - h of the other sublattice).  The transition matrices are
// products of one conditional shift per axis, so the sums factor axis by axis.  With sources
// a, b, c, d and rho = 1 + i, rhob = 1 - i:
//   upper spinor, per plane: X+- = a +- b at h_x = +-1; A = X+ + i X- of the row of h_y = +1,
//     B = X+ - i X- of the row of h_y = -1; S0 = rhob (A + i B) of the plane of h_z = +1,
//     S1 = rho (A - i B) of the plane of h_z = -1;
//   lower spinor, per column: V = c + i d of the row of h_y = +1, W = c - i d of the row of
//     h_y = -1, with c of the plane of h_z = -1 and d of the plane of h_z = +1;
//     G = rho (V - i W) of the column of h_x = +1, H = rhob (V + i W) of the column of h_x = -1;
//     S2 = H + G, S3 = H - G
// (52 real additions for a site on its own, 32 where neighbours share X, A, B, V, W, G, H as in
// qw_march.cuh, instead of 128 term by term), then the mass step (finish).
// src: component 0 of the other coset; (za, zb), (ya, yb), (xa, xb): its cells for h = +1 and
// h = -1 per axis, with pitches sz (z) and sy (y); own: component 0 of the own cell.
// PLANES: the loads plane by plane, a plane's together, so that a load from global memory waits on the ones before
// it only where it has to (a batch of per-site rounds on N = 32: 447 against 458 us for 50 steps); else in the order
// of use, with fewer values held, for tiles in shared memory (N = 64, eight steps FUSED: 46.5 against 49.8 us).
template <bool NC, bool PLANES = true, typename C, typename CF, typename I>
__device__ __forceinline__ void core_3d(const C* src, I sz, I sy, I za, I zb, I ya, I yb, I xa, I xb, I cs,
                                        const C* own, C (&r)[4], const CF& cf) {
  const C* app = src + za * sz + ya * sy + xa;  // plane of h_z = +1: (h_x, h_y) = (+, +)
  const C* apm = src + za * sz + yb * sy + xa;  // (+, -)
  const C* amp = src + za * sz + ya * sy + xb;  // (-, +)
  const C* amm = src + za * sz + yb * sy + xb;  // (-, -)
  const C* bpp = src + zb * sz + ya * sy + xa;  // plane of h_z = -1
  const C* bpm = src + zb * sz + yb * sy + xa;
  const C* bmp = src + zb * sz + ya * sy + xb;
  const C* bmm = src + zb * sz + yb * sy + xb;
  C S0, S1, G, H;
  if constexpr (PLANES) {
    const C a0 = ldg<NC>(app), b0 = ldg<NC>(app + cs), d0 = ldg<NC>(app + 3 * cs);
    const C a1 = ldg<NC>(apm), b1 = ldg<NC>(apm + cs), d1 = ldg<NC>(apm + 3 * cs);
    const C a2 = ldg<NC>(amp), b2 = ldg<NC>(amp + cs), d2 = ldg<NC>(amp + 3 * cs);
    const C a3 = ldg<NC>(amm), b3 = ldg<NC>(amm + cs), d3 = ldg<NC>(amm + 3 * cs);
    S0 = rhob(addi(addi(cadd(a0, b0), csub(a2, b2)), subi(cadd(a1, b1), csub(a3, b3))));
    const C e0 = ldg<NC>(bpp), f0 = ldg<NC>(bpp + cs), c0 = ldg<NC>(bpp + 2 * cs);
    const C e1 = ldg<NC>(bpm), f1 = ldg<NC>(bpm + cs), c1 = ldg<NC>(bpm + 2 * cs);
    const C e2 = ldg<NC>(bmp), f2 = ldg<NC>(bmp + cs), c2 = ldg<NC>(bmp + 2 * cs);
    const C e3 = ldg<NC>(bmm), f3 = ldg<NC>(bmm + cs), c3 = ldg<NC>(bmm + 2 * cs);
    S1 = rho(subi(addi(cadd(e0, f0), csub(e2, f2)), subi(cadd(e1, f1), csub(e3, f3))));
    G = rho(subi(addi(c0, d0), subi(c1, d1)));
    H = rhob(addi(addi(c2, d2), subi(c3, d3)));
  } else {
    auto xsum = [&](const C* p) { return cadd(ldg<NC>(p), ldg<NC>(p + cs)); };
    auto xdif = [&](const C* p) { return csub(ldg<NC>(p), ldg<NC>(p + cs)); };
    S0 = rhob(addi(addi(xsum(app), xdif(amp)), subi(xsum(apm), xdif(amm))));
    S1 = rho(subi(addi(xsum(bpp), xdif(bmp)), subi(xsum(bpm), xdif(bmm))));
    auto v = [&](const C* c, const C* d) { return addi(ldg<NC>(c + 2 * cs), ldg<NC>(d + 3 * cs)); };
    auto w = [&](const C* c, const C* d) { return subi(ldg<NC>(c + 2 * cs), ldg<NC>(d + 3 * cs)); };
    G = rho(subi(v(bpp, app), w(bpm, apm)));
    H = rhob(addi(v(bmp, amp), w(bmm, amm)));
  }
  const C o0 = ldg<NC>(own), o1 = ldg<NC>(own + cs), o2 = ldg<NC>(own + 2 * cs), o3 = ldg<NC>(own + 3 * cs);
  r[0] = finish(cf, S0, o2);
  r[1] = finish(cf, S1, o3);
  r[2] = finish(cf, cadd(H, G), o0);
  r[3] = finish(cf, csub(H, G), o1);
}

template <typename R, bool NC = true, typename I = int64_t>
__device__ __forceinline__ void site_update_3d(const typename CplxOf<R>::T* __restrict__ in,
                                               typename CplxOf<R>::T* __restrict__ out, I M, int c, I z, I y, I x,
                                               const typename CoefOf<R>::T& cf) {
  const I plane = M * M, vol = plane * M;
  const I xa = wrapm<I>(x - 1 + c, M), xb = wrapm<I>(x + c, M);
  const I ya = wrapm<I>(y - 1 + c, M), yb = wrapm<I>(y + c, M);
  const I za = wrapm<I>(z - 1 + c, M), zb = wrapm<I>(z + c, M);
  const I i = z * plane + y * M + x;
  typename CplxOf<R>::T r[4];
  core_3d<NC>(in + (I)(1 - c) * 4 * vol, plane, M, za, zb, ya, yb, xa, xb, vol, in + (I)c * 4 * vol + i, r, cf);
  typename CplxOf<R>::T* dst = out + (I)c * 4 * vol + i;
#pragma unroll
  for (int q = 0; q < 4; ++q) dst[q * vol] = r[q];
}

}  // namespace qw

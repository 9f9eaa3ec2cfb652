// Register-marching stencil kernels: several steps of the update rule (Eq. upd-rule) per pass
// over HBM, the field of every intermediate step held in registers.
//
// The Weyl part is the factored form of core_3d (qw_stencil_dev.cuh) in the same order, with X, A,
// B, V, W, G, H formed once per source and passed on: 32 real additions per site.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "qw_stencil_dev.cuh"

namespace qw {

__device__ __forceinline__ float2 shfl_c(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ double2 shfl_c(double2 v, int src) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// ---- the value of a site between two steps.  FP32: a register pair in one of two orders,
// (re, im) or (im, re), for the packed FP32 instructions (the rate per number of the scalar ones
// in half the issue slots).  The mass step of one component,
//   re = nq S.re - m o.im,  im = nq S.im + m o.re,
// pairs re with im when o is held in the order opposite to the result, so every step turns the
// order round (template parameter ORD) and no value is moved to swap its halves.
struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 pack2(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(F2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub2(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

template <int ORD> __device__ __forceinline__ F2 held(float2 v) { return ORD ? pack2(v.y, v.x) : pack2(v.x, v.y); }
template <int ORD> __device__ __forceinline__ double2 held(double2 v) { return v; }
template <int ORD> __device__ __forceinline__ float2 value(F2 a) {
  const float2 r = unpack2(a);
  return ORD ? make_float2(r.y, r.x) : r;
}
template <int ORD> __device__ __forceinline__ double2 value(double2 a) { return a; }

// The mass step (finish of qw_stencil_dev.cuh: the same products and sums in the same order) of a
// sum S held in order 1 - ORD and the partner component o held in order ORD.
struct CoefF2 {
  F2 nq_hi, nq_lo, m_hi[2], m_lo[2];  // m for o held as (re, im): (m, -m), as (im, re): (-m, m)
};
__device__ __forceinline__ CoefF2 spread(const Coef32& c) {
  return {pack2(c.nq_hi, c.nq_hi), pack2(c.nq_lo, c.nq_lo),
          {pack2(c.m_hi, -c.m_hi), pack2(-c.m_hi, c.m_hi)},
          {pack2(c.m_lo, -c.m_lo), pack2(-c.m_lo, c.m_lo)}};
}
__device__ __forceinline__ Coef64 spread(const Coef64& c) { return c; }
// The four components of a site; FP32 in passes over the coefficients, so that consecutive packed
// instructions share the coefficient register.
template <int ORD, typename CF>
__device__ __forceinline__ void finish4(const CF& c, const double2 (&s)[4], const double2 (&o)[4], double2 (&r)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) r[q] = finish(c, s[q], o[q ^ 2]);
}
template <int ORD, typename CF>
__device__ __forceinline__ void finish4(const CF& c, const F2 (&s)[4], const F2 (&o)[4], F2 (&r)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) r[q] = mul2(c.m_lo[ORD], o[q ^ 2]);
#pragma unroll
  for (int q = 0; q < 4; ++q) r[q] = fma2(c.nq_lo, s[q], r[q]);
#pragma unroll
  for (int q = 0; q < 4; ++q) r[q] = fma2(c.m_hi[ORD], o[q ^ 2], r[q]);
#pragma unroll
  for (int q = 0; q < 4; ++q) r[q] = fma2(c.nq_hi, s[q], r[q]);
}
template <typename R> struct HeldOf;
template <> struct HeldOf<float> { using T = F2; };
template <> struct HeldOf<double> { using T = double2; };

// One complex value from global to shared memory, asynchronously (8 or 16 bytes: element aligned).
template <typename C> __device__ __forceinline__ void cp_async_c(C* dst, const C* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src), "n"(sizeof(C))
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ------------------------------------------------------------------ BCC lattice
// The half-layers l = 2 z + c (coset c of layer z) are marched in order; half-layer l reads l - 1
// (h_z = +1) and l + 1 (h_z = -1) of the other coset.  A warp owns 32 KX cells along x (KX per
// lane) and KY rows, and the CTA's warps are stacked along y.  When half-layer l arrives at step
// level t, the level completes half-layer l - 1 of step t + 1, which is the arrival of level
// t + 1, and so on to level T, which is stored.  Neighbours along x come from the adjacent lanes
// by shuffle (one value per spinor), along y from the thread's own rows or, at the edge of a
// warp's rows, from the neighbouring warp through shared memory (one barrier per level).
// A tile is computed with the halo of its T steps (T physical sites per side), or, where the
// warp's cells (the CTA's rows) are exactly a period of the box, cyclically without one.
struct Tile3Geo {
  int M;           // cells per axis
  int perx, pery;  // cyclic tile along x / y
  int lanes;       // lanes in use (cyclic x tiles: M / KX, else 32)
  int tx, ty;      // cells a tile writes along x / y
};
template <typename C> struct March3 {
  const C* in[2][4];  // component planes of each coset
  C* out[2][4];
  Tile3Geo g;
  int ntx, nty;       // tiles
  // Which CTA marches which half-layers (march3_split): first `rounds` whole tiles per CTA; of the
  // `rest` tiles left, `per` CTAs each take `planes` half-layers per tile, and the CTAs beyond
  // those take `extra` half-layers each of what remains at the tiles' ends (tail per tile).
  int rounds, rest, per, planes, extra;
};

// Values of one step level that wait for the next arrivals: own = the last arrival; t0[u] = A + i B
// of the last arrival in a half iteration u, used by the next arrival of the same u; dprev = d of
// the arrival before the last.
template <typename R, int KX, int KY> struct Level3 {
  using C = typename CplxOf<R>::T;
  typename HeldOf<R>::T own[KY][KX][4];
  C t0[2][KY][KX], dprev[KY][KX];
};

// Arrival v of coset CO, held in order ORD, at a level (half iteration U); v becomes the completed
// half-layer of the next step, held in order 1 - ORD.  With SKIP only the rows of the mask are
// completed (one step per launch: no other row is used again).  xb: exchange rows of this level
// (2 KX x 32 values per warp).
template <int CO, int ORD, int U, bool SKIP, typename R, int KX, int KY, typename CF>
__device__ __forceinline__ void march3_arrive(Level3<R, KX, KY>& L, typename HeldOf<R>::T (&v)[KY][KX][4],
                                              typename CplxOf<R>::T* xb, int lane, int w, int wnb,
                                              unsigned rows, int sup, int sdn, const CF& cf) {
  using C = typename CplxOf<R>::T;
  using H = typename HeldOf<R>::T;
  constexpr int OC = 1 - CO;  // coset of the completed half-layer
  C A[KY][KX], B[KY][KX], V[KY][KX], W[KY][KX];
#pragma unroll
  for (int y = 0; y < KY; ++y) {
    C xp[KX], xm[KX];
#pragma unroll
    for (int k = 0; k < KX; ++k) {
      xp[k] = value<ORD>(add2(v[y][k][0], v[y][k][1]));
      xm[k] = value<ORD>(sub2(v[y][k][0], v[y][k][1]));
      const C c = value<ORD>(v[y][k][2]);
      V[y][k] = addi(c, L.dprev[y][k]);
      W[y][k] = subi(c, L.dprev[y][k]);
    }
    if constexpr (OC == 0) {  // X+ of cell x - 1
      const C e = shfl_c(xp[KX - 1], sup);
#pragma unroll
      for (int k = KX - 1; k > 0; --k) xp[k] = xp[k - 1];
      xp[0] = e;
    } else {  // X- of cell x + 1
      const C e = shfl_c(xm[0], sdn);
#pragma unroll
      for (int k = 0; k < KX - 1; ++k) xm[k] = xm[k + 1];
      xm[KX - 1] = e;
    }
#pragma unroll
    for (int k = 0; k < KX; ++k) {
      A[y][k] = addi(xp[k], xm[k]);
      B[y][k] = subi(xp[k], xm[k]);
    }
  }
  C* mine = xb + w * (2 * KX * 32) + lane;
  const C* nb = xb + wnb * (2 * KX * 32) + lane;
#pragma unroll
  for (int k = 0; k < KX; ++k) {
    mine[k * 32] = OC == 0 ? A[KY - 1][k] : B[0][k];
    mine[(KX + k) * 32] = OC == 0 ? V[KY - 1][k] : W[0][k];
  }
  __syncthreads();
  if constexpr (OC == 0) {  // A and V of row y - 1
#pragma unroll
    for (int k = 0; k < KX; ++k) {
#pragma unroll
      for (int y = KY - 1; y > 0; --y) {
        A[y][k] = A[y - 1][k];
        V[y][k] = V[y - 1][k];
      }
      A[0][k] = nb[k * 32];
      V[0][k] = nb[(KX + k) * 32];
    }
  } else {  // B and W of row y + 1
#pragma unroll
    for (int k = 0; k < KX; ++k) {
#pragma unroll
      for (int y = 0; y < KY - 1; ++y) {
        B[y][k] = B[y + 1][k];
        W[y][k] = W[y + 1][k];
      }
      B[KY - 1][k] = nb[k * 32];
      W[KY - 1][k] = nb[(KX + k) * 32];
    }
  }
#pragma unroll
  for (int y = 0; y < KY; ++y) {
    if (SKIP && !(rows >> y & 1u)) {  // not written: only what the next half-layers need
#pragma unroll
      for (int k = 0; k < KX; ++k) {
        L.dprev[y][k] = value<ORD>(L.own[y][k][3]);
        L.t0[U][y][k] = addi(A[y][k], B[y][k]);
#pragma unroll
        for (int q = 0; q < 4; ++q) L.own[y][k][q] = v[y][k][q];
      }
      continue;
    }
    C G[KX], Hh[KX];
#pragma unroll
    for (int k = 0; k < KX; ++k) {
      G[k] = rho(subi(V[y][k], W[y][k]));
      Hh[k] = rhob(addi(V[y][k], W[y][k]));
    }
    if constexpr (OC == 0) {  // G of cell x - 1
      const C e = shfl_c(G[KX - 1], sup);
#pragma unroll
      for (int k = KX - 1; k > 0; --k) G[k] = G[k - 1];
      G[0] = e;
    } else {  // H of cell x + 1
      const C e = shfl_c(Hh[0], sdn);
#pragma unroll
      for (int k = 0; k < KX - 1; ++k) Hh[k] = Hh[k + 1];
      Hh[KX - 1] = e;
    }
#pragma unroll
    for (int k = 0; k < KX; ++k) {
      H(&o)[4] = L.own[y][k];
      const H g = held<1 - ORD>(G[k]), h = held<1 - ORD>(Hh[k]);
      const H sum[4] = {held<1 - ORD>(rhob(L.t0[U][y][k])), held<1 - ORD>(rho(subi(A[y][k], B[y][k]))), add2(h, g),
                        sub2(h, g)};
      H r[4];
      finish4<ORD>(cf, sum, o, r);
      L.dprev[y][k] = value<ORD>(o[3]);
      L.t0[U][y][k] = addi(A[y][k], B[y][k]);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        o[q] = v[y][k][q];
        v[y][k][q] = r[q];
      }
    }
  }
}

// Levels LV .. T - 1 of one half-layer whose arrival at level 0 has coset C0.
template <int LV, int T, int C0, int U, typename R, int KX, int KY, typename CF>
__device__ __forceinline__ void march3_levels(Level3<R, KX, KY> (&L)[T], typename HeldOf<R>::T (&v)[KY][KX][4],
                                              typename CplxOf<R>::T* xch, int xsz, int lane, int w, int wup, int wdn,
                                              unsigned rows, int sup, int sdn, const CF& cf) {
  if constexpr (LV < T) {
    constexpr int CO = (C0 + LV) & 1;
    // exchange buffers alternate from one barrier to the next: a warp writes a buffer again only
    // after the following barrier, which every reader of its last contents has passed
    typename CplxOf<R>::T* xb = xch + ((U * T + LV) & 1) * xsz;
    march3_arrive<CO, (LV & 1), U, T == 1>(L[LV], v, xb, lane, w, CO == 1 ? wup : wdn, rows, sup, sdn, cf);
    march3_levels<LV + 1, T, C0, U>(L, v, xch, xsz, lane, w, wup, wdn, rows, sup, sdn, cf);
  }
}

constexpr int kMarch3Stages = 4;  // half-layers in flight per thread

template <typename R, int KX, int KY, int NW> constexpr int march3_smem() {
  return (int)sizeof(typename CplxOf<R>::T) * (kMarch3Stages * 4 * KX * KY * 32 * NW + 2 * 2 * KX * 32 * NW);
}

// The tile of NW warps of KX cells per lane and KY rows, T steps, on a box of M cells per axis.
__host__ __device__ inline Tile3Geo tile3_geo(int M, int kx, int ky, int t, int nw) {
  Tile3Geo g;
  g.M = M;
  g.perx = M <= 32 * kx && M % kx == 0;
  g.lanes = g.perx ? M / kx : 32;
  g.pery = nw * ky == M;
  g.tx = g.perx ? M : 32 * kx - t;
  g.ty = g.pery ? M : nw * ky - t;
  return g;
}

// Fill the split of p over `ctas` resident CTAs; returns the grid.  All CTAs walk whole tiles, or
// equal parts of them, at the same height, so that the halo a tile shares with its neighbours is
// read while it is in L2; only the CTAs that do not divide evenly take the tiles' ends.
template <typename C> inline int march3_split(March3<C>& p, int T, int ctas) {
  const int P = 2 * p.g.M, nt = p.ntx * p.nty;
  p.rounds = nt / ctas;
  p.rest = nt - p.rounds * ctas;
  p.per = p.planes = p.extra = 0;
  if (p.rest == 0) return ctas;
  p.per = ctas / p.rest < p.g.M ? ctas / p.rest : p.g.M;
  p.planes = 2 * ((p.g.M + p.per - 1) / p.per);
  const int help = ctas - p.rest * p.per;
  if (help > 0 && p.per < p.g.M) {
    // the longest even part of the main CTAs for which the helpers' load is no longer than theirs
    const int segs = (p.rest + help - 1) / help;
    for (int m = 2; m <= p.planes; m += 2) {
      const int64_t tail = P - (int64_t)p.per * m;
      if (tail <= 0) break;
      const int64_t ex = 2 * ((p.rest * (tail / 2) + help - 1) / help);
      if (ex + (segs + 1) * 2 * T <= m + 2 * T) {
        p.planes = m;
        p.extra = (int)ex;
        return ctas;
      }
    }
  }
  return p.rounds > 0 ? ctas : p.rest * p.per;
}

// Half-layers [ls, le) (ls even) of tile (itx, ity), T steps on from the field whose component q of
// coset c starts at in(c, q), to out(c, q).  All NW warps of the CTA; march_smem as march3_smem says.
// A component plane of a coset has M^3 < 2^32 cells (a field beyond that would not fit the device),
// so 32-bit indices on top of the planes' addresses: one instruction a load.
template <typename R, int KX, int KY, int T, int NW, bool EXACT, typename IN, typename OUT, typename CF>
__device__ __forceinline__ void march3_segment(const Tile3Geo& g, int itx, int ity, int ls, int le,
                                               unsigned char* march_smem, IN in, OUT out, const CF& cf) {
  using C = typename CplxOf<R>::T;
  using H = typename HeldOf<R>::T;
  constexpr int NT = 32 * NW, SLOT = 4 * KX * KY * NT;  // threads, values of one staged half-layer
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  C* const stage = reinterpret_cast<C*>(march_smem) + tid;  // [stage][q][ky][kx][thread]
  C* const xch = reinterpret_cast<C*>(march_smem) + kMarch3Stages * SLOT;
  const int M = g.M, P = 2 * M;
  const unsigned layer = (unsigned)M * M, zend = (unsigned)M * layer;
  const int sup = g.perx ? (lane == 0 ? g.lanes - 1 : lane - 1) : max(lane - 1, 0);
  const int sdn = g.perx ? (lane == g.lanes - 1 ? 0 : lane + 1) : min(lane + 1, 31);
  const int wup = w == 0 ? NW - 1 : w - 1, wdn = w == NW - 1 ? 0 : w + 1;
  // first cell of the tile's box: a halo of lo0 cells (coset 0) before the first written cell
  constexpr int lo0 = (T + 1) / 2, lo1 = T / 2;
  const int xb = g.perx ? 0 : itx * g.tx - lo0, yb = g.pery ? 0 : ity * g.ty - lo0;
  const int iters = le - ls + 2 * T;

  // cell indices in a layer, and which of them are written (bit per cell, by coset) and, with EXACT,
  // read: not those past what a short last tile needs, which another CTA may be writing (their values
  // reach no output)
  const int mx = g.perx ? M - 1 : min(g.tx, M - itx * g.tx) + T - 1;
  const int my = g.pery ? M - 1 : min(g.ty, M - ity * g.ty) + T - 1;
  unsigned off[KY][KX], rd = 0u, wr[2] = {0u, 0u}, wrow[2] = {0u, 0u};
#pragma unroll
  for (int y = 0; y < KY; ++y) {
    const int ly = w * KY + y;
    int gy = (yb + ly) % M;
    if (gy < 0) gy += M;
#pragma unroll
    for (int k = 0; k < KX; ++k) {
      const int lx = lane * KX + k;
      int gx = (xb + lx) % M;
      if (gx < 0) gx += M;
      off[y][k] = (unsigned)gy * M + gx;
      if (EXACT && lx <= mx && ly <= my) rd |= 1u << (y * KX + k);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int lo = c == 0 ? lo0 : lo1;
        const bool okx = g.perx ? lx < M : (lx >= lo && lx - lo < g.tx && itx * g.tx + lx - lo < M);
        const bool oky = g.pery ? ly < M : (ly >= lo && ly - lo < g.ty && ity * g.ty + ly - lo < M);
        if (okx && oky) wr[c] |= 1u << (y * KX + k);
        if (oky) wrow[c] |= 1u << y;
      }
    }
  }

  // half-layer ls - T + i is iteration i's arrival; its coset is that of T + i (ls is even)
  int lin = (ls - T) % P;
  if (lin < 0) lin += P;
  unsigned zin = (unsigned)(lin >> 1) * layer;  // first index of its layer
  int left = iters;
  // load the next half-layer, of coset CI, into slot
  auto issue = [&](auto coset, int slot) {
    constexpr int CI = decltype(coset)::value;
    if (left > 0) {
      C* d = stage + slot * SLOT;
#pragma unroll
      for (int y = 0; y < KY; ++y)
#pragma unroll
        for (int k = 0; k < KX; ++k)
          if (!EXACT || (rd >> (y * KX + k) & 1u)) {
#pragma unroll
            for (int q = 0; q < 4; ++q) cp_async_c(d + ((q * KY + y) * KX + k) * NT, in(CI, q) + (zin + off[y][k]));
          }
      if (CI == 1) {
        zin += layer;
        if (zin == zend) zin = 0;
      }
    }
    --left;
    cp_async_commit();
  };
  using Even = std::integral_constant<int, T & 1>;  // coset of iterations 0, 2, ...
  using Odd = std::integral_constant<int, (T + 1) & 1>;
  issue(Even(), 0);
  issue(Odd(), 1);
  issue(Even(), 2);
  static_assert(kMarch3Stages == 4, "three half-layers ahead");

  Level3<R, KX, KY> L[T];
#pragma unroll
  for (int t = 0; t < T; ++t)
#pragma unroll
    for (int y = 0; y < KY; ++y)
#pragma unroll
      for (int k = 0; k < KX; ++k) {
        L[t].t0[0][y][k] = L[t].t0[1][y][k] = L[t].dprev[y][k] = C{0, 0};
#pragma unroll
        for (int q = 0; q < 4; ++q) L[t].own[y][k][q] = held<0>(C{0, 0});
      }

  unsigned zout = (unsigned)(ls >> 1) * layer;  // layer being written
  int pair = 0;                                 // slots 0, 1 or 2, 3 hold this pair of arrivals
  for (int j = 0; j < iters; j += 2) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (u == 0)
        issue(Odd(), (pair ^ 2) + 1);
      else
        issue(Even(), pair);
      cp_async_wait<kMarch3Stages - 1>();
      const unsigned rows = j >= 2 * T ? wrow[u] : 0u;
      H v[KY][KX][4];
      const C* s = stage + (pair + u) * SLOT;
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int y = 0; y < KY; ++y)
#pragma unroll
          for (int k = 0; k < KX; ++k) v[y][k][q] = held<0>(s[((q * KY + y) * KX + k) * NT]);
      if (u == 0)
        march3_levels<0, T, (T & 1), 0>(L, v, xch, 2 * KX * NT, lane, w, wup, wdn, rows, sup, sdn, cf);
      else
        march3_levels<0, T, ((T + 1) & 1), 1>(L, v, xch, 2 * KX * NT, lane, w, wup, wdn, rows, sup, sdn, cf);
      if (j >= 2 * T) {  // half-layer ls + j + u - 2 T: coset u
#pragma unroll
        for (int y = 0; y < KY; ++y)
#pragma unroll
          for (int k = 0; k < KX; ++k)
            if (wr[u] >> (y * KX + k) & 1u) {
#pragma unroll
              for (int q = 0; q < 4; ++q) out(u, q)[zout + off[y][k]] = value<(T & 1)>(v[y][k][q]);
            }
        if (u == 1) zout += layer;
      }
    }
    pair ^= 2;
  }
}

template <typename R, int KX, int KY, int T, int NW, int CTAS>
__global__ void __launch_bounds__(32 * NW, CTAS)
    march3d_kernel(const __grid_constant__ March3<typename CplxOf<R>::T> p, const typename CoefOf<R>::T coef) {
  extern __shared__ __align__(16) unsigned char march_smem[];
  const auto cf = spread(coef);
  const int P = 2 * p.g.M;
  grid_wait();
  // the CTA's segments [ls, le) of a tile
  const int main_ctas = p.rest * p.per, b = blockIdx.x, tail = P - p.per * p.planes;
  int64_t pos = (int64_t)(b - main_ctas) * p.extra;  // in the remaining tiles' tails, one after another
  const int64_t end = min(pos + p.extra, (int64_t)p.rest * tail);
  for (int r = 0;; ++r) {
    int tile, ls, le;
    if (r < p.rounds) {
      tile = r * gridDim.x + b;
      ls = 0;
      le = P;
    } else if (b < main_ctas) {
      if (r > p.rounds) break;
      tile = p.rounds * gridDim.x + b % p.rest;
      ls = b / p.rest * p.planes;
      le = min(ls + p.planes, P);
      if (ls >= le) break;
    } else {
      if (pos >= end) break;
      const int t = (int)(pos / tail), o = (int)(pos - (int64_t)t * tail);
      tile = p.rounds * gridDim.x + t;
      ls = p.per * p.planes + o;
      le = (int)min((int64_t)P, ls + (end - pos));
      pos += le - ls;
    }
    march3_segment<R, KX, KY, T, NW, false>(
        p.g, tile % p.ntx, tile / p.ntx, ls, le, march_smem, [&](int c, int q) { return p.in[c][q]; },
        [&](int c, int q) { return p.out[c][q]; }, cf);
  }
}

}  // namespace qw

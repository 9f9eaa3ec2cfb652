// Register-marching kernel of the square lattice (complex64): several steps per pass over HBM (the
// update of core_2d, qw_stencil_dev.cuh, in the same order).
//
// A warp owns a strip of 32 KX columns (KX per lane) and marches along y.  When row r arrives at
// step level t, the level completes row r - 1 of step t + 1, which is the arrival of level t + 1,
// and so on to level T, which is stored.  Neighbours along x come from the adjacent lanes by shuffle
// (one number per spinor and side), the row below from the level's registers, so the warps need
// neither shared memory for the exchange nor a barrier.  A strip is computed with a halo of T
// columns per side, a chunk of rows with T rows per end.
#pragma once

#include "qw_march.cuh"

namespace qw {

struct March2 {
  const float2* in[4];
  float2* out[4];
  int N;
  int ntx;      // strips (of 32 KX - 2 T written columns)
  int rows;     // rows a warp writes
  int chunks;   // chunks of rows per strip
};

// own: the last arrival; k3, l3: (a + i b) and (c - d) of the arrival before it.
template <int KX> struct Level2 {
  F2 own[KX][4];
  float2 k3[KX], l3[KX];
};

// Arrival v, held in order ORD, at a level; v becomes the completed row of the next step, held in
// order 1 - ORD.
template <int ORD, int KX>
__device__ __forceinline__ void march2_arrive(Level2<KX>& L, F2 (&v)[KX][4], int up, int dn, const CoefF2& cf) {
  float2 m01[KX], p01[KX], m23[KX], p23[KX];  // of the row being completed
#pragma unroll
  for (int k = 0; k < KX; ++k) {
    const float2 a = value<ORD>(L.own[k][0]), b = value<ORD>(L.own[k][1]);
    m01[k] = subi(a, b);
    p01[k] = addi(a, b);
    m23[k] = value<ORD>(sub2(L.own[k][2], L.own[k][3]));
    p23[k] = value<ORD>(add2(L.own[k][2], L.own[k][3]));
  }
  const float2 mu = shfl_c(m01[KX - 1], up), du = shfl_c(m23[KX - 1], up);
  const float2 pd = shfl_c(p01[0], dn), sd = shfl_c(p23[0], dn);
#pragma unroll
  for (int k = 0; k < KX; ++k) {
    const float2 K1 = k > 0 ? m01[k > 0 ? k - 1 : 0] : mu, K2 = k < KX - 1 ? p01[k < KX - 1 ? k + 1 : 0] : pd;
    const float2 L1 = k > 0 ? m23[k > 0 ? k - 1 : 0] : du, L2 = k < KX - 1 ? p23[k < KX - 1 ? k + 1 : 0] : sd;
    const float2 K4 = subi(value<ORD>(v[k][0]), value<ORD>(v[k][1])), L4 = value<ORD>(add2(v[k][2], v[k][3]));
    float2 S[4];
    sums_2d(K1, K2, L.k3[k], K4, L1, L2, L.l3[k], L4, S);
    F2 s[4], r[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] = held<1 - ORD>(S[q]);
    finish4<ORD>(cf, s, L.own[k], r);
    L.k3[k] = p01[k];
    L.l3[k] = m23[k];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      L.own[k][q] = v[k][q];
      v[k][q] = r[q];
    }
  }
}

// One row through the levels: the arrival of a level is what the level before completed.
template <int LV, int T, int KX>
__device__ __forceinline__ void march2_levels(Level2<KX> (&lev)[T], F2 (&v)[KX][4], int up, int dn, const CoefF2& cf) {
  if constexpr (LV < T) {
    march2_arrive<LV & 1>(lev[LV], v, up, dn, cf);
    march2_levels<LV + 1, T>(lev, v, up, dn, cf);
  }
}

constexpr int kMarch2Stages = 4;  // rows in flight per warp

template <int KX, int NW> constexpr int march2_smem() { return 8 * kMarch2Stages * 4 * KX * 32 * NW; }

// Rows [ys, ye) of a strip by one warp (w of NW in the CTA), T steps on from the field whose component q
// starts at in(q), to out(q).  A component plane has N^2 < 2^32 sites: 32-bit indices.
template <int KX, int T, int NW, bool EXACT, typename IN, typename OUT>
__device__ __forceinline__ void march2_rows(int N, int strip, int ys, int ye, unsigned char* march_smem, IN in, OUT out,
                                            const CoefF2& cf) {
  constexpr int NT = 32 * NW, SLOT = 4 * KX * NT, TX = 32 * KX - 2 * T;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  // [stage][q][warp][column]: a row's columns are fetched 32 apart (whole sectors) and read KX
  // neighbours at a time
  float2* const stage = reinterpret_cast<float2*>(march_smem) + w * (32 * KX);
  const int iters = ye - ys + 2 * T;
  const int up = max(lane - 1, 0), dn = min(lane + 1, 31);

  // the columns the lane fetches (with EXACT, none past those a short last strip needs, which another
  // warp may be writing: their values reach no output), and those it owns
  const int mx = min(TX, N - strip * TX) + T - 1;
  unsigned fetch[KX], off[KX], rd = 0u, wr = 0u;
#pragma unroll
  for (int k = 0; k < KX; ++k) {
    int fx = (strip * TX + k * 32 + lane - T) % N;
    if (fx < 0) fx += N;
    fetch[k] = fx;
    if (EXACT && k * 32 + lane - T <= mx) rd |= 1u << k;
    const int lx = lane * KX + k - T;  // column relative to the strip's first written one
    int gx = (strip * TX + lx) % N;
    if (gx < 0) gx += N;
    off[k] = gx;
    if (lx >= 0 && lx < TX && strip * TX + lx < N) wr |= 1u << k;
  }
  int rin = (ys - T) % N;
  if (rin < 0) rin += N;
  unsigned yin = (unsigned)rin * N;
  const unsigned yend = (unsigned)N * N;
  int left = iters;
  auto issue = [&](int slot) {
    if (left > 0) {
      float2* d = stage + slot * SLOT;
#pragma unroll
      for (int k = 0; k < KX; ++k)
        if (!EXACT || (rd >> k & 1u)) {
#pragma unroll
          for (int q = 0; q < 4; ++q) cp_async_c(d + q * KX * NT + k * 32 + lane, in(q) + (yin + fetch[k]));
        }
      yin += N;
      if (yin == yend) yin = 0;
    }
    --left;
    cp_async_commit();
  };
#pragma unroll
  for (int s = 0; s < kMarch2Stages - 1; ++s) issue(s);

  Level2<KX> L[T];
  const F2 zero = pack2(0.f, 0.f);
#pragma unroll
  for (int t = 0; t < T; ++t)
#pragma unroll
    for (int k = 0; k < KX; ++k) {
      L[t].k3[k] = L[t].l3[k] = make_float2(0.f, 0.f);
#pragma unroll
      for (int q = 0; q < 4; ++q) L[t].own[k][q] = zero;
    }

  unsigned yout = (unsigned)ys * N;
  int slot = 0;
  // two rows per iteration: the registers of an arrival become the level's own row without moves
#pragma unroll 1
  for (int j = 0; j < iters; j += 2) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      issue((slot + u + kMarch2Stages - 1) & (kMarch2Stages - 1));
      cp_async_wait<kMarch2Stages - 1>();
      __syncwarp();
      F2 v[KX][4];
      const float2* s = stage + (slot + u) * SLOT;
      static_assert(KX == 2, "two columns per 16-byte load");
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 c = *reinterpret_cast<const float4*>(s + q * KX * NT + 2 * lane);
        v[0][q] = pack2(c.x, c.y);
        v[1][q] = pack2(c.z, c.w);
      }
      __syncwarp();
      march2_levels<0, T>(L, v, up, dn, cf);
      if (j + u >= 2 * T && j + u < iters) {
#pragma unroll
        for (int k = 0; k < KX; ++k)
          if (wr >> k & 1u) {
#pragma unroll
            for (int q = 0; q < 4; ++q) out(q)[yout + off[k]] = value<(T & 1)>(v[k][q]);
          }
        yout += N;
      }
    }
    slot ^= 2;
  }
}

template <int KX, int T, int NW, int CTAS>
__global__ void __launch_bounds__(32 * NW, CTAS) march2d_kernel(const __grid_constant__ March2 p, const Coef32 coef) {
  extern __shared__ __align__(16) unsigned char march_smem[];
  const CoefF2 cf = spread(coef);
  grid_wait();
  const int64_t item = (int64_t)blockIdx.x * NW + (threadIdx.x >> 5);
  if (item >= (int64_t)p.ntx * p.chunks) return;  // whole warps: nothing below meets another warp
  const int ys = (int)(item / p.ntx) * p.rows;
  march2_rows<KX, T, NW, false>(
      p.N, (int)(item % p.ntx), ys, min(ys + p.rows, p.N), march_smem, [&](int q) { return p.in[q]; },
      [&](int q) { return p.out[q]; }, cf);
}

}  // namespace qw

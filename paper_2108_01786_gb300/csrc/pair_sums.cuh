// Matrix-free sums of the periodic Cauchy kernel over the boundary nodes, in
// double-float, for the boundary velocity, the energy's stream function and the
// Plemelj boundary values: sum_{l != m} W_l G_ml, G_ml = 1/2 cot((zeta_l - zeta_m)/2).
//
// FP32 arithmetic bounds these sums (37e12 lane operations a second on the GB300,
// scalar or packed: a packed instruction takes the pipe for two cycles and saves
// only the issue slot), so what counts is the number of operations per pair: ~125
// here, ~190 and three branches in the general pair kernel.  A CTA takes one
// 32-node target tile and its eight warps the source tiles in turn (tiles never
// span two boundaries), two sources per thread in the lanes of df2:
// d = P_l Q_m - 1 as one combined product sum, i/d W accumulated as one product
// per component with 1/|d|^2, and the constant i/2 part of G from the tile's sum
// of weights.  Pairs with |d| < 0.1 take i/d = 1/R from the FP64 node difference
// (near_R), evaluated for both sources and the whole warp at once.  That is a chain
// of ~3500 cycles a pair, so the tiles whose boxes are closer than PSUM_GAP are left
// to a second pass in which the eight warps share each of them, two pairs per warp
// (one warp per close tile held its CTA for ~30 us).
#pragma once
#include "common.cuh"
#include "pair_kernel.cuh"
#include "df2.cuh"
#include "psum_index.h"

#define PSUM_WARPS 8
#define PSUM_THREADS (32 * PSUM_WARPS)
#define PSUM_TILE 32
#define PSUM_GAP 0.11f     // boxes further apart hold no |d| < 0.1 (FAST_GAP of the assembly)
#define PSUM_NEAR2 0.01f   // |d|^2 below which i/d comes from the node difference

struct PsumNodes {
  const float4* nP;       // e^{i zeta} (df complex)
  const float4* nQ;       // e^{-i zeta}
  const float4* nPQc;     // third words of P (x, y) and Q (z, w)
  const double2* z64;
  const float2* Tall;     // 1/2 cot(pi j / M_k) of every boundary, df
};

// acc + a b
__device__ __forceinline__ df2 d2_macc(df2 acc, df2 a, df2 b) {
  const float2 p = p_mul(a.hi, b.hi);
  float2 e = p_fma(a.hi, b.hi, p_neg(p));
  const df2 s = d2_two_sum(acc.hi, p);
  e = p_add(e, p_add(s.lo, acc.lo));
  e = p_fma(a.hi, b.lo, e);
  e = p_fma(a.lo, b.hi, e);
  return d2_fast_two_sum(s.hi, e);
}
__device__ __forceinline__ df2 d2_of(const float4& v) { return {f2(v.x, v.y), f2(v.z, v.w)}; }
__device__ __forceinline__ dfl d2_fold(df2 a) { return dfl{a.hi.x, a.lo.x} + dfl{a.hi.y, a.lo.y}; }

// box of a tile's nodes (centre and half-width in x, then y), by one warp
__device__ __forceinline__ float4 psum_box(double2 z) {
  const float x0 = __shfl_sync(0xffffffffu, (float)z.x, 0);
  const float dx = (float)z.x - x0, y = (float)z.y;
  float xl = dx, xh = dx, yl = y, yh = y;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    xl = fminf(xl, __shfl_xor_sync(0xffffffffu, xl, o));
    xh = fmaxf(xh, __shfl_xor_sync(0xffffffffu, xh, o));
    yl = fminf(yl, __shfl_xor_sync(0xffffffffu, yl, o));
    yh = fmaxf(yh, __shfl_xor_sync(0xffffffffu, yh, o));
  }
  return make_float4(x0 + 0.5f * (xl + xh), 0.5f * (xh - xl) + 1e-5f, 0.5f * (yl + yh), 0.5f * (yh - yl) + 1e-5f);
}
// boxes more than PSUM_GAP apart in x (periodically) or y
__device__ __forceinline__ bool psum_apart(const float4& u, const float4& v) {
  float dcx = v.x - u.x;
  dcx -= 6.2831853f * rintf(dcx * 0.15915494f);
  return fmaxf(fabsf(dcx) - u.y - v.y, fabsf(v.z - u.z) - u.w - v.w) > PSUM_GAP;
}

// tile t of the boundaries: its boundary, first node and node count
__host__ __device__ inline int psum_ntile(const Blocks& B) {
  int n = 0;
  for (int k = 0; k < B.nb; ++k) n += (B.M[k] + PSUM_TILE - 1) / PSUM_TILE;
  return n;
}
// tiles of the surface alone (the first ones)
inline int psum_ntile0(const Blocks& B) { return (B.M[0] + PSUM_TILE - 1) / PSUM_TILE; }
// Source splits (CTAs per target tile): about nine CTAs per SM (three resident),
// so that the last wave costs little, but a tile or more per warp
// (1472 x 2944 node pairs: 11 splits 52 us, 9 splits 58)
inline int psum_nsplit(int ntile_targets, int ntile) {
  const int n = (1368 + ntile_targets / 2) / ntile_targets, most = ntile / PSUM_WARPS;
  const int s = n < most ? n : most;
  return s > 1 ? s : 1;
}
#define PSUM_MAXTILES ((1 << 17) / PSUM_TILE + BIE_MAXB)   // of 2^17 nodes
__device__ __forceinline__ void psum_tile(const Blocks& B, int t, int& k, int& l0, int& n) {
  k = 0;
  int c = (B.M[0] + PSUM_TILE - 1) / PSUM_TILE;
  while (t >= c) {
    t -= c;
    ++k;
    c = (B.M[k] + PSUM_TILE - 1) / PSUM_TILE;
  }
  l0 = B.off[k] + t * PSUM_TILE;
  n = min(PSUM_TILE, B.M[k] - t * PSUM_TILE);
}

// One staged source tile per warp: pair p holds sources p and p + 16 in the two
// lanes (hi a, hi b, lo a, lo b)
template <int CW>   // weights per source (their sums are taken of the first two)
struct PsumStage {
  float4 Pr[16], Pi[16], Pc[16], W[CW][16];
};

// Stage sources l0 .. l0 + n - 1 (lanes past n repeat a real source with zero
// weight), by one warp; load_w(l, w) gives the CW weights of source l.
template <int CW, class F>
__device__ __forceinline__ void psum_stage(PsumStage<CW>& S, const PsumNodes& nd, int l0, int n, F load_w,
                                           dfl* wsum, float4& box) {
  const int lane = threadIdx.x & 31;
  const int l = l0 + min(lane, n - 1);
  dfl w[CW];
  load_w(l, w);
  const float4 p = nd.nP[l], c = nd.nPQc[l];
  box = psum_box(nd.z64[l]);
  const int k = lane & 15, h = lane >> 4;
  __syncwarp();   // the previous tile has been read
  float* a = reinterpret_cast<float*>(&S.Pr[k]);
  a[h] = p.x;
  a[2 + h] = p.y;
  a = reinterpret_cast<float*>(&S.Pi[k]);
  a[h] = p.z;
  a[2 + h] = p.w;
  a = reinterpret_cast<float*>(&S.Pc[k]);
  a[h] = c.x;
  a[2 + h] = c.y;
#pragma unroll
  for (int q = 0; q < CW; ++q) {
    if (lane >= n) w[q] = {0.f, 0.f};
    a = reinterpret_cast<float*>(&S.W[q][k]);
    a[h] = w[q].hi;
    a[2 + h] = w[q].lo;
    if (q < 2) wsum[q] = warp_sum(w[q]);
  }
  __syncwarp();
}

// The target's data: one target per lane
struct PsumTarget {
  df2 Qr, Qi, nQi;
  float2 Qcx, Qcy, nQcy;
  double2 z;
  __device__ __forceinline__ void load(const PsumNodes& nd, int m) {
    const float4 q = nd.nQ[m], c = nd.nPQc[m];
    Qr = {f2(q.x), f2(q.y)};
    Qi = {f2(q.z), f2(q.w)};
    nQi = d2_neg(Qi);
    Qcx = f2(c.z);
    Qcy = f2(c.w);
    nQcy = f2(-c.w);
    z = nd.z64[m];
  }
};

// i/d = 1/R for both sources of a pair and every lane of the warp; taken where
// na / nb: then (di + i dr) inv = 1/R = conj(R)/|R|^2
__device__ __forceinline__ void psum_near(double2 za, double2 zb, double2 zm, bool na, bool nb, df2& dr,
                                          df2& di, df2& inv) {
  const double2 a = node_delta(za, zm), b = node_delta(zb, zm);
  const dfl ax = df_from_double(a.x), ay = df_from_double(a.y), bx = df_from_double(b.x), by = df_from_double(b.y);
  const df2 Dr = {f2(ax.hi, bx.hi), f2(ax.lo, bx.lo)}, Di = {f2(ay.hi, by.hi), f2(ay.lo, by.lo)};
  const float ma = na ? fmaf(ax.hi, ax.hi, ay.hi * ay.hi) : 0.f, mb = nb ? fmaf(bx.hi, bx.hi, by.hi * by.hi) : 0.f;
  const float m2 = fmaxf(ma, mb);
  const unsigned full = 0xffffffffu;
  // terms of E(w) = (e^w - 1)/w for the largest |Delta| taken in the warp
  const int K = __any_sync(full, m2 >= 3.6e-3f) ? 11 : __any_sync(full, m2 >= 4e-4f) ? 9
                : __any_sync(full, m2 >= 1.6e-5f) ? 7 : 5;
  const df2 nDi = d2_neg(Di), nDr = d2_neg(Dr);   // w = i Delta = (-Di, Dr)
  float2 c = c_taylor_df[K];
  df2 Er = {f2(c.x), f2(c.y)}, Ei = {f2(0.f), f2(0.f)};
#pragma unroll 1
  for (int n = K - 1; n >= 0; --n) {
    c = c_taylor_df[n];
    const df2 tr = d2_dot2<true>(Er, nDi, Ei, nDr, f2(c.x), f2(c.y));
    Ei = d2_dot2<false>(Er, Dr, Ei, nDi, f2(0.f), f2(0.f));
    Er = tr;
  }
  const df2 Rr = d2_dot2<false>(Dr, Er, nDi, Ei, f2(0.f), f2(0.f));
  const df2 Ri = d2_dot2<false>(Dr, Ei, Di, Er, f2(0.f), f2(0.f));
  const df2 iv = d2_rcp(d2_dot2<false>(Rr, Rr, Ri, Ri, f2(0.f), f2(0.f)));
  if (na) {
    di.hi.x = Rr.hi.x;
    di.lo.x = Rr.lo.x;
    dr.hi.x = -Ri.hi.x;
    dr.lo.x = -Ri.lo.x;
    inv.hi.x = iv.hi.x;
    inv.lo.x = iv.lo.x;
  }
  if (nb) {
    di.hi.y = Rr.hi.y;
    di.lo.y = Rr.lo.y;
    dr.hi.y = -Ri.hi.y;
    dr.lo.y = -Ri.lo.y;
    inv.hi.y = iv.hi.y;
    inv.lo.y = iv.lo.y;
  }
}

// For pair p of the staged tile (sources la = l0 + p and la + 16) and this lane's
// target m: i/d = (di + i dr) inv; inv = 0 for the target itself.  `close` (the
// same in the whole warp): the tile may hold near pairs or the target.
template <class ST>
__device__ __forceinline__ void psum_pair(const ST& S, int p, const PsumNodes& nd, const PsumTarget& T,
                                          bool close, int l0, int n, int m, df2& dr, df2& di, df2& inv) {
  const df2 Pr = d2_of(S.Pr[p]), Pi = d2_of(S.Pi[p]);
  const float4 c4 = S.Pc[p];
  const float2 Pcx = f2(c4.x, c4.y), Pcy = f2(c4.z, c4.w);
  // third-word cross terms of P Q
  float2 cr = p_mul(Pr.hi, T.Qcx);
  cr = p_fma(Pi.hi, T.nQcy, cr);
  cr = p_fma(Pcx, T.Qr.hi, cr);
  cr = p_fma(Pcy, T.nQi.hi, cr);
  float2 ci = p_mul(Pr.hi, T.Qcy);
  ci = p_fma(Pi.hi, T.Qcx, ci);
  ci = p_fma(Pcx, T.Qi.hi, ci);
  ci = p_fma(Pcy, T.Qr.hi, ci);
  dr = d2_dot2<true>(Pr, T.Qr, Pi, T.nQi, f2(-1.f), cr);
  di = d2_dot2<false>(Pr, T.Qi, Pi, T.Qr, f2(0.f), ci);
  const df2 n2 = d2_dot2<false>(dr, dr, di, di, f2(0.f), f2(0.f));
  inv = d2_rcp(n2);
  if (!close) return;
  const int la = l0 + p, lb = la + 16;
  const bool na = n2.hi.x < PSUM_NEAR2, nb = n2.hi.y < PSUM_NEAR2;
  if (!__any_sync(0xffffffffu, na || nb)) return;
  // a lane past the tile's end repeats its last source: zero weight, so any finite value will do
  const bool ua = la == m || p >= n, ub = lb == m || p + 16 >= n;
  psum_near(nd.z64[min(la, l0 + n - 1)], nd.z64[min(lb, l0 + n - 1)], T.z, na && !ua, nb && !ub, dr, di, inv);
  if (ua) inv.hi.x = inv.lo.x = 0.f;
  if (ub) inv.hi.y = inv.lo.y = 0.f;
}

// What the second pass shares of a close tile
template <int CW>
struct PsumClose {
  dfl ws[CW];
  int t;
};

// The source tiles blockIdx.y PSUM_WARPS + warp, + gridDim.y PSUM_WARPS, ... of a CTA:
//   tile(t, kl, l0, n)      of source tile t (psum_tile)
//   stage(w, l0, n, ws)     stages it in slot w and gives the target's `close`
//   work(w, t, ws, p0, p1, close, own)  pairs p0 .. p1 - 1; own: add the tile's constants
template <int CW, class Stage, class Work>
__device__ __forceinline__ void psum_tiles(const Blocks& B, int ntile, PsumClose<CW>* sc, unsigned* mask,
                                           Stage stage, Work work) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int step = gridDim.y * PSUM_WARPS, t0 = blockIdx.y * PSUM_WARPS;
  const int nloc = ntile > t0 ? (ntile - t0 + step - 1) / step * PSUM_WARPS : 0;   // local index i: tile t0 + (i / 8) step + i % 8
  for (int i = threadIdx.x; i < (nloc + 31) / 32; i += blockDim.x) mask[i] = 0u;
  __syncthreads();
  for (int i = warp; i < nloc; i += PSUM_WARPS) {
    const int t = t0 + (i / PSUM_WARPS) * step + warp;
    if (t >= ntile) break;
    int kl, l0, n;
    psum_tile(B, t, kl, l0, n);
    dfl ws[CW];
    if (stage(warp, l0, n, ws)) {
      if (lane == 0) atomicOr(&mask[i >> 5], 1u << (i & 31));
      continue;
    }
    work(warp, kl, l0, n, ws, 0, 16, false, true);
  }
  __syncthreads();
  // close tiles, eight at a time in the order of their index
  int word = 0;
  unsigned bits = nloc > 0 ? mask[0] : 0u;
  const int nword = (nloc + 31) / 32;
  while (true) {
    int found = 0, mine = -1;
    while (found < PSUM_WARPS && word < nword) {   // the same walk in every thread
      if (!bits) {
        if (++word < nword) bits = mask[word];
        continue;
      }
      const int i = 32 * word + __ffs(bits) - 1;
      bits &= bits - 1;
      if (found == warp) mine = i;
      ++found;
    }
    if (found == 0) break;
    if (mine >= 0) {
      const int t = t0 + (mine / PSUM_WARPS) * step + mine % PSUM_WARPS;
      int kl, l0, n;
      psum_tile(B, t, kl, l0, n);
      dfl ws[CW];
      stage(warp, l0, n, ws);
      if (lane == 0) {
#pragma unroll
        for (int q = 0; q < CW; ++q) sc[warp].ws[q] = ws[q];
        sc[warp].t = t;
      }
    }
    __syncthreads();
    for (int f = 0; f < found; ++f) {
      int kl, l0, n;
      psum_tile(B, sc[f].t, kl, l0, n);
      dfl ws[CW];
#pragma unroll
      for (int q = 0; q < CW; ++q) ws[q] = sc[f].ws[q];
      const int per = 16 / PSUM_WARPS;
      work(f, kl, l0, n, ws, per * warp, per * warp + per, true, f == warp);
    }
    __syncthreads();
  }
}

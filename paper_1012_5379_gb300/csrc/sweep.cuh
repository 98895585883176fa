// The grid-wide sweep passes of the complex64 V-cycle: k_1..k_S of a GMRES(S) sweep and the
// Gram matrix of k_0..k_S from one read of R_0 (gram.cuh).
//
// A point of k_S depends on R_0 within S points in every direction, so a CTA forms k_j on
// its own points plus S - j points around them, redundantly with its neighbours, and no
// CTA waits for another.  In all three kernels a warp's 32 lanes are 32 neighbouring x
// positions, of which the inner 32 - 2S are the CTA's own: x neighbours come from shuffles
// or shared memory, and lanes at the rim hold values that are wrong beyond S - j points
// and are never used.  Outside the domain every value is zero without a test: R_0 is
// loaded as zero there and the 1D coefficients are zero.
#pragma once
#include <type_traits>

#include "gram.cuh"

namespace helm {

HELM_HD constexpr int sw_ox(int S) { return 32 - 2 * S; }  // own points of a warp row

// 1D coefficients of one axis position times the basis scale t (exact: a power of two).
struct SwCoef {
  float2 a, d, c;
};
__device__ __forceinline__ SwCoef sw_coef(const float2* ca, int i, int n, float t) {
  SwCoef r;
  r.a = r.d = r.c = make_float2(0.f, 0.f);
  if ((unsigned)i < (unsigned)n) {
    const float2 a = __ldg(ca + i), d = __ldg(ca + n + i), c = __ldg(ca + 2 * n + i);
    r.a = make_float2(a.x * t, a.y * t);
    r.d = make_float2(d.x * t, d.y * t);
    r.c = make_float2(c.x * t, c.y * t);
  }
  return r;
}

// ------------------------------------------------------------------ 2D
// A CTA of 8 warps holds a 32 x 8 QY region in registers, QY consecutive rows per warp;
// only the rows at a warp's edges pass through shared memory.  Its own points are the
// inner (32 - 2H) x (8 QY - 2H), H = S for a sweep from b and S + 1 for one from the residual
// of an iterate (one point more, as the fused pass forms that residual itself).
constexpr int SW2_NW = 8;
HELM_HD constexpr int sw2_own(int R, int H) { return R - 2 * H; }
HELM_HD inline int sw2_units(int H, int QY, int n) {
  return ceil_div(n, sw2_own(32, H)) * ceil_div(n, sw2_own(SW2_NW * QY, H));
}

template <int S, int QY>
struct Sw2Shared {
  float4 yac[SW2_NW * QY];                // y coefficients a, c of the region's rows
  float2 yd[SW2_NW * QY];
  float2 edge[2][SW2_NW + 2][2][32];      // [parity][warp + 1][first / last row][lane]
  float2 gs[(SW2_NW + 1) * gram_nv(S)];
  float2 wsum[SW2_NW * gram_ns(S)];
};

// A thread's place in its CTA's region and the stencil there (times the basis scale t).
template <int S, int QY>
struct Sw2Region {
  int n, P, H, x, y0, xr, yr, lane, warp, par;
  SwCoef cx;
  float ph[QY];
  Sw2Shared<S, QY>& sh;
  __device__ __forceinline__ Sw2Region(const LevelDev<float2>& L, int unit, int halo, Sw2Shared<S, QY>& shared)
      : sh(shared) {
    lane = threadIdx.x;
    warp = threadIdx.y;
    n = L.n;
    P = L.P;
    H = halo;
    par = 0;
    const float t = L.kt;
    const int ox = sw2_own(32, H), oy = sw2_own(SW2_NW * QY, H), ntx = ceil_div(n, ox);
    xr = (unit % ntx) * ox - H;
    yr = (unit / ntx) * oy - H;
    x = xr + lane;
    y0 = yr + warp * QY;
    cx = sw_coef(L.ca, x, n, t);
    const int tid = warp * 32 + lane;
    if (tid < SW2_NW * QY) {
      const SwCoef c = sw_coef(L.ca, yr + tid, n, t);
      sh.yac[tid] = make_float4(c.a.x, c.a.y, c.c.x, c.c.y);
      sh.yd[tid] = c.d;
    }
    if (warp < 2) {  // the rows beyond the region
      sh.edge[warp][0][1][lane] = make_float2(0.f, 0.f);
      sh.edge[warp][SW2_NW + 1][0][lane] = make_float2(0.f, 0.f);
    }
    const float phc = L.phir * t;
#pragma unroll
    for (int q = 0; q < QY; ++q)
      ph[q] = (L.phi && inside(x, y0 + q, 0, n)) ? __ldg(L.phi + pidx(x, y0 + q, 0, P)) * t : phc;
  }
  __device__ __forceinline__ bool own_row(int q) const {  // uniform over the warp
    const int ry = warp * QY + q;
    return ry >= H && ry < SW2_NW * QY - H && y0 + q < n;
  }
  __device__ __forceinline__ bool own_x() const { return lane >= H && lane < 32 - H && x < n; }
  // o = t (M - sg) v on the region (wrong one point further in from its rim each time); the
  // diagonal's term, the largest, is added last in every stencil: one rounding of its size
  __device__ __forceinline__ void apply(const float2 (&v)[QY], const float2 sg, float2 (&o)[QY]) {
    sh.edge[par][warp + 1][0][lane] = v[0];
    sh.edge[par][warp + 1][1][lane] = v[QY - 1];
    __syncthreads();
    const float2 up = sh.edge[par][warp][1][lane], dn = sh.edge[par][warp + 2][0][lane];
    par ^= 1;
#pragma unroll
    for (int q = 0; q < QY; ++q) {
      const float4 ac = sh.yac[warp * QY + q];
      float2 dg = cadd(cx.d, sh.yd[warp * QY + q]);
      dg.x = (dg.x - ph[q]) - sg.x;
      dg.y -= sg.y;
      float2 p = cmul(cx.a, shfl_up_c(v[q], 1));
      p = cfma(cx.c, shfl_down_c(v[q], 1), p);
      p = cfma(make_float2(ac.x, ac.y), q > 0 ? v[q > 0 ? q - 1 : 0] : up, p);
      p = cfma(make_float2(ac.z, ac.w), q < QY - 1 ? v[q < QY - 1 ? q + 1 : q] : dn, p);
      o[q] = cfma(dg, v[q], p);
    }
  }
  // k_1..k_S from k_0, the own points' k_j to p[j - 1] (j <= nstore), and the Gram matrix.
  __device__ __forceinline__ void sweep(const LevelDev<float2>& L, const float2 (&sg)[S], bool wide,
                                        float2 (&k)[S + 1][QY], float2* const* p, int nstore, int unit, int nunits) {
#pragma unroll
    for (int j = 0; j < S; ++j) apply(k[j], sg[j], k[j + 1]);
    const bool ownx = own_x();
    auto own_points = [&](auto sum) {
#pragma unroll
      for (int q = 0; q < QY; ++q) {
        if (!own_row(q) || !ownx) continue;
        float2 kk[S + 1];
#pragma unroll
        for (int j = 0; j <= S; ++j) kk[j] = k[j][q];
        sum(kk);
#pragma unroll
        for (int j = 1; j <= S; ++j)
          if (j <= nstore) p[j - 1][pidx(x, y0 + q, 0, P)] = kk[j];
      }
      pdl_trigger();  // the main work is done: let the next pass launch
    };
    float acc[gram_ns(S)];
#pragma unroll
    for (int i = 0; i < gram_ns(S); ++i) acc[i] = 0.f;
    if (wide) {
      float c[gram_ns(S)];
#pragma unroll
      for (int i = 0; i < gram_ns(S); ++i) c[i] = 0.f;
      own_points([&](const float2 (&kk)[S + 1]) { gram_point_wide<S>(kk, acc, c); });
      gram_block_sum_wide<S, SW2_NW>(acc, c, sh.wsum, sh.gs);
    } else {
      own_points([&](const float2 (&kk)[S + 1]) { gram_point<S>(kk, acc); });
      gram_block_sum<S, SW2_NW>(acc, sh.wsum, sh.gs);
    }
    gram_finish<S, SW2_NW>(L, sg, wide, unit, nunits, sh.gs);
  }
};

// W: whether the problems' levels are wide (their sums need more registers, so that is a kernel
// of its own), or W_ANY: each problem's own flag.
enum { W_NO, W_YES, W_ANY };
__device__ __forceinline__ bool wide_level(const LevelDev<float2>& L, int W) {
  return W == W_ANY ? L.wide != 0 : W == W_YES;
}

template <int S, int QY, int W>
__device__ __forceinline__ void sweep2_body(const LevelDev<float2>* __restrict__ levs, int nunits, int first,
                                            int store_last, int vblk, Sw2Shared<S, QY>& sh) {
  const int prob = vblk / nunits, unit = vblk - prob * nunits;
  const LevelDev<float2>& L = levs[prob];
  const bool wide = wide_level(L, W);
  Sw2Region<S, QY> G(L, unit, first ? S : S + 1, sh);
  pdl_wait();
  float2 sg[S];
  gram_shifts<S>(L, first != 0, wide, sg);
  const float2* R0 = first ? L.b : L.r0;
  float2 k[S + 1][QY];
#pragma unroll
  for (int q = 0; q < QY; ++q) k[0][q] = ldc<float2>(R0, G.x, G.y0 + q, 0, G.n, G.P);
  G.sweep(L, sg, wide, k, L.p, store_last ? S : S - 1, unit, nunits);
}
template <int S, int QY, int W>
__global__ void __launch_bounds__(256, 2)
k_sweep2(const LevelDev<float2>* __restrict__ levs, int nunits, int first, int store_last) {
  __shared__ Sw2Shared<S, QY> sh;
  sweep2_body<S, QY, W>(levs, nunits, first, store_last, blockIdx.x, sh);
}

// ------------------------------------------------------------------ 2D, fused V(1,1) passes
// A level of a V(1,1) cycle in two launches instead of five: the pass that sweeps also forms
// what it sweeps from, redundantly with its neighbours, so that the restriction, the coarse
// correction, its residual and the updates need no passes and no vectors of their own.
// Levels of this size live in L2 and a chained pass takes about 3 us whatever its size (5 to 6
// with the Gram reduction), so launches are what they cost: 127^2 14 launches, 67.7 us, before
// and 7, 53 us, now; 639^2 164 -> 121, 1023^2 209 -> 159.  Larger levels (the line of the
// marching sweep) keep passes of their own: rereading a region's rim costs them more than a
// launch (4095^2, s = 4: 4.3 ms fused, 3.1 ms apart).  The values are the separate passes', in
// the same order of operations.
//
// Descent: b = full weighting of the finer level's residual sum_k rho_k k_k (its last sweep),
// which a lane forms for its column from two fine columns, the third being its neighbour's
// first.  A problem whose finest level this is takes b as given.
template <int S, int QY, int WIDE>
__global__ void __launch_bounds__(256, 2)
k_sweep2_down(const LevelDev<float2>* __restrict__ levs, int nunits) {
  __shared__ Sw2Shared<S, QY> sh;
  const int prob = blockIdx.x / nunits, unit = blockIdx.x - prob * nunits;
  const LevelDev<float2>& L = levs[prob];
  Sw2Region<S, QY> W(L, unit, S, sh);
  pdl_wait();
  float2 sg[S];
  gram_shifts<S>(L, true, WIDE, sg);
  float2 k[S + 1][QY];
  if (L.top) {
#pragma unroll
    for (int q = 0; q < QY; ++q) k[0][q] = ldc(L.b, W.x, W.y0 + q, 0, W.n, W.P);
  } else {
    const int nf = 2 * W.n + 1, Pf = nf + 1, m = L.scf->m, f0 = 2 * W.y0;
    float2 rc[S + 1];
    const float2* R[S + 1];
#pragma unroll
    for (int j = 0; j <= S; ++j) {
      rc[j] = L.scf->rcoef[j];
      R[j] = j == 0 ? L.fb : L.fp[j > 0 ? j - 1 : 0];
    }
    // the column right of lane 31's pair: lane i takes fine row f0 + i
    float2 er = make_float2(0.f, 0.f);
    {
      const int ec = 2 * (W.xr + 32), er_row = f0 + W.lane;
      const bool ok = W.lane <= 2 * QY && (unsigned)er_row < (unsigned)nf && (unsigned)ec < (unsigned)Pf;
#pragma unroll
      for (int j = 0; j <= S; ++j)
        {
          const float2 v = ok ? R[j][(size_t)er_row * Pf + ec] : make_float2(0.f, 0.f);
          if (j <= m) er = cfma(rc[j], v, er);
        }
    }
    const int fc = 2 * W.x;
    const bool colok = (unsigned)fc < (unsigned)Pf;  // a pair: Pf and fc are even
    float2 out[QY];
#pragma unroll
    for (int q = 0; q < QY; ++q) out[q] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i <= 2 * QY; ++i) {
      const int f = f0 + i;
      const bool ok = colok && (unsigned)f < (unsigned)nf;
      float2 r0 = make_float2(0.f, 0.f), r1 = r0;
#pragma unroll
      for (int j = 0; j <= S; ++j) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ok) v = *reinterpret_cast<const float4*>(R[j] + (size_t)f * Pf + fc);  // not after m: its load is in flight
        if (j <= m) {  // uniform
          r0 = cfma(rc[j], make_float2(v.x, v.y), r0);
          r1 = cfma(rc[j], make_float2(v.z, v.w), r1);
        }
      }
      const float2 rn = shfl_down_c(r0, 1);
      const float2 re = make_float2(__shfl_sync(0xffffffffu, er.x, i), __shfl_sync(0xffffffffu, er.y, i));
      const float2 r2 = W.lane == 31 ? re : rn;
#pragma unroll
      for (int q = 0; q < QY; ++q) {
        if (i < 2 * q || i > 2 * q + 2) continue;
        const float w = i == 2 * q + 1 ? 0.125f : 0.0625f;
        out[q] = cadd(out[q], cscale(r0, w));
        out[q] = cadd(out[q], cscale(r1, 2.0f * w));
        out[q] = cadd(out[q], cscale(r2, w));
      }
    }
#pragma unroll
    for (int q = 0; q < QY; ++q) {
      k[0][q] = inside(W.x, W.y0 + q, 0, W.n) ? out[q] : make_float2(0.f, 0.f);
      if (W.own_row(q) && W.own_x()) L.b[pidx(W.x, W.y0 + q, 0, W.P)] = k[0][q];
    }
  }
  W.sweep(L, sg, WIDE, k, L.p, S, unit, nunits);
}

// Coarse points around a 32 x R region of fine points: the coarser level's output there, its
// last sweep's update included if that has no pass of its own (L.cr0), to es.
template <int S>
__device__ __forceinline__ float2 coarse_value(const LevelDev<float2>& L, const float2 (&yc)[S], int mc, int X, int Y) {
  if ((unsigned)X >= (unsigned)L.nc || (unsigned)Y >= (unsigned)L.nc) return make_float2(0.f, 0.f);
  const size_t i = (size_t)Y * L.Pc + X;
  const float2 xv = L.xcb[i];
  if (!L.cr0) return xv;
  float2 dx = make_float2(0.f, 0.f);
#pragma unroll
  for (int j = 0; j < S; ++j)
  {
    const float2 v = j == 0 ? L.cr0[i] : L.cp[j > 0 ? j - 1 : 0][i];
    if (j < mc) dx = cfma(yc[j], v, dx);
  }
  return cadd(xv, dx);
}
template <int S>
__device__ __forceinline__ int coarse_update(const LevelDev<float2>& L, float2 (&yc)[S]) {
#pragma unroll
  for (int j = 0; j < S; ++j) yc[j] = L.cr0 ? L.scc->xcoef[j] : make_float2(0.f, 0.f);
  return L.cr0 ? L.scc->m : 0;
}
// Bilinear interpolation from rows of staged coarse values at fine (x, y), (X0, Y0) the first.
template <int EX>
__device__ __forceinline__ float2 staged_interp(const float2 (*es)[EX], int X0, int Y0, int x, int y) {
  const int X = (x >> 1) - X0, Y = (y >> 1) - Y0;
  float2 a = make_float2(0.f, 0.f);
  float w = 1.0f;
  if (!(x & 1)) w *= 0.5f;
  if (!(y & 1)) {
    w *= 0.5f;
    if (!(x & 1)) a = cadd(a, es[Y - 1][X - 1]);
    a = cadd(a, es[Y - 1][X]);
  }
  if (!(x & 1)) a = cadd(a, es[Y][X - 1]);
  a = cadd(a, es[Y][X]);
  return cscale(a, w);
}

// Ascent: x_b = sum_k y_k k_k + P e_c (the pre-smoothing sweep from b, and the corrected
// coarser output), R_0 = b - M x_b, and the sweep from it.  The new vectors go to L.q: other
// CTAs still read the old ones.
template <int S, int QY, int WIDE>
__global__ void __launch_bounds__(256, 2)
k_sweep2_up(const LevelDev<float2>* __restrict__ levs, int nunits) {
  constexpr int EX = 18, EY = SW2_NW * QY / 2 + 2;
  __shared__ Sw2Shared<S, QY> sh;
  __shared__ float2 es[EY][EX];
  const int prob = blockIdx.x / nunits, unit = blockIdx.x - prob * nunits;
  const LevelDev<float2>& L = levs[prob];
  Sw2Region<S, QY> W(L, unit, S + 1, sh);
  pdl_wait();
  const int m = L.sc->m;
  float2 xc[S], yc[S], sg[S];
#pragma unroll
  for (int j = 0; j < S; ++j) xc[j] = L.sc->xcoef[j];
  const int mc = coarse_update<S>(L, yc);
  gram_shifts<S>(L, false, WIDE, sg);
  float2 b[QY], dx[QY];
#pragma unroll
  for (int q = 0; q < QY; ++q) {
    const bool in = inside(W.x, W.y0 + q, 0, W.n);
    const size_t i = pidx(W.x, W.y0 + q, 0, W.P);
    b[q] = in ? L.b[i] : make_float2(0.f, 0.f);
    dx[q] = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < S; ++j)
    {  // loaded whatever m is: m's own load is in flight
      const float2 v = j == 0 ? b[q] : in ? L.p[j > 0 ? j - 1 : 0][i] : make_float2(0.f, 0.f);
      if (j < m) dx[q] = cfma(xc[j], v, dx[q]);
    }
  }
  const int X0 = (W.xr >> 1) - 1, Y0 = (W.yr >> 1) - 1;
  for (int i = W.warp * 32 + W.lane; i < EX * EY; i += 256)
    es[i / EX][i % EX] = coarse_value<S>(L, yc, mc, X0 + i % EX, Y0 + i / EX);
  __syncthreads();
  float2 v[QY], k[S + 1][QY];
#pragma unroll
  for (int q = 0; q < QY; ++q) {
    v[q] = make_float2(0.f, 0.f);
    if (inside(W.x, W.y0 + q, 0, W.n)) v[q] = cadd(dx[q], staged_interp<EX>(es, X0, Y0, W.x, W.y0 + q));
  }
  W.apply(v, make_float2(0.f, 0.f), k[0]);
  const float it = __frcp_rn(L.kt);  // exact
#pragma unroll
  for (int q = 0; q < QY; ++q) {
    k[0][q] = csub(b[q], cscale(k[0][q], it));
    if (W.own_row(q) && W.own_x()) {
      const size_t i = pidx(W.x, W.y0 + q, 0, W.P);
      L.xb[i] = v[q];
      L.r0[i] = k[0][q];
    }
  }
  W.sweep(L, sg, WIDE, k, L.q, S - 1, unit, nunits);
}

// Coarse correction and residual of a larger level (the sweep after it marches), 64 x 16 tiles:
// x_a from the last sweep if the restriction was fused (xk), else as stored.
template <int S>
__global__ void __launch_bounds__(256, 5)  // 4095^2: 150 us, 157 at three
k_prolong2_gram(const LevelDev<float2>* __restrict__ levs, int ntiles, int xk) {
  constexpr int TX = 64, TY = 16, EX = TX / 2 + 2, EY = TY / 2 + 2;
  __shared__ float2 es[EY][EX];
  __shared__ float2 vt[TY + 2][TX + 2];
  const int prob = blockIdx.x / ntiles, tile = blockIdx.x - prob * ntiles;
  const LevelDev<float2>& L = levs[prob];
  const int n = L.n, P = L.P, ntx = ceil_div(P, TX);
  const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
  const int lx = threadIdx.x, ly = threadIdx.y, tid = ly * 32 + lx;
  pdl_wait();
  const int m = L.sc->m;
  float2 xc[S], yc[S];
#pragma unroll
  for (int j = 0; j < S; ++j) xc[j] = L.sc->xcoef[j];
  const int mc = coarse_update<S>(L, yc);
  const int X0 = x0 / 2 - 1, Y0 = y0 / 2 - 1;
  for (int i = tid; i < EX * EY; i += 256)
    es[i / EX][i % EX] = coarse_value<S>(L, yc, mc, X0 + i % EX, Y0 + i / EX);
  auto before = [&](int x, int y, float2& b) {  // x_a and b
    const bool in = inside(x, y, 0, n);
    const size_t i = pidx(x, y, 0, P);
    b = in ? L.b[i] : make_float2(0.f, 0.f);
    if (!xk) return in ? L.xa[i] : make_float2(0.f, 0.f);
    float2 d = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < S; ++j)
      {
        const float2 v = j == 0 ? b : in ? L.p[j > 0 ? j - 1 : 0][i] : make_float2(0.f, 0.f);
        if (j < m) d = cfma(xc[j], v, d);
      }
    return d;
  };
  float2 bq[4], xv[4], hv = make_float2(0.f, 0.f);
#pragma unroll
  for (int q = 0; q < 4; ++q) xv[q] = before(x0 + lx + 32 * (q & 1), y0 + ly + 8 * (q >> 1), bq[q]);
  int hx = 0, hy = 0;
  const bool halo = tid < 2 * (TX + TY);  // the tile's rim, corners excepted
  if (halo) {
    if (tid < 2 * TX) {
      hx = tid % TX;
      hy = tid < TX ? -1 : TY;
    } else {
      hx = tid - 2 * TX < TY ? -1 : TX;
      hy = (tid - 2 * TX) % TY;
    }
    float2 b;
    hv = before(x0 + hx, y0 + hy, b);
  }
  __syncthreads();
  auto value = [&](float2 xa, int x, int y) {
    return inside(x, y, 0, n) ? cadd(xa, staged_interp<EX>(es, X0, Y0, x, y)) : make_float2(0.f, 0.f);
  };
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int ox = lx + 32 * (q & 1), oy = ly + 8 * (q >> 1);
    vt[oy + 1][ox + 1] = value(xv[q], x0 + ox, y0 + oy);
  }
  if (halo) vt[hy + 1][hx + 1] = value(hv, x0 + hx, y0 + hy);
  __syncthreads();
  const SwCoef cx[2] = {sw_coef(L.ca, x0 + lx, n, 1.0f), sw_coef(L.ca, x0 + lx + 32, n, 1.0f)};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int ox = lx + 32 * (q & 1), oy = ly + 8 * (q >> 1), x = x0 + ox, y = y0 + oy;
    if (x >= n || y >= n) continue;  // the ghost row and column stay zero
    const SwCoef cy = sw_coef(L.ca, y, n, 1.0f);
    const size_t i = pidx(x, y, 0, P);
    float2 dg = cadd(cx[q & 1].d, cy.d);
    dg.x -= L.phi ? __ldg(L.phi + i) : L.phir;
    float2 p = cmul(cx[q & 1].a, vt[oy + 1][ox]);
    p = cfma(cx[q & 1].c, vt[oy + 1][ox + 2], p);
    p = cfma(cy.a, vt[oy][ox + 1], p);
    p = cfma(cy.c, vt[oy + 2][ox + 1], p);
    p = cfma(dg, vt[oy + 1][ox + 1], p);
    L.xb[i] = vt[oy + 1][ox + 1];
    L.r0[i] = csub(bq[q], p);
  }
  pdl_trigger();
}

// ------------------------------------------------------------------ 2D, large levels
// Every warp marches in y on its own 64-column strip, two neighbouring columns per lane (own:
// the inner 56): x neighbours by shuffle, y neighbours in registers (four rows of each
// vector), rows of R_0 loaded four steps ahead; no barrier and no shared vector.  In the step
// that takes row y of R_0 it forms k_j of row y - j for every j.  A CTA's four warps take
// neighbouring strips of one chunk of `rows` rows and share its y coefficients.
// Bound by instruction issue (68% active, 192 lane instructions a point, 16 warps per SM at
// 128 registers).  4095^2, s = 3: 129 us a sweep, 3.7 TB/s; a register-region kernel like the
// one above with 8 rows per warp took 303 us (259 instructions a point, 45% issue: its
// barriers and exposed loads).
constexpr int SV2_NW = 4, SV2_OX = 56;
HELM_HD inline int sv2_groups(int n) { return ceil_div(ceil_div(n, SV2_OX), SV2_NW); }
HELM_HD inline int sv2_units(int n, int rows) { return sv2_groups(n) * ceil_div(n, rows); }
HELM_HD constexpr unsigned sv2_smem(int S, int rows) { return (unsigned)(rows + 2 * S) * 24u; }

template <int S, bool PHI>
__global__ void __launch_bounds__(SV2_NW * 32, 4)
k_sweep2_march(const LevelDev<float2>* __restrict__ levs, int nunits, int rows, int first, int store_last) {
  constexpr int NS = gram_ns(S), NV = gram_nv(S), W = 4;
  static_assert(S <= 3, "register windows hold four rows");
  extern __shared__ __align__(16) float2 swsm[];
  __shared__ float2 wsum[SV2_NW * NS];
  __shared__ float2 gs[(SV2_NW + 1) * NV];
  const int prob = blockIdx.x / nunits, unit = blockIdx.x - prob * nunits;
  const LevelDev<float2>& L = levs[prob];
  const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
  const int n = L.n, P = L.P;
  const float t = L.kt, phir = L.phir, phc = phir * t;
  const float* const phi = L.phi;
  const int ng = sv2_groups(n);
  const int x = ((unit % ng) * SV2_NW + warp) * SV2_OX - 4 + 2 * lane;  // columns x, x + 1
  const int yb = (unit / ng) * rows, ye = min(yb + rows, n);
  float4* const yac = reinterpret_cast<float4*>(swsm);
  float2* const yd = reinterpret_cast<float2*>(yac + rows + 2 * S);
  const SwCoef cx[2] = {sw_coef(L.ca, x, n, t), sw_coef(L.ca, x + 1, n, t)};
  for (int i = tid; i < ye - yb + 2 * S; i += SV2_NW * 32) {
    const SwCoef c = sw_coef(L.ca, yb - S + i, n, t);
    yac[i] = make_float4(c.a.x, c.a.y, c.c.x, c.c.y);
    yd[i] = c.d;
  }
  pdl_wait();
  __syncthreads();
  float2 sg[S];
  gram_shifts<S>(L, first != 0, false, sg);
  const float2* R0 = first ? L.b : L.r0;
  const bool in = (unsigned)x < (unsigned)P;  // the pair lies in the row (P is even, x too)
  float2 win[S][W][2];  // k_j of the last rows, slot = step & 3
#pragma unroll
  for (int j = 0; j < S; ++j)
#pragma unroll
    for (int w = 0; w < W; ++w) win[j][w][0] = win[j][w][1] = make_float2(0.f, 0.f);
  float phw[W][2] = {};
  float4 nxt[W];
  float2 phn[W];
  auto fetch = [&](int y, float4& v, float2& f) {
    const bool ok = in && (unsigned)y < (unsigned)n;
    v = ok ? *reinterpret_cast<const float4*>(R0 + (size_t)y * P + x) : make_float4(0.f, 0.f, 0.f, 0.f);
    if (PHI)  // some problem of the launch has a field; this one may not
      f = (ok && phi) ? __ldg(reinterpret_cast<const float2*>(phi + (size_t)y * P + x)) : make_float2(phir, phir);
  };
  float acc[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) acc[i] = 0.f;
  const bool own = lane >= 2 && lane < 30 && x < n;
  const int yf = yb - S, steps = ye - yb + 2 * S;
#pragma unroll
  for (int u = 0; u < W; ++u) fetch(u < steps ? yf + u : -1, nxt[u], phn[u]);
#pragma unroll 1
  for (int i0 = 0; i0 < steps; i0 += W) {
#pragma unroll
    for (int u = 0; u < W; ++u) {
      const int i = i0 + u;
      if (i >= steps) break;  // uniform
      const int y = yf + i;
      win[0][u][0] = make_float2(nxt[u].x, nxt[u].y);
      win[0][u][1] = make_float2(nxt[u].z, nxt[u].w);
      if (PHI) {
        phw[u][0] = phn[u].x * t;
        phw[u][1] = phn[u].y * t;
      }
      if (i + W < steps) fetch(y + W, nxt[u], phn[u]);
      float2 last[2];
#pragma unroll
      for (int j = 1; j <= S; ++j) {
        // k_j at row y - j from k_{j-1} at rows y - j - 1 .. y - j + 1
        const int c = (u - j) & 3, b = (u - j - 1) & 3, f = (u - j + 1) & 3;
        float2 r[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        if (i >= j) {  // uniform
          const float4 ya = yac[i - j];
          const float2 ydd = yd[i - j];
          const float2 v0 = win[j - 1][c][0], v1 = win[j - 1][c][1];
          const float2 vl = shfl_up_c(v1, 1), vr = shfl_down_c(v0, 1);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            float2 dg = cadd(cx[q].d, ydd);
            dg.x = (dg.x - (PHI ? phw[c][q] : phc)) - sg[j - 1].x;
            dg.y -= sg[j - 1].y;
            float2 p = cmul(make_float2(ya.x, ya.y), win[j - 1][b][q]);
            p = cfma(make_float2(ya.z, ya.w), win[j - 1][f][q], p);
            p = cfma(cx[q].a, q ? v0 : vl, p);
            p = cfma(cx[q].c, q ? vr : v1, p);
            r[q] = cfma(dg, q ? v1 : v0, p);
          }
        }
        if (j < S) {
          win[j][c][0] = r[0];
          win[j][c][1] = r[1];
        } else {
          last[0] = r[0];
          last[1] = r[1];
        }
      }
      if (i >= 2 * S && own) {
        const int c = (u - S) & 3;
        const size_t at = (size_t)(y - S) * P + x;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          float2 kk[S + 1];
#pragma unroll
          for (int j = 0; j < S; ++j) kk[j] = win[j][c][q];
          kk[S] = last[q];
          gram_point<S>(kk, acc);
        }
#pragma unroll
        for (int j = 1; j <= S; ++j)
          if (j < S || store_last) {
            const float2 a = j < S ? win[j < S ? j : 0][c][0] : last[0], b = j < S ? win[j < S ? j : 0][c][1] : last[1];
            *reinterpret_cast<float4*>(L.p[j - 1] + at) = make_float4(a.x, a.y, b.x, b.y);
          }
      }
    }
  }
  pdl_trigger();  // the main work is done: let the next pass launch
  gram_block_sum<S, SV2_NW>(acc, wsum, gs);
  gram_finish<S, SV2_NW>(L, sg, false, unit, nunits, gs);
}

// ------------------------------------------------------------------ 3D, small levels
// A CTA of 8 warps owns (32 - 2S) x O x O points and keeps k_0..k_{S-1} on the region
// around them in shared memory, one warp per (y, z) row at a time.  Every row of a stage is
// independent, so a level of a few thousand points finishes in S short stages.
constexpr int SW3_NW = 8;
HELM_HD inline int sw3_units(int S, int O, int n) {
  return ceil_div(n, sw_ox(S)) * ceil_div(n, O) * ceil_div(n, O);
}
HELM_HD constexpr int sw3_rows(int S, int O) {
  int r = 0;
  for (int j = 0; j < S; ++j) r += (O + 2 * S - 2 * j) * (O + 2 * S - 2 * j);
  return r;
}
HELM_HD constexpr unsigned sw3_smem(int S, int O) { return (unsigned)sw3_rows(S, O) * 256u; }

template <int S, int O, int J>
__device__ __forceinline__ int sw3_base() {  // first row of k_J in the shared array
  int r = 0;
#pragma unroll
  for (int j = 0; j < J; ++j) r += (O + 2 * S - 2 * j) * (O + 2 * S - 2 * j);
  return r;
}

// Row (ry, rz) of stage J (its region O + 2 (S - J) rows wide) of the basis.
template <int S, int O, int J>
__device__ __forceinline__ float2 sw3_row(const float2* sm, const SwCoef& cx, const float4* yac, const float2* yd,
                                          const float4* zac, const float2* zd, const float2 sg, float ph, int ry,
                                          int rz, int lane) {
  constexpr int Hp = O + 2 * (S - J) + 2;  // rows of stage J - 1
  const float2* src = sm + (size_t)(sw3_base<S, O, J - 1>() + (rz + 1) * Hp + ry + 1) * 32 + lane;
  const float2 v = src[0], vs = src[-32], vn = src[32], vb = src[-32 * Hp], vt = src[32 * Hp];
  const float4 ya = yac[ry + J], za = zac[rz + J];
  float2 dg = cadd(cx.d, yd[ry + J]);
  dg.x = (dg.x - ph) - sg.x;
  dg.y -= sg.y;
  float2 p = cmul(cx.a, shfl_up_c(v, 1));
  p = cfma(cx.c, shfl_down_c(v, 1), p);
  p = cfma(make_float2(ya.x, ya.y), vs, p);
  p = cfma(make_float2(ya.z, ya.w), vn, p);
  p = cfma(make_float2(za.x, za.y), vb, p);
  p = cfma(make_float2(za.z, za.w), vt, p);
  p = cfma(zd[rz + J], v, p);
  return cfma(dg, v, p);
}

template <int S, int O, int W>
__device__ __forceinline__ void sweep3_body(const LevelDev<float2>* __restrict__ levs, int nunits, int first,
                                            int store_last, int vblk, float2* sm) {
  constexpr int NS = gram_ns(S), NV = gram_nv(S), R = O + 2 * S;
  __shared__ float4 yac[R], zac[R];
  __shared__ float2 yd[R], zd[R];
  __shared__ float2 wsum[SW3_NW * NS];
  __shared__ float2 gs[(SW3_NW + 1) * NV];
  const int prob = vblk / nunits, unit = vblk - prob * nunits;
  const LevelDev<float2>& L = levs[prob];
  const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
  const int n = L.n, P = L.P;
  const float t = L.kt, phc = L.phir * t;
  const float* const phi = L.phi;
  const int ntx = ceil_div(n, sw_ox(S)), nty = ceil_div(n, O);
  const int x = (unit % ntx) * sw_ox(S) - S + lane;
  const int y0 = ((unit / ntx) % nty) * O - S, z0 = (unit / (ntx * nty)) * O - S;
  const SwCoef cx = sw_coef(L.ca, x, n, t);
  for (int i = tid; i < 2 * R; i += 256) {
    const int q = i < R ? i : i - R;
    const SwCoef c = sw_coef(L.ca, (i < R ? y0 : z0) + q, n, t);
    (i < R ? yac : zac)[q] = make_float4(c.a.x, c.a.y, c.c.x, c.c.y);
    (i < R ? yd : zd)[q] = c.d;
  }
  pdl_wait();
  float2 sg[S];
  const bool wide = wide_level(L, W);
  gram_shifts<S>(L, first != 0, wide, sg);
  const float2* R0 = first ? L.b : L.r0;
#pragma unroll 4
  for (int r = warp; r < R * R; r += SW3_NW)
    sm[r * 32 + lane] = ldc<float2>(R0, x, y0 + r % R, z0 + r / R, n, P);
  __syncthreads();
  auto phi_of = [&](int y, int z) -> float {
    return phi ? (inside(x, y, z, n) ? __ldg(phi + pidx(x, y, z, P)) * t : 0.f) : phc;
  };
  // stages 1 .. S - 1 into shared memory
  auto stage = [&](auto jc) {
    constexpr int J = decltype(jc)::value;
    constexpr int H = O + 2 * (S - J);
    for (int r = warp; r < H * H; r += SW3_NW) {
      const int ry = r % H, rz = r / H;
      sm[(sw3_base<S, O, J>() + r) * 32 + lane] = sw3_row<S, O, J>(
          sm, cx, yac, yd, zac, zd, sg[J - 1], phi_of(y0 + ry + J, z0 + rz + J), ry, rz, lane);
    }
    __syncthreads();
  };
  if constexpr (S >= 2) stage(std::integral_constant<int, 1>());
  if constexpr (S >= 3) stage(std::integral_constant<int, 2>());
  if constexpr (S >= 4) stage(std::integral_constant<int, 3>());
  const bool ownx = lane >= S && lane < 32 - S && x < n;
  auto own_points = [&](auto sum) {
    for (int r = warp; r < O * O; r += SW3_NW) {
      const int ry = r % O, rz = r / O, y = y0 + ry + S, z = z0 + rz + S;
      if (y >= n || z >= n) continue;  // uniform over the warp
      float2 kk[S + 1];
      kk[S] = sw3_row<S, O, S>(sm, cx, yac, yd, zac, zd, sg[S - 1], phi_of(y, z), ry, rz, lane);
      kk[0] = sm[((rz + S) * R + ry + S) * 32 + lane];
      if constexpr (S >= 2) kk[1] = sm[(sw3_base<S, O, 1>() + (rz + S - 1) * (R - 2) + ry + S - 1) * 32 + lane];
      if constexpr (S >= 3) kk[2] = sm[(sw3_base<S, O, 2>() + (rz + S - 2) * (R - 4) + ry + S - 2) * 32 + lane];
      if constexpr (S >= 4) kk[3] = sm[(sw3_base<S, O, 3>() + (rz + S - 3) * (R - 6) + ry + S - 3) * 32 + lane];
      if (ownx) {
        sum(kk);
#pragma unroll
        for (int j = 1; j <= S; ++j)
          if (j < S || store_last) L.p[j - 1][pidx(x, y, z, P)] = kk[j];
      }
    }
    pdl_trigger();  // the main work is done: let the next pass launch
  };
  float acc[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) acc[i] = 0.f;
  if (wide) {
    float c[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) c[i] = 0.f;
    own_points([&](const float2 (&kk)[S + 1]) { gram_point_wide<S>(kk, acc, c); });
    gram_block_sum_wide<S, SW3_NW>(acc, c, wsum, gs);
  } else {
    own_points([&](const float2 (&kk)[S + 1]) { gram_point<S>(kk, acc); });
    gram_block_sum<S, SW3_NW>(acc, wsum, gs);
  }
  gram_finish<S, SW3_NW>(L, sg, wide, unit, nunits, gs);
}
template <int S, int O, int W>
__global__ void __launch_bounds__(256, W == W_NO && S <= 3 ? 4 : 1)
k_sweep3(const LevelDev<float2>* __restrict__ levs, int nunits, int first, int store_last) {
  extern __shared__ __align__(16) float2 swsm[];
  sweep3_body<S, O, W>(levs, nunits, first, store_last, blockIdx.x, swsm);
}

// ------------------------------------------------------------------ 3D, large levels
// A CTA of 16 warps holds a 32 x 32 column of the level (two rows per warp) and marches in
// z.  In the step that loads plane z of R_0 it forms k_j of plane z - j for every j: the z
// neighbours are in registers (four planes of each vector), the x and y neighbours were
// published to shared memory in the previous step, so one barrier per step suffices.  Planes
// of R_0 (and phi) arrive in a ring of four by asynchronous copies issued two steps ahead
// (loaded to registers ahead, their waits fell together and the field's variant spilled).
// Bound by issue (61% active, 16 warps at 128 registers).  255^3, s = 3: 205 us a sweep, 238
// with a field; 248 and 311 with the loads in registers.
// Own points: (32 - 2S)^2 columns of `zc` planes.
constexpr int SM3_NW = 16, SM3_R = 32;
HELM_HD inline int sm3_units(int S, int n, int zc) {
  return ceil_div(n, sw_ox(S)) * ceil_div(n, sw_ox(S)) * ceil_div(n, zc);
}
// published planes: [parity][vector][row][lane], one guard row at either end
HELM_HD constexpr unsigned sm3_plane() { return (SM3_R + 2) * 32; }
// planes of R_0 and phi kept: four, or eight where the registers hold no window of k_0 (S = 4)
HELM_HD constexpr int sm3_ring(int S) { return S > 3 ? 8 : 4; }
HELM_HD constexpr unsigned sm3_smem(int S, int zc) {
  return (sm3_ring(S) + 2u * (S - 1)) * sm3_plane() * 8u + sm3_ring(S) * SM3_R * 32u * 4u + (unsigned)(zc + 2 * S) * 24u;
}
// Asynchronous copies to shared memory; with ok false they fill zeros and read nothing.
__device__ __forceinline__ void copy8_async(float2* dst, const float2* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(ok ? 8 : 0)
               : "memory");
}
__device__ __forceinline__ void copy4_async(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(ok ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copies_wait() {  // all but the N newest groups
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <int S, bool PHI>
__global__ void __launch_bounds__(SM3_NW * 32, 1)
k_sweep3_march(const LevelDev<float2>* __restrict__ levs, int nunits, int zc, int first, int store_last) {
  constexpr int NS = gram_ns(S), NV = gram_nv(S), W = 4;
  constexpr int RING = sm3_ring(S);
  constexpr bool K0 = RING == W;  // k_0 and phi of the last planes in registers too
  // s = 4: sums of four planes at a time to double-float (127^3 point source: error 3e-7, 1.5e-6
  // with one binary32 chain a thread, 7% of the time; s <= 3 has the smaller error either way)
  constexpr bool FOLD = S > 3;
  extern __shared__ __align__(16) float2 swsm[];
  __shared__ float2 wsum[SM3_NW * NS];
  __shared__ float2 gs[(SM3_NW + 1) * NV];
  const int prob = blockIdx.x / nunits, unit = blockIdx.x - prob * nunits;
  const LevelDev<float2>& L = levs[prob];
  const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
  const int n = L.n, P = L.P;
  const float t = L.kt, phir = L.phir, phc = phir * t;
  const float* const phi = L.phi;
  const int nt = ceil_div(n, sw_ox(S));
  const int x = (unit % nt) * sw_ox(S) - S + lane;
  const int ry = 2 * warp, y = ((unit / nt) % nt) * sw_ox(S) - S + ry;  // rows y, y + 1
  const int zb = (unit / (nt * nt)) * zc, ze = min(zb + zc, n);
  float2* const ring = swsm;                                             // R_0: plane i in slot i & (RING - 1)
  float2* const pub = ring + RING * sm3_plane();                         // [parity][k_1 .. k_{S-1}]
  float* const phring = reinterpret_cast<float*>(pub + 2 * (S - 1) * sm3_plane());
  float4* const zac = reinterpret_cast<float4*>(phring + RING * SM3_R * 32);
  float2* const zd = reinterpret_cast<float2*>(zac + (zc + 2 * S));
  const SwCoef cx = sw_coef(L.ca, x, n, t), cy0 = sw_coef(L.ca, y, n, t), cy1 = sw_coef(L.ca, y + 1, n, t);
  const float2 dxy[2] = {cadd(cx.d, cy0.d), cadd(cx.d, cy1.d)};
  for (int i = tid; i < ze - zb + 2 * S; i += SM3_NW * 32) {
    const SwCoef c = sw_coef(L.ca, zb - S + i, n, t);
    zac[i] = make_float4(c.a.x, c.a.y, c.c.x, c.c.y);
    zd[i] = c.d;
  }
  for (int i = tid; i < (RING + 2 * (S - 1)) * (int)sm3_plane(); i += SM3_NW * 32) ring[i] = make_float2(0.f, 0.f);
  pdl_wait();
  float2 sg[S];
  gram_shifts<S>(L, first != 0, false, sg);
  const float2* R0 = first ? L.b : L.r0;
  const bool in0 = (unsigned)x < (unsigned)n && (unsigned)y < (unsigned)n;
  const bool in1 = (unsigned)x < (unsigned)n && (unsigned)(y + 1) < (unsigned)n;
  const long long col = (long long)y * P + x;
  const size_t PP = (size_t)P * P;
  float2 win[S][W][2];  // k_j of the last planes, slot = plane & 3
#pragma unroll
  for (int j = K0 ? 0 : 1; j < S; ++j)
#pragma unroll
    for (int w = 0; w < W; ++w) win[j][w][0] = win[j][w][1] = make_float2(0.f, 0.f);
  float phw[W][2] = {};
  const bool field = PHI && phi;  // some problem of the launch has a field; this one may not
  const int at0 = (ry + 1) * 32 + lane;
  auto fetch = [&](int z, int slot) {
    const bool zin = (unsigned)z < (unsigned)n, ok0 = zin && in0, ok1 = zin && in1;
    const long long i = col + (long long)(z * PP);
    float2* const d = ring + slot * sm3_plane() + at0;
    copy8_async(d, ok0 ? R0 + i : R0, ok0);
    copy8_async(d + 32, ok1 ? R0 + i + P : R0, ok1);
    if (PHI && field) {
      float* const f = phring + slot * SM3_R * 32 + ry * 32 + lane;
      copy4_async(f, ok0 ? phi + i : phi, ok0);
      copy4_async(f + 32, ok1 ? phi + i + P : phi, ok1);
    }
  };
  float acc[NS], gsum = 0.f, gerr = 0.f;
#pragma unroll
  for (int i = 0; i < NS; ++i) acc[i] = 0.f;
  const bool ox = lane >= S && lane < 32 - S && x < n;
  const bool own0 = ox && ry >= S && ry < SM3_R - S && y < n;
  const bool own1 = ox && ry + 1 >= S && ry + 1 < SM3_R - S && y + 1 < n;
  const int zf = zb - S, zl = ze + S;  // planes loaded: zf .. zl - 1
  constexpr int AHEAD = 2;             // planes of copies in flight beyond the current one
  __syncthreads();                     // the ring is cleared before copies land in it
#pragma unroll
  for (int u = 0; u < AHEAD; ++u) {
    fetch(zf + u, u);
    copies_commit();
  }
  copies_wait<AHEAD - 1>();
  __syncthreads();
  // step i takes plane zf + i; slots are indexed by i & 3, which the unrolling by four
  // makes static.  Its copies overwrite plane i - 2, last read in the step before.
#pragma unroll 1
  for (int i0 = 0; i0 < zl - zf; i0 += W) {
#pragma unroll
    for (int u = 0; u < W; ++u) {
      const int i = i0 + u;
      if (i >= zl - zf) break;  // uniform
      const int z = zf + i;
      auto slot = [&](int d) { return K0 ? (u + d) & 3 : (i + d) & (RING - 1); };  // of plane i + d
      auto k0 = [&](int d, int q) { return ring[slot(d) * (int)sm3_plane() + at0 + 32 * q]; };
      auto ph = [&](int d, int q) {
        return field ? phring[slot(d) * SM3_R * 32 + (ry + q) * 32 + lane] * t : phc;
      };
      if (z + AHEAD < zl) fetch(z + AHEAD, slot(AHEAD));
      copies_commit();
      const float2* const r0 = ring + u * sm3_plane() + at0;
      if (K0) {
        win[0][u][0] = r0[0];
        win[0][u][1] = r0[32];
      }
      if (PHI && K0) {
        const float* const f = phring + u * SM3_R * 32 + ry * 32 + lane;
        phw[u][0] = field ? f[0] * t : phc;
        phw[u][1] = field ? f[32] * t : phc;
      }
      const float2* rd = pub + (size_t)((u & 1) ^ 1) * (S - 1) * sm3_plane() + at0;
      float2* wr = pub + (size_t)(u & 1) * (S - 1) * sm3_plane() + at0;
      float2 last[2];
#pragma unroll
      for (int j = 1; j <= S; ++j) {
        // k_j at plane z - j from k_{j-1} at planes z - j - 1 .. z - j + 1
        const int c = (u - j) & 3, b = (u - j - 1) & 3, f = (u - j + 1) & 3;
        float2 r[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        const int iz = i - j;  // index into the staged z coefficients
        if (iz >= 0) {         // uniform
          const float4 za = zac[iz];
          const float2 zdd = zd[iz];
          // k_{j-1} of plane z - j as published
          const float2* s = j == 1 ? ring + slot(-1) * sm3_plane() + at0 : rd + (size_t)(j > 1 ? j - 2 : 0) * sm3_plane();
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const bool reg = K0 || j > 1;
            float2 dg = dxy[q];
            dg.x = (dg.x - (PHI ? (K0 ? phw[c][q] : ph(-j, q)) : phc)) - sg[j - 1].x;
            dg.y -= sg[j - 1].y;
            const float2 v = reg ? win[j - 1][c][q] : k0(-1, q);
            const SwCoef& cy = q ? cy1 : cy0;
            // the diagonal's terms, the largest, are rounded once on their own and once in the sum
            // (first in one chain all later roundings are of their size: errors 5 to 10% larger;
            // last in it, the same errors, 255^3 1227 us a V-cycle instead of 1214)
            float2 d0 = cmul(dg, v);
            d0 = cfma(zdd, v, d0);
            float2 p = cmul(cx.a, s[32 * q - 1]);
            p = cfma(cx.c, s[32 * q + 1], p);
            p = cfma(cy.a, q ? (reg ? win[j - 1][c][0] : s[0]) : s[-32], p);
            p = cfma(cy.c, q ? s[64] : (reg ? win[j - 1][c][1] : s[32]), p);
            p = cfma(make_float2(za.x, za.y), reg ? win[j - 1][b][q] : k0(-2, q), p);
            p = cfma(make_float2(za.z, za.w), reg ? win[j - 1][f][q] : k0(0, q), p);
            r[q] = cadd(d0, p);
          }
        }
        if (j < S) {
          win[j][c][0] = r[0];
          win[j][c][1] = r[1];
          wr[(size_t)(j - 1) * sm3_plane()] = r[0];
          wr[(size_t)(j - 1) * sm3_plane() + 32] = r[1];
        } else {
          last[0] = r[0];
          last[1] = r[1];
        }
      }
      const int zo = z - S;
      if (i >= 2 * S) {  // uniform: zo is one of the CTA's planes
        const int c = (u - S) & 3;
        const size_t at = (size_t)(col + (long long)(zo * PP));
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          if (q ? own1 : own0) {
            float2 kk[S + 1];
            kk[0] = K0 ? win[0][c][q] : k0(-S, q);
#pragma unroll
            for (int j = 1; j < S; ++j) kk[j] = win[j][c][q];
            kk[S] = last[q];
            gram_point<S>(kk, acc);
#pragma unroll
            for (int j = 1; j <= S; ++j)
              if (j < S || store_last) L.p[j - 1][at + (q ? P : 0)] = kk[j];
          }
        }
      }
      copies_wait<AHEAD - 1>();
      __syncthreads();
    }
    if (FOLD) {
      const float tot = warp_transpose_sum_f<NS>(acc, lane);
      float sum, e;
      df_two_sum(gsum, tot, sum, e);
      gsum = sum;
      gerr += e;
#pragma unroll
      for (int k = 0; k < NS; ++k) acc[k] = 0.f;
    }
  }
  pdl_trigger();  // the main work is done: let the next pass launch
  if (FOLD) gram_block_total<S, SM3_NW>(make_float2(gsum, gerr), wsum, gs);
  else gram_block_sum<S, SM3_NW>(acc, wsum, gs);
  gram_finish<S, SM3_NW>(L, sg, false, unit, nunits, gs);
}

}  // namespace helm

// The complex64 2D V-cycle passes of the polynomial smoother (Sec. 4), one pass per sweep.
//
// A sweep is three Richardson steps x <- x + w_j (b - M x), without reductions, so a CTA can
// take all three on its own points and a rim of recomputed ones, together with what comes
// before (x = x_a + P e_c) and after (b_c = full weighting of b - M x): a level is one launch
// down and one up instead of nine (five steps and transfers down, four up), and its vectors
// are read once.  The CTA's 8 warps hold a 32 x 8 QY region in registers as the 2D sweep
// pass does (sweep.cuh); its own points start at the fifth and are 24 x (8 QY - 8): three
// steps, the residual and the full weighting reach four points (from zero the first step
// needs no neighbours; from a vector and with the coarse right-hand side they reach five to
// the far side: 22 x (8 QY - 10)).  Small levels are bound by the launch chain (about 3 us a
// pass), large ones by issue (1.8 regions' points formed per own point at 32 rows).  V-cycle
// 1023^2: 64 launches, 324-343 us, before; 13 launches, 89-101 us; 4095^2 2190 -> 920 us.
#pragma once
#include "sweep.cuh"

namespace helm {

constexpr int PO_H = 4;
HELM_HD constexpr int po_own(int R, int SRC, int END) { return R - 2 * PO_H - (SRC == 1 && END == 1 ? 2 : 0); }
HELM_HD inline int po_units(int QY, int SRC, int END, int n) {
  return ceil_div(n, po_own(32, SRC, END)) * ceil_div(n, po_own(SW2_NW * QY, SRC, END));
}

// SRC 0: from zero, 1: from `src`, 2: from x_a + P e_c; END 0: x only, 1: and the coarse
// right-hand side.
template <int QY, int SRC, int END>  // (three CTAs per SM: 1023^2 81 us a V-cycle, 88 at two)
__global__ void __launch_bounds__(256, 3)
k_poly2(const LevelDev<float2>* __restrict__ levs, const float2* __restrict__ pw, int nunits, int src, int dst) {
  constexpr int RY = SW2_NW * QY, OX = po_own(32, SRC, END), OY = po_own(RY, SRC, END);
  __shared__ float2 edge[2][SW2_NW + 2][2][32];
  __shared__ float4 yac[RY];
  __shared__ float2 yd[RY];
  __shared__ float2 rt[END ? RY : 1][33];
  const int prob = blockIdx.x / nunits, unit = blockIdx.x - prob * nunits;
  const LevelDev<float2>& L = levs[prob];
  const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
  const int n = L.n, P = L.P;
  const int ntx = ceil_div(n, OX);
  const int xo = (unit % ntx) * OX, yo = (unit / ntx) * OY;  // first own point
  const int x = xo - PO_H + lane, y0 = yo - PO_H + warp * QY;
  const SwCoef cx = sw_coef(L.ca, x, n, 1.0f);
  if (tid < RY) {
    const SwCoef c = sw_coef(L.ca, yo - PO_H + tid, n, 1.0f);
    yac[tid] = make_float4(c.a.x, c.a.y, c.c.x, c.c.y);
    yd[tid] = c.d;
  }
  if (warp < 2) {  // the rows beyond the region
    edge[warp][0][1][lane] = make_float2(0.f, 0.f);
    edge[warp][SW2_NW + 1][0][lane] = make_float2(0.f, 0.f);
  }
  const float ph = L.phir;  // constant k
  const float2 w[3] = {__ldg(pw + 3 * prob), __ldg(pw + 3 * prob + 1), __ldg(pw + 3 * prob + 2)};
  pdl_wait();
  float2 b[QY], v[QY];
#pragma unroll
  for (int q = 0; q < QY; ++q) {
    b[q] = ldc(L.b, x, y0 + q, 0, n, P);
    if (SRC == 0) v[q] = cmul(w[0], b[q]);
    if (SRC == 1) v[q] = ldc((const float2*)poly_vec(L, src), x, y0 + q, 0, n, P);
    if (SRC == 2)
      v[q] = cadd(ldc((const float2*)L.xa, x, y0 + q, 0, n, P), interp<float2>(L.xcb, n, L.nc, L.Pc, x, y0 + q, 0, 2));
  }
  int par = 0;
  // b - M v on the region (valid one point less far out each time)
  auto residual = [&](float2 (&r)[QY]) {
    edge[par][warp + 1][0][lane] = v[0];
    edge[par][warp + 1][1][lane] = v[QY - 1];
    __syncthreads();
    const float2 up = edge[par][warp][1][lane], dn = edge[par][warp + 2][0][lane];
    par ^= 1;
#pragma unroll
    for (int q = 0; q < QY; ++q) {
      const float4 ac = yac[warp * QY + q];
      float2 dg = cadd(cx.d, yd[warp * QY + q]);
      dg.x -= ph;
      float2 p = cmul(cx.a, shfl_up_c(v[q], 1));
      p = cfma(cx.c, shfl_down_c(v[q], 1), p);
      p = cfma(make_float2(ac.x, ac.y), q > 0 ? v[q > 0 ? q - 1 : 0] : up, p);
      p = cfma(make_float2(ac.z, ac.w), q < QY - 1 ? v[q < QY - 1 ? q + 1 : q] : dn, p);
      r[q] = csub(b[q], cfma(dg, v[q], p));
    }
  };
#pragma unroll
  for (int j = SRC == 0 ? 1 : 0; j < 3; ++j) {
    float2 r[QY];
    residual(r);
#pragma unroll
    for (int q = 0; q < QY; ++q) v[q] = cadd(v[q], cmul(w[j], r[q]));  // (a multiply-add rounds twice at v's size)
  }
  float2* const out = poly_vec(L, dst);
  const bool ownx = lane >= PO_H && lane < PO_H + OX && x < n;
#pragma unroll
  for (int q = 0; q < QY; ++q) {
    const int ry = warp * QY + q;
    if (ownx && ry >= PO_H && ry < PO_H + OY && y0 + q < n) out[pidx(x, y0 + q, 0, P)] = v[q];
  }
  if constexpr (END != 0) {
    float2 r[QY];
    residual(r);
#pragma unroll
    for (int q = 0; q < QY; ++q)
      rt[warp * QY + q][lane] = (y0 + q < n && x < n) ? r[q] : make_float2(0.f, 0.f);
    __syncthreads();
    const int nc = L.nc, Pc = L.Pc;
    if (tid < (OX / 2) * (OY / 2)) {  // one coarse point each
      const int px = tid % (OX / 2), py = tid / (OX / 2);
      const int fx = PO_H + 2 * px + 1, fy = PO_H + 2 * py + 1;
      float2 o = make_float2(0.f, 0.f);
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx)
          o = cadd(o, cscale(rt[fy + dy][fx + dx], (dx == 0 ? 0.5f : 0.25f) * (dy == 0 ? 0.5f : 0.25f)));
      const int Ix = xo / 2 + px, Iy = yo / 2 + py;
      if (Ix < nc && Iy < nc) L.bc[pidx(Ix, Iy, 0, Pc)] = o;
    }
  }
  pdl_trigger();
}

}  // namespace helm

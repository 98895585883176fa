// One GMRES(s) smoothing sweep from the Gram matrix of its Krylov basis (complex64).
//
// A sweep minimises ||R_0 - M K y|| over the Krylov space of R_0 (Sec. 3.1).  Instead of
// orthogonalising step by step (s passes, each ending in a grid-wide reduction that the
// next one waits for), the basis is generated by a fixed recurrence,
//
//     k_0 = R_0,   k_{j+1} = t (M - sigma_j) k_j,   t a power of two near 1 / rho(M),
//
// so k_1..k_s need no reduction in between and one pass over R_0 forms all of them.  The
// pass reduces the Gram matrix G = K^H K; the minimisation then follows from
// M K_s = K_{s+1} B (B lower bidiagonal: sigma_j on the diagonal, 1/t below) and
// G = L D L^H:  min_y ||D^{1/2} L^H (e_0 - B y)||, an (s+1) x s Hessenberg least-squares
// problem.  In exact arithmetic this is GMRES(s) (a Krylov space does not depend on its
// basis); x += K_s y and r = K_{s+1} (e_0 - B y) are combinations of the stored vectors.
//
// Accuracy.  Errors of G are amplified by the square of the basis's condition number, so
// the sums beyond a warp, the factorisation and the Schur complements are held as pairs of
// binary32 numbers (dfloat.cuh); the warp sums' binary32 roundings are independent and
// average out over the level.  The shifts keep the basis well conditioned: sigma_1 is the
// stencil's diagonal (the middle of the spectrum), sigma_0 = 0, so that k_1 carries M k_0
// to full relative accuracy when k_0 is smooth, where M k_0 is small and a shifted k_1
// would lose it.  The first sweep on the finest level meets arbitrary right-hand sides:
// there sigma_0 is the Rayleigh quotient estimated from the differences of neighbouring
// values (taken by the pass that writes the right-hand side).  Shifts carry 8 significant
// bits, so that subtracting one from a binary32 diagonal is exact.  Measured over whole
// V-cycles on the CPU in complex64, relative to 64 bits: 3.4e-7 / 2.2e-7 on white noise
// (step-by-step orthogonalisation in binary32: 3.3e-7 / 2.0e-7), 2.4-5e-7 on a point source
// (8.1e-7), 2.5e-7 on the Gaussian model's source (3.4e-7).
#pragma once
#include "device_common.cuh"
#include "dfloat.cuh"
#include "vcycle.cuh"

namespace helm {

// ------------------------------------------------------------------ layout of G
// The upper triangle row by row: diagonal entries one real, the others re, im.
HELM_HD constexpr int gram_nv(int S) { return (S + 1) * (S + 1); }
HELM_HD constexpr int gram_at(int S, int i, int j) {
  // rows 0..i-1 hold 1 + 2 (S - row) values each
  return i + 2 * (i * S - i * (i - 1) / 2) + (j == i ? 0 : 1 + 2 * (j - i - 1));
}
HELM_HD constexpr int gram_ns(int S) { return gram_nv(S) <= 16 ? 16 : 32; }  // butterfly width
// double-float slots per CTA: GRAM_SLOT (helm_internal.h), enough for S = SMAX
static_assert(gram_nv(SMAX) <= GRAM_SLOT, "partial slot too small");

// acc += the Gram products of one point's basis values k[0..S].
template <int S>
__device__ __forceinline__ void gram_point(const float2 (&k)[S + 1], float (&acc)[gram_ns(S)]) {
#pragma unroll
  for (int i = 0; i <= S; ++i) {
    float& d = acc[gram_at(S, i, i)];
    d = fmaf(k[i].x, k[i].x, fmaf(k[i].y, k[i].y, d));
#pragma unroll
    for (int j = i + 1; j <= S; ++j) {
      float& re = acc[gram_at(S, i, j)];
      float& im = acc[gram_at(S, i, j) + 1];
      re = fmaf(k[i].x, k[j].x, fmaf(k[i].y, k[j].y, re));
      im = fmaf(k[i].x, k[j].y, fmaf(-k[i].y, k[j].x, im));
    }
  }
}

// Sum NS (16 or 32) per-lane binary32 values over the warp by butterflies that halve the
// values kept; lane L ends with the total of value L (NS = 32) or L >> 1 (NS = 16).
template <int NS>
__device__ __forceinline__ float warp_transpose_sum_f(float (&v)[NS], int lane) {
  int o = 16;
#pragma unroll
  for (int c = NS / 2; c >= 1; c >>= 1, o >>= 1) {
    const bool hi = lane & o;
#pragma unroll
    for (int k = 0; k < c; ++k) {
      const float send = hi ? v[k] : v[k + c];
      const float keep = hi ? v[k + c] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return NS == 32 ? v[0] : v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// ------------------------------------------------------------------ double-float scalars
__device__ __forceinline__ float2 df_fast2(float s, float c) {
  const float t = __fadd_rn(s, c);
  return make_float2(t, __fsub_rn(c, __fsub_rn(t, s)));
}
__device__ __forceinline__ float2 df_mul2(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float e = fmaf(a.x, b.x, -p);
  e = fmaf(a.x, b.y, fmaf(a.y, b.x, e));
  return df_fast2(p, e);
}
// a - b c
__device__ __forceinline__ float2 df_fms2(float2 a, float2 b, float2 c) {
  const float p = __fmul_rn(b.x, c.x);
  float e = fmaf(b.x, c.x, -p);
  e = fmaf(b.x, c.y, fmaf(b.y, c.x, e));
  float t, r;
  df_two_sum(a.x, -p, t, r);
  return df_fast2(t, __fadd_rn(__fadd_rn(r, a.y), -e));
}
__device__ __forceinline__ float2 df_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 df_recip(float2 b) {
  const float r = __frcp_rn(b.x);
  const float e = fmaf(-b.y, r, fmaf(-b.x, r, 1.0f));
  return df_fast2(r, __fmul_rn(r, e));
}

// ------------------------------------------------------------------ the minimisation
// A pivot of the factorisation below this fraction of its diagonal entry means that k_j is
// a combination of the earlier vectors (to the rounding of binary32 vectors and of their
// Gram sums): the sweep stops at j Krylov steps.
constexpr float GRAM_TAU = 1e-7f;

// g: the NV double-float sums; sg[j] = t sigma_j.  Results: m Krylov steps, x += sum_{k<m}
// xc[k] k_k, r = sum_{k<=m} rc[k] k_k.  One thread's work (every lane of a warp may run it).
template <int S>
__device__ __forceinline__ int gram_solve(const float2* g, const float2 (&sg)[S], float t, float2 (&xc)[S],
                                          float2 (&rc)[S + 1]) {
#pragma unroll
  for (int k = 0; k < S; ++k) xc[k] = make_float2(0.f, 0.f);
#pragma unroll
  for (int k = 0; k <= S; ++k) rc[k] = make_float2(k == 0 ? 1.f : 0.f, 0.f);
  const float g00 = g[0].x;
  if (!(g00 > 0.0f) || !isfinite(g00)) return 0;
  // scale by a power of two so that G_00 is near one (exact; the products' low parts then
  // stay far from underflow)
  const unsigned e = (__float_as_uint(g00) >> 23) & 0xffu;
  const float sc = __uint_as_float(min(max(254u - e, 1u), 253u) << 23);
  float2 re[S + 1][S + 1], im[S + 1][S + 1];  // upper triangle, then D and U = L^H
  float dg[S + 1];
#pragma unroll
  for (int i = 0; i <= S; ++i)
#pragma unroll
    for (int j = i; j <= S; ++j) {
      const float2 a = g[gram_at(S, i, j)];
      re[i][j] = make_float2(a.x * sc, a.y * sc);
      if (j > i) {
        const float2 b = g[gram_at(S, i, j) + 1];
        im[i][j] = make_float2(b.x * sc, b.y * sc);
      } else {
        dg[i] = re[i][i].x;
      }
    }
  int m = S;
  bool alive = true;
  float w[S + 1];  // square roots of the pivots
  float2 u[S + 1][S + 1];
#pragma unroll
  for (int i = 0; i <= S; ++i) {
    const float d = re[i][i].x;
    if (alive && !(d > GRAM_TAU * dg[i])) {
      m = min(m, i);
      alive = false;
    }
    w[i] = alive ? sqrtf(d) : 0.0f;
    if (i == S) break;
    const float2 r = df_recip(alive ? re[i][i] : make_float2(1.f, 0.f));
    float2 ur[S + 1], ui[S + 1];
#pragma unroll
    for (int j = i + 1; j <= S; ++j) {
      ur[j] = df_mul2(re[i][j], r);
      ui[j] = df_mul2(im[i][j], r);
      u[i][j] = make_float2(ur[j].x, ui[j].x);
    }
    // S_jk -= conj(U_ij) S_ik
#pragma unroll
    for (int j = i + 1; j <= S; ++j)
#pragma unroll
      for (int k = j; k <= S; ++k) {
        re[j][k] = df_fms2(df_fms2(re[j][k], ur[j], re[i][k]), ui[j], im[i][k]);
        if (k > j) im[j][k] = df_fms2(df_fms2(im[j][k], ur[j], im[i][k]), df_neg(ui[j]), re[i][k]);
      }
  }
  // A = D^{1/2} U (t B): column j is sg_j U_{.j} + U_{.,j+1}
  float2 A[S + 1][S];
#pragma unroll
  for (int i = 0; i <= S; ++i)
#pragma unroll
    for (int j = 0; j < S; ++j) {
      float2 v = make_float2(0.f, 0.f);
      if (i < j) v = cmul(u[i][j], sg[j]);
      if (i == j) v = sg[j];
      if (i < j + 1) v = cadd(v, u[i][j + 1]);
      if (i == j + 1) v.x += 1.0f;
      A[i][j] = make_float2(v.x * w[i], v.y * w[i]);
    }
  // Givens rotations (the subdiagonal w[j + 1] is real); right-hand side w_0 e_0
  float2 q[S + 1];
  float rinv[S];
  q[0] = make_float2(w[0], 0.f);
#pragma unroll
  for (int j = 0; j < S; ++j) {
    const float2 a = A[j][j];
    const float b = A[j + 1][j].x;
    const float r2 = fmaf(a.x, a.x, fmaf(a.y, a.y, b * b));
    const float inv = r2 > 0.0f ? rsqrtf(r2) : 0.0f;
    const float2 ca = make_float2(a.x * inv, -a.y * inv);  // conj(a) / r
    const float sb = b * inv;
    rinv[j] = inv;
#pragma unroll
    for (int l = j + 1; l < S; ++l) {
      const float2 t0 = A[j][l], t1 = A[j + 1][l];
      A[j][l] = cadd(cmul(ca, t0), make_float2(sb * t1.x, sb * t1.y));
      A[j + 1][l] = csub(cmul(fconj(ca), t1), make_float2(sb * t0.x, sb * t0.y));
    }
    const float2 q0 = q[j];
    q[j] = cmul(ca, q0);
    q[j + 1] = make_float2(-sb * q0.x, -sb * q0.y);
  }
  float2 y[S];
#pragma unroll
  for (int j = S - 1; j >= 0; --j) {
    float2 v = q[j];
#pragma unroll
    for (int l = j + 1; l < S; ++l) v = csub(v, cmul(A[j][l], y[l]));
    y[j] = j < m ? make_float2(v.x * rinv[j], v.y * rinv[j]) : make_float2(0.f, 0.f);
  }
#pragma unroll
  for (int j = 0; j < S; ++j) {
    xc[j] = make_float2(t * y[j].x, t * y[j].y);
    const float2 sy = cmul(sg[j], y[j]);
    rc[j] = csub(rc[j], sy);
    rc[j + 1] = csub(rc[j + 1], y[j]);
  }
  return m;
}

// The (scaled) shifts of a sweep on level L: sigma_0 = 0, or the estimate left by the pass
// that wrote the right-hand side (finest level, first sweep), sigma_1 = sigma_3 = the
// stencil's diagonal, sigma_2 = 0.
template <int S>
__device__ __forceinline__ void gram_shifts(const LevelDev<float2>& L, bool first, float2 (&sg)[S]) {
  const float t = L.kt;
#pragma unroll
  for (int j = 0; j < S; ++j) {
    float2 s = make_float2(0.f, 0.f);
    if (j & 1) s = L.ksh;
    else if (j == 0 && first && L.top) s = L.sc->sig0;
    sg[j] = make_float2(s.x * t, s.y * t);
  }
}

// End of a sweep pass: every thread's Gram sums `acc` are reduced over its warp (binary32),
// the CTA and the level (double-float, fixed order); the last CTA of the problem solves the
// minimisation and writes the sweep's coefficients.  Every thread of the block calls it.
// `wsum` is NW * NS floats, `gs` gram_nv(S) * 8 float2 of shared memory.
template <int S, int NW>
__device__ __forceinline__ void gram_finish(float (&acc)[gram_ns(S)], const LevelDev<float2>& L, const float2 (&sg)[S],
                                            int unit, int nunits, float* wsum, float2* gs) {
  constexpr int NV = gram_nv(S), NS = gram_ns(S);
  constexpr int H = NS == 16 ? 2 : 1;  // slot groups a warp sums at a time
  __shared__ int s_last;
  const int tid = flat_tid(), lane = tid & 31, warp = tid >> 5;
  const float tot = warp_transpose_sum_f<NS>(acc, lane);
  if (NS == 32) wsum[warp * NS + lane] = tot;
  else if ((lane & 1) == 0) wsum[warp * NS + (lane >> 1)] = tot;
  __syncthreads();
  auto* sc = L.sc;
  float2* const part = reinterpret_cast<float2*>(L.part);
  const int v = NS == 16 ? (lane & 15) : lane, h = NS == 16 ? lane >> 4 : 0;
  if (warp == 0) {
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int q = h; q < NW; q += H) {
      float t, r;
      df_two_sum(s, wsum[q * NS + v], t, r);
      s = t;
      c += r;
    }
    if (H == 2) {
      const float s2 = __shfl_xor_sync(0xffffffffu, s, 16), c2 = __shfl_xor_sync(0xffffffffu, c, 16);
      float t, r;
      df_two_sum(s, s2, t, r);
      c = (c + c2) + r;
      s = t;
    }
    const float2 w = df_fast2(s, c);
    if (nunits > 1) {
      if (h == 0 && v < NV) __stcg(part + (size_t)unit * GRAM_SLOT + v, w);
      __syncwarp();
      if (lane == 0) {
        __threadfence();
        s_last = (atomicAdd(&sc->counter, 1u) == (unsigned)nunits - 1u);
      }
    } else {
      if (h == 0 && v < NV) gs[v] = w;
      if (lane == 0) s_last = 1;
    }
  }
  __syncthreads();
  if (!s_last) return;
  if (nunits > 1) {
    __threadfence();
    // warp w sums slots w H + h, + NW H, ... of value v, four loads in flight
    float s = 0.f, c = 0.f;
    for (int u0 = warp * H + h; u0 < nunits; u0 += 4 * NW * H) {
      float2 p[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int u = u0 + q * NW * H;
        p[q] = (u < nunits && v < NV) ? __ldcg(part + (size_t)u * GRAM_SLOT + v) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float t, r;
        df_two_sum(s, p[q].x, t, r);
        s = t;
        c += r + p[q].y;
      }
    }
    if (H == 2) {
      const float s2 = __shfl_xor_sync(0xffffffffu, s, 16), c2 = __shfl_xor_sync(0xffffffffu, c, 16);
      float t, r;
      df_two_sum(s, s2, t, r);
      c = (c + c2) + r;
      s = t;
    }
    if (h == 0 && v < NV) gs[warp * NV + v] = make_float2(s, c);
    __syncthreads();
    if (warp == 0) {
      float s1 = 0.f, c1 = 0.f;
      if (v < NV)
        for (int q = h; q < NW; q += H) {
          const float2 p = gs[q * NV + v];
          float t, r;
          df_two_sum(s1, p.x, t, r);
          s1 = t;
          c1 += r + p.y;
        }
      if (H == 2) {
        const float s2 = __shfl_xor_sync(0xffffffffu, s1, 16), c2 = __shfl_xor_sync(0xffffffffu, c1, 16);
        float t, r;
        df_two_sum(s1, s2, t, r);
        c1 = (c1 + c2) + r;
        s1 = t;
      }
      __syncwarp();
      if (h == 0 && v < NV) gs[v] = df_fast2(s1, c1);
      __syncwarp();
    }
  }
  if (warp == 0) {
    __syncwarp();
    float2 xc[S], rc[S + 1];
    const int m = gram_solve<S>(gs, sg, L.kt, xc, rc);
    if (lane == 0) {
      sc->m = m;
#pragma unroll
      for (int k = 0; k < S; ++k) sc->xcoef[k] = xc[k];
#pragma unroll
      for (int k = 0; k <= S; ++k) sc->rcoef[k] = rc[k];
      sc->counter = 0u;
    }
  }
}

}  // namespace helm

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
// M K_s = K_{s+1} B (B lower bidiagonal: sigma_j on the diagonal, 1/t below) and one
// linear system with G (gram_solve).  In exact arithmetic this is GMRES(s) (a Krylov space does not depend on its
// basis); x += K_s y and r = K_{s+1} (e_0 - B y) are combinations of the stored vectors.
//
// Accuracy.  Errors of G are amplified by the square of the basis's condition number, so
// the sums beyond a warp, the factorisation and the Schur complements are held as pairs of
// binary32 numbers (dfloat.cuh); the warp sums' binary32 roundings are independent and
// average out over the level.  The shifts keep the basis well conditioned: sigma_1 = sigma_3
// is the middle of the spectrum (the stencil's diagonal at the middle of the field's range),
// sigma_0 = sigma_2 = 0, so that k_1 carries M k_0 to full relative accuracy when k_0 is smooth,
// where M k_0 is small and a shifted k_1 would lose it.  The first sweep on the finest level
// meets arbitrary right-hand sides: there sigma_0 is the Rayleigh quotient estimated from the
// differences of neighbouring values (taken by the pass that writes the right-hand side), and
// a smooth right-hand side takes no shifts: its M k_0, M^2 k_0, ... are small and independent,
// where (M - sigma) k_1 is -sigma k_1 to a few digits (Gaussian source of 9 points' width,
// 127^2, s = 4: error 2.2e-2 with shifts, 2e-3 without and with step-by-step
// orthogonalisation).  Shifts carry 8 significant bits.
//
// Wide levels.  Where a wavenumber field's range exceeds the diagonal (GRAM_WIDE; the coarse
// levels of media with a contrast of three or more, where phi h^2 is large), the spectrum falls
// into clusters at the field's values and the k_j become dependent to 1e-4 and less: G and its
// solution then need all of double-float's digits.  There the warp sums are double-float too
// (ten instructions a product instead of one; 255^2 with discs 75 us a V-cycle, 69 without), a
// pivot counts down to GRAM_TAU_WIDE, and the shifts are 0 and the diagonal at the field's
// smallest value, middle and largest.  Whole V-cycles with layers and discs of contrast 3 to 27, against 64 bits, norm: at
// most 1.8 times and in the mean 0.4 times the error of step-by-step orthogonalisation in
// binary32; with binary32 sums and shifts that ignore the field up to 1e5 times (6e-2 instead of
// 6e-6 for discs of 12 at 255^2, s = 3).  On the CPU, lines from 0.25 to 2 diagonals gave the
// same errors; at one, media within +-30% keep the binary32 sums on all levels but the smallest.
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

// The same in double-float, sums s + c: the products are exact (TwoProduct) and so is every
// addition into s (TwoSum).
template <int S>
__device__ __forceinline__ void gram_point_wide(const float2 (&k)[S + 1], float (&s)[gram_ns(S)], float (&c)[gram_ns(S)]) {
  auto mac = [&](int i, float a, float b) { df_mac1(s[i], c[i], a, 0.f, b); };
#pragma unroll
  for (int i = 0; i <= S; ++i) {
    mac(gram_at(S, i, i), k[i].x, k[i].x);
    mac(gram_at(S, i, i), k[i].y, k[i].y);
#pragma unroll
    for (int j = i + 1; j <= S; ++j) {
      const int re = gram_at(S, i, j), im = re + 1;
      mac(re, k[i].x, k[j].x);
      mac(re, k[i].y, k[j].y);
      mac(im, k[i].x, k[j].y);
      mac(im, -k[i].y, k[j].x);
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

// warp_transpose_sum_f in double-float.
template <int NS>
__device__ __forceinline__ float2 warp_transpose_sum_df(float (&s)[NS], float (&c)[NS], int lane) {
  int o = 16;
  auto add = [](float& s, float& c, float s2, float c2) {
    float t, r;
    df_two_sum(s, s2, t, r);
    c = (c + c2) + r;
    s = t;
  };
#pragma unroll
  for (int n = NS / 2; n >= 1; n >>= 1, o >>= 1) {
    const bool hi = lane & o;
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const float s2 = __shfl_xor_sync(0xffffffffu, hi ? s[k] : s[k + n], o);
      const float c2 = __shfl_xor_sync(0xffffffffu, hi ? c[k] : c[k + n], o);
      if (hi) {
        s[k] = s[k + n];
        c[k] = c[k + n];
      }
      add(s[k], c[k], s2, c2);
    }
  }
  if (NS == 16) add(s[0], c[0], __shfl_xor_sync(0xffffffffu, s[0], 1), __shfl_xor_sync(0xffffffffu, c[0], 1));
  return make_float2(s[0], c[0]);
}

// ------------------------------------------------------------------ the minimisation
// min ||K_{s+1} rho|| over rho = e_0 - B y.  B's left null vector c (c_0 = 1, c_{j+1} =
// -t sigma_j c_j: the basis polynomials' values at zero) makes the constraint c^T rho = 1,
// so rho = w / (c^T w) with G w = conj(c), and y follows from B's subdiagonal,
// y_{j-1} = -rho_j - t sigma_j y_j.
//
// One warp, one entry of [G | conj(c)] per lane (row j, column k), Gauss-Jordan elimination
// without pivoting (G is positive definite) in double-float.  The step runs once per sweep,
// in one warp, usually on an SM that has not run it before, so instruction fetch counts as
// much as the arithmetic: this form is about 3 KB of code (1650-1900 cycles for s = 3 whatever
// the instruction caches hold).  Unrolled in one thread it is 12 KB: 1520 cycles with the code
// in the first-level cache, 2300-2600 from the next one, 4700-4900 from L2.
//
// A pivot below GRAM_TAU of its diagonal entry means that k_i is a combination of the
// earlier vectors (to the rounding of binary32 vectors and of their Gram sums): rho is then
// that combination, m = i Krylov steps.
constexpr float GRAM_TAU = 1e-7f;
constexpr float GRAM_TAU_WIDE = 1e-13f;  // double-float sums: a few 2^-45

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// s - a b - c d in double-float
__device__ __forceinline__ float2 df_fms2x2(float2 s, float2 a, float2 b, float2 c, float2 d) {
  const float p = __fmul_rn(a.x, b.x), q = __fmul_rn(c.x, d.x);
  const float e = fmaf(a.x, b.y, fmaf(a.y, b.x, fmaf(a.x, b.x, -p)));
  const float f = fmaf(c.x, d.y, fmaf(c.y, d.x, fmaf(c.x, d.x, -q)));
  float t, x, v, y;
  df_two_sum(s.x, -p, t, x);
  df_two_sum(t, -q, v, y);
  return df_fast2(v, ((s.y - e) - f) + (x + y));
}

// g: the NV double-float sums; sg: t sigma_j (sigma_2 = 0 and sigma_3 = sigma_1, or on wide
// levels sigma_0 = 0: in both cases c_j = 0 from j = 3 on).
// Lane k < S returns x's coefficient xk of k_k (x += sum_{k<m} x_k k_k), lane k <= S the
// residual's rk (r = sum_{k<=m} r_k k_k); every lane returns m.  The whole warp calls it.
template <int S>
__device__ __forceinline__ int gram_solve(const float2* g, const float2 (&sg)[S], bool wide, float t, int lane,
                                          float2& xk, float2& rk) {
  constexpr int NC = S + 2, N = S + 1;
  const float2 sg0 = sg[0], sg1 = sg[S > 1 ? 1 : 0];
  const unsigned full = 0xffffffffu;
  xk = make_float2(0.f, 0.f);
  rk = make_float2(lane == 0 ? 1.f : 0.f, 0.f);
  const float g00 = g[0].x;
  if (!(g00 > 0.0f) || !isfinite(g00)) return 0;
  // scale by a power of two so that G_00 is near one (exact; the products' low parts then
  // stay far from underflow)
  const unsigned ex = (__float_as_uint(g00) >> 23) & 0xffu;
  const float sc = __uint_as_float(min(max(254u - ex, 1u), 253u) << 23);
  const int j = min(lane / NC, S), k = lane - (lane / NC) * NC;
  // c_0 = 1, c_1 = -sg0, c_2 = sg0 sg1, then 0 (sigma_2 = 0)
  const float2 c2 = cmul(sg0, sg1);
  auto cq = [&](int q) {
    return q == 0 ? make_float2(1.f, 0.f) : q == 1 ? make_float2(-sg0.x, -sg0.y) : q == 2 ? c2 : make_float2(0.f, 0.f);
  };
  float2 re, im;
  {
    const int lo = min(j, k), hi = min(max(j, k), S);
    const int at = gram_at(S, lo, hi);
    const float2 a = g[at], b = g[lo < hi ? at + 1 : at];
    const float s = j < k ? sc : j > k ? -sc : 0.f;
    re = make_float2(a.x * sc, a.y * sc);
    im = make_float2(b.x * s, b.y * s);
    if (k > S) {
      const float2 c = cq(j);
      re = make_float2(c.x, 0.f);
      im = make_float2(-c.y, 0.f);
    }
  }
  const float tau = re.x * (wide ? GRAM_TAU_WIDE : GRAM_TAU);  // lanes (i, i): the threshold of pivot i
  int m = N, ii = 0, ji = j * NC, ik = k;
  float dinv = 0.f;                   // lane i: 1 / d_i
#pragma unroll 1
  for (int i = 0; i < N; ++i) {
    const unsigned ok = __ballot_sync(full, re.x > tau);
    const float dx = __shfl_sync(full, re.x, ii), dy = __shfl_sync(full, re.y, ii);
    const float2 ar = make_float2(__shfl_sync(full, re.x, ji), __shfl_sync(full, re.y, ji));
    const float2 ai = make_float2(__shfl_sync(full, im.x, ji), __shfl_sync(full, im.y, ji));
    const float2 br = make_float2(__shfl_sync(full, re.x, ik), __shfl_sync(full, re.y, ik));
    const float2 bi = make_float2(__shfl_sync(full, im.x, ik), __shfl_sync(full, im.y, ik));
    const float r = rcp_approx(dx), rl = r * fmaf(-dy, r, fmaf(-dx, r, 1.0f));
    if (m == N && !((ok >> ii) & 1u)) m = i;  // the remaining steps change nothing
    if (m == N && lane == i) dinv = r + rl;
    // u = S_ji / d, then row j minus u times row i
    const float urx = __fmul_rn(ar.x, r), uix = __fmul_rn(ai.x, r);
    const float2 ur = make_float2(urx, fmaf(ar.x, r, -urx) + fmaf(ar.x, rl, ar.y * r));
    const float2 ui = make_float2(uix, fmaf(ai.x, r, -uix) + fmaf(ai.x, rl, ai.y * r));
    const float2 nr = df_fms2x2(re, ur, br, make_float2(-ui.x, -ui.y), bi);
    const float2 ni = df_fms2x2(im, ur, bi, ui, br);
    if (m == N && j != i) {
      re = nr;
      im = ni;
    }
    ii += NC + 1;
    ji += 1;
    ik += NC;
  }
  // w_i in lane i; after a breakdown at m the null vector: w_m = 1, w_i = 0 beyond
  const int src = min(lane, S) * NC + (m < N ? m : S + 1);
  float2 w = make_float2(__shfl_sync(full, re.x, src) * dinv, __shfl_sync(full, im.x, src) * dinv);
  if (m < N) w = lane < m ? make_float2(-w.x, -w.y) : make_float2(lane == m ? 1.f : 0.f, 0.f);
  if (lane > S) w = make_float2(0.f, 0.f);
  m = min(m, S);
  // rho = w / (c^T w); c_i = 0 from i = 3 on
  float2 cw = cmul(cq(lane), w);
#pragma unroll
  for (int o = 1; o <= 2; o <<= 1)
    cw = make_float2(cw.x + __shfl_xor_sync(full, cw.x, o), cw.y + __shfl_xor_sync(full, cw.y, o));
  cw = make_float2(__shfl_sync(full, cw.x, 0), __shfl_sync(full, cw.y, 0));
  const float n2 = fabs2(cw), in = 1.0f / n2;
  if (!(n2 > 0.0f) || !isfinite(in)) return 0;  // M is singular on the space: no step
  rk = cmul(w, make_float2(cw.x * in, -cw.y * in));
  // y_j = -rho_{j+1} - sg_{j+1} y_{j+1}: sg_2 = 0, so odd j end there and even j take one more
  const float2 r1 = make_float2(__shfl_down_sync(full, rk.x, 1), __shfl_down_sync(full, rk.y, 1));
  const float2 r2 = make_float2(__shfl_down_sync(full, rk.x, 2), __shfl_down_sync(full, rk.y, 2));
  float2 y = csub(cmul((lane & 1) ? make_float2(0.f, 0.f) : sg1, r2), r1);
  if (wide) {  // all the way down: y_{S-1} = -rho_S, y_{j-1} = -rho_j - sg_j y_j
    float2 yj = make_float2(0.f, 0.f);
    y = yj;
#pragma unroll
    for (int j = S; j >= 1; --j) {
      const float2 rj = make_float2(__shfl_sync(full, rk.x, j), __shfl_sync(full, rk.y, j));
      yj = j < S ? csub(make_float2(-rj.x, -rj.y), cmul(sg[j < S ? j : 0], yj)) : make_float2(-rj.x, -rj.y);
      if (lane == j - 1) y = yj;
    }
  }
  xk = make_float2(t * y.x, t * y.y);
  return m;
}

// The (scaled) shifts of a sweep on level L: sigma_0 = 0, or the estimate left by the pass
// that wrote the right-hand side (finest level, first sweep; not on a wide level), then the
// level's own.  An estimate of 0 marks a smooth right-hand side: no shifts.
template <int S>
__device__ __forceinline__ void gram_shifts(const LevelDev<float2>& L, bool first, bool wide, float2 (&sg)[S]) {
  const float t = L.kt;
  const bool est = first && L.top && !wide;
  const float2 s0 = est ? L.sc->sig0 : make_float2(0.f, 0.f);
  const float tj = est && s0.x == 0.0f && s0.y == 0.0f ? 0.0f : t;
  sg[0] = make_float2(s0.x * t, s0.y * t);
#pragma unroll
  for (int j = 1; j < S; ++j) {  // (ordinary levels: sigma_2 = 0, sigma_3 = sigma_1)
    const float2 k = wide ? L.ksh[j - 1] : j == 2 ? make_float2(0.f, 0.f) : L.ksh[0];
    sg[j] = make_float2(k.x * tj, k.y * tj);
  }
}

// Sum of NW double-floats per value, gs-style: thread v NW + w holds part w of value v (NW a
// power of two up to 16); the thread with w = 0 ends with the total.  Whole warps call it.
template <int NW>
__device__ __forceinline__ float2 df_group_sum(float2 a) {
#pragma unroll
  for (int o = NW / 2; o > 0; o >>= 1) {
    const float2 b = make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
    float t, r;
    df_two_sum(a.x, b.x, t, r);
    a = make_float2(t, (a.y + b.y) + r);
  }
  return df_fast2(a.x, a.y);
}

// The warps' sums of a CTA of NW warps, combined: gs[0..NV-1].  Every thread calls it (it
// starts with a barrier; another must precede the reads of gs).
template <int S, int NW>
__device__ __forceinline__ void gram_block_sum(float (&acc)[gram_ns(S)], float2* wsum2, float2* gs) {
  constexpr int NV = gram_nv(S), NS = gram_ns(S);
  const int tid = flat_tid(), lane = tid & 31, warp = tid >> 5;
  float* const wsum = reinterpret_cast<float*>(wsum2);
  const float tot = warp_transpose_sum_f<NS>(acc, lane);
  if (NS == 32) wsum[warp * NS + lane] = tot;
  else if ((lane & 1) == 0) wsum[warp * NS + (lane >> 1)] = tot;
  __syncthreads();
  const int v = tid / NW, w = tid % NW;
  if (warp * 32 < NV * NW) {  // uniform over the warp
    const float2 a = df_group_sum<NW>(make_float2(v < NV ? wsum[w * NS + v] : 0.f, 0.f));
    if (w == 0 && v < NV) gs[v] = a;
  }
}

// The same from the warps' double-float totals (as warp_transpose_sum_f leaves them).
template <int S, int NW>
__device__ __forceinline__ void gram_block_total(float2 tot, float2* wsum, float2* gs) {
  constexpr int NV = gram_nv(S), NS = gram_ns(S);
  const int tid = flat_tid(), lane = tid & 31, warp = tid >> 5;
  if (NS == 32) wsum[warp * NS + lane] = tot;
  else if ((lane & 1) == 0) wsum[warp * NS + (lane >> 1)] = tot;
  __syncthreads();
  const int v = tid / NW, w = tid % NW;
  if (warp * 32 < NV * NW) {  // uniform over the warp
    const float2 a = df_group_sum<NW>(v < NV ? wsum[w * NS + v] : make_float2(0.f, 0.f));
    if (w == 0 && v < NV) gs[v] = a;
  }
}
// The same from every thread's double-float sums.
template <int S, int NW>
__device__ __forceinline__ void gram_block_sum_wide(float (&s)[gram_ns(S)], float (&c)[gram_ns(S)], float2* wsum,
                                                    float2* gs) {
  gram_block_total<S, NW>(warp_transpose_sum_df<gram_ns(S)>(s, c, flat_tid() & 31), wsum, gs);
}

// End of a sweep pass, after the CTA's sums (gram_block_sum): they are added over the level
// (double-float, fixed order); the last CTA of the problem solves the minimisation and writes
// the sweep's coefficients.  Every thread of the block calls it.  (The block sum's `wsum` is
// NW * NS float2, `gs` gram_nv(S) * (NW + 1) float2 of shared memory.)
template <int S, int NW>
__device__ __forceinline__ void gram_finish(const LevelDev<float2>& L, const float2 (&sg)[S], bool wide, int unit,
                                            int nunits, float2* gs) {
  constexpr int NV = gram_nv(S), NS = gram_ns(S);
  constexpr int H = NS == 16 ? 2 : 1;  // slots a warp reads at a time
  __shared__ int s_last;
  const int tid = flat_tid(), lane = tid & 31, warp = tid >> 5;
  __syncthreads();
  auto* sc = L.sc;
  if (nunits > 1) {
    float2* const part = reinterpret_cast<float2*>(L.part);
    if (warp == 0) {
      if (lane < NV) __stcg(part + (size_t)unit * GRAM_SLOT + lane, gs[lane]);
      __syncwarp();
      if (lane == 0) {
        __threadfence();
        s_last = (atomicAdd(&sc->counter, 1u) == (unsigned)nunits - 1u);
      }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // warp w sums slots w H + h, + NW H, ... of value v, four loads in flight
    const int v = NS == 16 ? (lane & 15) : lane, h = NS == 16 ? lane >> 4 : 0;
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
    float2* const gw = gs + NV;  // [warp][value]
    if (h == 0 && v < NV) gw[warp * NV + v] = make_float2(s, c);
    __syncthreads();
    const int vv = tid / NW, w = tid % NW;
    if (warp * 32 < NV * NW) {
      const float2 a = df_group_sum<NW>(vv < NV ? gw[w * NV + vv] : make_float2(0.f, 0.f));
      if (w == 0 && vv < NV) gs[vv] = a;
    }
    __syncthreads();
  }
  if (warp == 0) {
    float2 xk, rk;
    const int m = gram_solve<S>(gs, sg, wide, L.kt, lane, xk, rk);
    if (lane < S) sc->xcoef[lane] = xk;
    if (lane <= S) sc->rcoef[lane] = rk;
    if (lane == 0) {
      sc->m = m;
      sc->counter = 0u;
    }
  }
}

}  // namespace helm

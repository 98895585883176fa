// The coarse sub-cycle of the complex64 V-cycle: every level of at most 31^2 or 7^3 points,
// down to the coarsest and up again, by one CTA per problem.
//
// Bound by latency: a level is one or two points per thread, and a sweep is a chain of
// stencils, one Gram reduction and one small minimisation (gram.cuh), each behind a
// barrier.  So every thread keeps the stencil coefficients of its points and its values of
// k_0..k_S in registers for the whole sweep; shared memory only carries what neighbours
// read, in the padded layout (row pitch P = n + 1, ghosts zero), whose ghosts and the ghost
// rows of the vector before make the stencil free of bounds checks.  The coarsest system is
// solved with its inverse, formed in binary64 at set-up and held as double-floats: a matrix
// times vector, all rows at once, instead of 2 m dependent elimination steps on the FP64
// pipe.  From 31^2: about 20 us (18 Arnoldi passes with a barrier-separated reduction and
// algebra each, and the elimination, took 90 us), 2.9 us a sweep; 512 threads of two points
// each, 256 of four are 1-2% slower.  Everything that does not depend on the previous kernel is loaded before the wait.
#pragma once
#include "gram.cuh"

namespace helm {

constexpr int CG_THREADS = 512, CG_NW = CG_THREADS / 32, CG_PT = 2;
constexpr int CG_COARSE_POINTS = CG_THREADS * CG_PT;  // most interior points of a level
constexpr int CG_INV = 1024;                          // entries of the inverse staged in shared memory
constexpr int CG_COEF = 3 * 64;                       // 1D coefficients of all levels (31 + 15 + 7 + 3 per array)
static_assert(coarse_threshold(2, 1) * coarse_threshold(2, 1) <= CG_COARSE_POINTS &&
                  coarse_threshold(3, 1) * coarse_threshold(3, 1) * coarse_threshold(3, 1) <= CG_COARSE_POINTS &&
                  2 * coarse_threshold(2, 1) <= CG_COEF / 3,
              "a thread holds CG_PT points of a level; the levels halve");

// b, x, r, k_1..k_{S-1} and, where a level is wide, k_S; S = 0 stands for the polynomial smoother
HELM_HD constexpr int cg_vectors(int S, bool wide = false) { return 3 + (S > 1 ? S - 1 : 0) + (wide ? 1 : 0); }

// One thread's points of a level and the level's vectors.
template <int S, int DIM>
struct CgLevel {
  int n, P;
  float t, it;                         // basis scale and its reciprocal
  float2 *b, *x, *r, *k[S > 1 ? S - 1 : 1];
  float2* kv;                          // k_1 .. (at strides of np)
  int np;                              // padded points
  int off[CG_PT], cx[CG_PT], cy[CG_PT], cz[CG_PT];
  bool on[CG_PT];
  float2 ax[CG_PT], qx[CG_PT], ay[CG_PT], qy[CG_PT], az[CG_PT], qz[CG_PT], dg[CG_PT], dz[CG_PT];

  // coef: the level's 1D coefficients a, d, c times t
  __device__ __forceinline__ void stencil_setup(const LevelDev<float2>& L, const float2* coef, int tid) {
    n = L.n;
    P = L.P;
    t = L.kt;
    it = __frcp_rn(t);
    const float rn = __frcp_rn((float)n);  // i / n for i < 1024: exact with half a unit added
    const int np = DIM == 3 ? n * n * n : n * n;
    const float phc = L.phir * t;
#pragma unroll
    for (int q = 0; q < CG_PT; ++q) {
      const int i = tid + q * CG_THREADS;
      on[q] = i < np;
      const int ii = on[q] ? i : 0;
      const int yy = (int)(((float)ii + 0.5f) * rn);
      cx[q] = ii - yy * n;
      cz[q] = DIM == 3 ? (int)(((float)yy + 0.5f) * rn) : 0;
      cy[q] = yy - cz[q] * n;
      off[q] = (cz[q] * P + cy[q]) * P + cx[q];
      ax[q] = coef[cx[q]];
      qx[q] = coef[2 * n + cx[q]];
      ay[q] = coef[cy[q]];
      qy[q] = coef[2 * n + cy[q]];
      dg[q] = cadd(coef[n + cx[q]], coef[n + cy[q]]);
      if (DIM == 3) {
        az[q] = coef[cz[q]];
        qz[q] = coef[2 * n + cz[q]];
        dz[q] = coef[n + cz[q]];
      }
      dg[q].x -= L.phi ? __ldg(L.phi + off[q]) * t : phc;
    }
  }
  // t (M - sigma) v at point q; v0 the point's own value
  __device__ __forceinline__ float2 apply(const float2* v, float2 v0, int q, float2 sg) const {
    float2 d = dg[q];
    d.x -= sg.x;
    d.y -= sg.y;
    const float2* s = v + off[q];
    float2 p = cmul(ax[q], s[-1]);
    p = cfma(qx[q], s[1], p);
    p = cfma(ay[q], s[-P], p);
    p = cfma(qy[q], s[P], p);
    if (DIM == 3) {
      p = cfma(az[q], s[-P * P], p);
      p = cfma(qz[q], s[P * P], p);
      p = cfma(dz[q], v0, p);  // apart: the sum of the three diagonals would be rounded
    }
    return cfma(d, v0, p);
  }
};

struct CgShared {
  float2 wsum[CG_NW * 16];
  float2 gs[gram_nv(SMAX)];
  float2 xc[SMAX], rc[SMAX + 1];
};

// The Gram matrix of a wide level in double-float: a warp per value, all of the level's points
// from shared memory (k_0 at R0, k_j at kv + (j - 1) np; ghosts are zero).  A loop of a few
// instructions: as thread sums of both points and a transposed butterfly it was 14 KB of
// straight-line code, fetched from L2 for every launch (a 3D sub-cycle took 31 us, 16 without).
template <int S>
__device__ __forceinline__ void cg_gram_wide(const float2* R0, const float2* kv, int np, float2* gs) {
  const int lane = threadIdx.x & 31;
  for (int v = threadIdx.x >> 5; v < gram_nv(S); v += CG_NW) {
    int i = 0, e = v;  // row i, entry e of it: the diagonal, then re and im of each column
    while (e > 2 * (S - i)) {
      e -= 1 + 2 * (S - i);
      ++i;
    }
    const int j = i + (e + 1) / 2;
    const bool im = e > 0 && !(e & 1);
    const float2 *A = i == 0 ? R0 : kv + (size_t)(i - 1) * np, *B = j == 0 ? R0 : kv + (size_t)(j - 1) * np;
    float s = 0.f, c = 0.f;
    for (int p = lane; p < np; p += 32) {
      const float2 a = A[p], b = B[p];
      df_mac1(s, c, a.x, 0.f, im ? b.y : b.x);
      df_mac1(s, c, a.y, 0.f, im ? -b.x : b.y);
    }
    const float2 tot = df_group_sum<32>(make_float2(s, c));
    if (lane == 0) gs[v] = tot;
  }
}

// One sweep: k0 (this thread's values of R_0, already in shared memory at R0 and visible to
// the CTA) -> x += dx and k0 = the new residual.
template <int S, int DIM>
__device__ __forceinline__ void cg_sweep(const CgLevel<S, DIM>& V, const float2* R0, float2 (&k0)[CG_PT],
                                         float2 (&x)[CG_PT], const float2 (&sg)[S], bool wide, CgShared& sh) {
  constexpr int NS = gram_ns(S);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float2 k[CG_PT][S + 1];
#pragma unroll
  for (int q = 0; q < CG_PT; ++q) k[q][0] = k0[q];
#pragma unroll
  for (int j = 1; j <= S; ++j) {
    const float2* src = j == 1 ? R0 : V.k[j >= 2 ? j - 2 : 0];
#pragma unroll
    for (int q = 0; q < CG_PT; ++q) {
      k[q][j] = make_float2(0.f, 0.f);
      if (V.on[q]) {
        k[q][j] = V.apply(src, k[q][j - 1], q, sg[j - 1]);
        if (j < S) V.k[j >= 1 && j < S ? j - 1 : 0][V.off[q]] = k[q][j];
        else if (wide) V.kv[(S - 1) * V.np + V.off[q]] = k[q][j];
      }
    }
    if (j < S) __syncthreads();
  }
  if (wide) {
    __syncthreads();
    cg_gram_wide<S>(R0, V.kv, V.np, sh.gs);
  } else {
    float acc[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) acc[i] = 0.f;
#pragma unroll
    for (int q = 0; q < CG_PT; ++q) gram_point<S>(k[q], acc);
    gram_block_sum<S, CG_NW>(acc, sh.wsum, sh.gs);
  }
  __syncthreads();
  if (warp == 0) {
    float2 xk, rk;
    gram_solve<S>(sh.gs, sg, wide, V.t, lane, xk, rk);
    if (lane < S) sh.xc[lane] = xk;
    if (lane <= S) sh.rc[lane] = rk;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < CG_PT; ++q) {
    float2 dx = make_float2(0.f, 0.f), r = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < S; ++i) dx = cfma(sh.xc[i], k[q][i], dx);
#pragma unroll
    for (int i = 0; i <= S; ++i) r = cfma(sh.rc[i], k[q][i], r);
    x[q] = cadd(x[q], dx);
    k0[q] = r;
  }
}

// One sweep of the polynomial smoother (Sec. 4): x <- x + w_j (b - M x), j = 0, 1, 2, from
// zero where `zero`.  x is published to V.x and V.r in turn (`tog`), one barrier a step.
template <int S, int DIM>
__device__ __forceinline__ void cg_poly(const CgLevel<S, DIM>& V, const float2 (&b)[CG_PT], float2 (&x)[CG_PT],
                                        const float2* w, bool zero, int& tog) {
  const float2 z0 = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int j = 0; j < 3; ++j) {
    const float2 wj = w[j];
    float2* buf = tog ? V.r : V.x;
    if (!(zero && j == 0)) {
#pragma unroll
      for (int q = 0; q < CG_PT; ++q)
        if (V.on[q]) buf[V.off[q]] = x[q];
      __syncthreads();
      tog ^= 1;
    }
#pragma unroll
    for (int q = 0; q < CG_PT; ++q) {
      float2 r = b[q];
      if (!(zero && j == 0) && V.on[q]) {
        const float2 p = V.apply(buf, x[q], q, z0);
        r = csub(r, make_float2(p.x * V.it, p.y * V.it));
      }
      x[q] = cadd(x[q], cmul(wj, r));
    }
  }
}

template <int S, int DIM, int WIDE>  // 1: some level of the problem's is wide
__global__ void __launch_bounds__(CG_THREADS, 1)
k_coarse_gram(const LevelDev<float2>* __restrict__ levs_all, int lev_stride, const CoarseLU* __restrict__ lus,
              const float2* __restrict__ pw, int nu1, int nu2, int from_res) {
  extern __shared__ __align__(16) float2 cgsm[];
  __shared__ LevelDev<float2> Ls[MAX_COARSE_LEVELS_HOST];
  __shared__ int s_base[MAX_COARSE_LEVELS_HOST], s_cof[MAX_COARSE_LEVELS_HOST];
  __shared__ float2 coef[CG_COEF];
  __shared__ float4 inv_sm[CG_INV];
  __shared__ CgShared sh;
  constexpr int NVEC = cg_vectors(S, WIDE);
  const int tid = threadIdx.x, prob = blockIdx.x;
  const LevelDev<float2>* G = levs_all + (size_t)prob * lev_stride;
  const CoarseLU lu = lus[prob];
  const int nlev = lu.nlev;
  {  // descriptors (a word per thread)
    constexpr int W = (int)(sizeof(LevelDev<float2>) / sizeof(int));
    for (int i = tid; i < nlev * W; i += CG_THREADS)
      reinterpret_cast<int*>(Ls)[i] = reinterpret_cast<const int*>(G)[i];
  }
  __syncthreads();
  int total = 0, ctot = 0;
  for (int l = 0; l < nlev; ++l) {
    const int P = Ls[l].P, np = DIM == 3 ? P * P * P : P * P;
    if (tid == 0) {
      s_base[l] = total + np / P;  // a guard row (plane) of zeros before the level's first vector
      s_cof[l] = ctot;
    }
    total += np / P + NVEC * np;
    ctot += 3 * Ls[l].n;
  }
  for (int i = tid; i < total; i += CG_THREADS) cgsm[i] = make_float2(0.f, 0.f);
  __syncthreads();
  for (int l = 0; l < nlev; ++l)
    for (int i = tid; i < 3 * Ls[l].n; i += CG_THREADS) {
      const float2 v = __ldg(Ls[l].ca + i);
      coef[s_cof[l] + i] = make_float2(v.x * Ls[l].kt, v.y * Ls[l].kt);
    }
  const bool staged = lu.m * lu.m <= CG_INV;
  if (staged)
    for (int i = tid; i < lu.m * lu.m; i += CG_THREADS) inv_sm[i] = __ldg(lu.inv + i);
  __syncthreads();
  CgLevel<S, DIM> V;
  auto enter = [&](int l) {
    const int P = Ls[l].P, np = DIM == 3 ? P * P * P : P * P;
    float2* v = cgsm + s_base[l];
    V.b = v;
    V.x = v + np;
    V.r = v + 2 * np;
    V.kv = v + 3 * np;
    V.np = np;
#pragma unroll
    for (int j = 0; j + 1 < S; ++j) V.k[j] = V.kv + j * np;
    V.stencil_setup(Ls[l], coef + s_cof[l], tid);
  };
  enter(0);
  pdl_wait();
  pdl_trigger();
  if (S > 0 && DIM == 2 && from_res && !Ls[0].top) {
    // b = full weighting of the finer level's residual (k_sweep2_down does the same)
    const LevelDev<float2>& L = Ls[0];
    const int m = L.scf->m, Pf = 2 * L.P;
    float2 rc[S + 1];
#pragma unroll
    for (int j = 0; j <= S; ++j) rc[j] = L.scf->rcoef[j];
    // a warp per coarse row (n <= 31), fine points in pairs, each row read once per coarse row:
    // nine single loads a point and vector took 2 us more at n = 31
    const int lane = tid & 31, n = L.n;
    for (int y = tid >> 5; y < n; y += CG_NW) {
      float4 v[3][S + 1];
      const bool ok = lane <= n;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j <= S; ++j) {
          const float2* R = j == 0 ? L.fb : L.fp[j > 0 ? j - 1 : 0];
          v[i][j] = ok ? *reinterpret_cast<const float4*>(R + (size_t)(2 * y + i) * Pf + 2 * lane)
                       : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      float2 out = make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        float2 r0 = make_float2(0.f, 0.f), r1 = r0;
#pragma unroll
        for (int j = 0; j <= S; ++j)
          if (j <= m) {  // uniform
            r0 = cfma(rc[j], make_float2(v[i][j].x, v[i][j].y), r0);
            r1 = cfma(rc[j], make_float2(v[i][j].z, v[i][j].w), r1);
          }
        const float2 r2 = shfl_down_c(r0, 1);
        const float w = i == 1 ? 0.125f : 0.0625f;
        out = cadd(out, cscale(r0, w));
        out = cadd(out, cscale(r1, 2.0f * w));
        out = cadd(out, cscale(r2, w));
      }
      if (lane < n) V.b[y * L.P + lane] = out;
    }
  } else {
#pragma unroll
    for (int q = 0; q < CG_PT; ++q)
      if (V.on[q]) V.b[V.off[q]] = G[0].b[V.off[q]];
  }
  __syncthreads();
  // descent
  for (int l = 0; l < nlev - 1; ++l) {
    if (l > 0) enter(l);
    float2 k0[CG_PT], x[CG_PT];
#pragma unroll
    for (int q = 0; q < CG_PT; ++q) {
      k0[q] = V.on[q] ? V.b[V.off[q]] : make_float2(0.f, 0.f);
      x[q] = make_float2(0.f, 0.f);
    }
    if constexpr (S == 0) {
      if (nu1 > 0) {
        int tog = 0;
        for (int sw = 0; sw < nu1; ++sw)
          cg_poly<S, DIM>(V, k0, x, pw + 3 * ((size_t)prob * lev_stride + l), sw == 0, tog);
        __syncthreads();  // the last step's readers of V.x are done
#pragma unroll
        for (int q = 0; q < CG_PT; ++q)
          if (V.on[q]) V.x[V.off[q]] = x[q];
        __syncthreads();
        const float2 z0 = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < CG_PT; ++q)
          if (V.on[q]) {
            const float2 p = V.apply(V.x, x[q], q, z0);
            V.r[V.off[q]] = csub(k0[q], make_float2(p.x * V.it, p.y * V.it));
          }
        __syncthreads();
      }
    } else {
    const float2* R0 = V.b;
    for (int sw = 0; sw < nu1; ++sw) {
      float2 sg[S];
      const bool wide = WIDE && Ls[l].wide;
      gram_shifts<S>(Ls[l], sw == 0, wide, sg);
      cg_sweep<S, DIM>(V, R0, k0, x, sg, wide, sh);
      R0 = V.r;
#pragma unroll
      for (int q = 0; q < CG_PT; ++q)
        if (V.on[q]) V.r[V.off[q]] = k0[q];
      __syncthreads();
    }
    }
    const float2* rr = nu1 > 0 ? V.r : V.b;
#pragma unroll
    for (int q = 0; q < CG_PT; ++q)
      if (V.on[q]) V.x[V.off[q]] = x[q];
    // b_c = full weighting of the residual
    const int nc = Ls[l + 1].n, Pc = Ls[l + 1].P, P = V.P;
    const int ncp = DIM == 3 ? nc * nc * nc : nc * nc;
    float2* bc = cgsm + s_base[l + 1];
    const float rnc = __frcp_rn((float)nc);
    for (int i = tid; i < ncp; i += CG_THREADS) {
      const int yy = (int)(((float)i + 0.5f) * rnc), X = i - yy * nc;
      const int Z = DIM == 3 ? (int)(((float)yy + 0.5f) * rnc) : 0, Y = yy - Z * nc;
      const float2* f = rr + (DIM == 3 ? (2 * Z + 1) * P * P : 0) + (2 * Y + 1) * P + 2 * X + 1;
      float2 out = make_float2(0.f, 0.f);
#pragma unroll
      for (int dz = (DIM == 3 ? -1 : 0); dz <= (DIM == 3 ? 1 : 0); ++dz)
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
          for (int dx = -1; dx <= 1; ++dx) {
            const float wgt = (dx == 0 ? 0.5f : 0.25f) * (dy == 0 ? 0.5f : 0.25f) * (DIM == 3 ? (dz == 0 ? 0.5f : 0.25f) : 1.0f);
            const float2 v = f[(dz * P + dy) * P + dx];
            out.x = fmaf(wgt, v.x, out.x);
            out.y = fmaf(wgt, v.y, out.y);
          }
      bc[((DIM == 3 ? Z * Pc : 0) + Y) * Pc + X] = out;
    }
    __syncthreads();
  }
  // coarsest: x = A^{-1} b, sixteen lanes per row, double-float sums
  {
    const LevelDev<float2>& L = Ls[nlev - 1];
    const int m = lu.m, n = L.n, P = L.P, np = DIM == 3 ? P * P * P : P * P;
    const float2* b = cgsm + s_base[nlev - 1];
    float2* x = cgsm + s_base[nlev - 1] + np;
    const float4* inv = staged ? inv_sm : lu.inv;
    const int l16 = tid & 15;
    auto at = [&](int i) {
      const int yy = i / n, X = i - yy * n, Z = DIM == 3 ? yy / n : 0, Y = yy - Z * n;
      return (Z * P + Y) * P + X;
    };
    for (int r0 = 0; r0 < m; r0 += CG_THREADS / 16) {  // the same trips for every thread
      const int row = r0 + (tid >> 4);
      float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f;
      if (row < m)
        for (int j = l16; j < m; j += 16) {
          const float4 a = inv[(size_t)row * m + j];
          const float2 v = b[at(j)];
          df_mac1(sr, cr, a.x, a.y, v.x);
          df_mac1(sr, cr, -a.z, -a.w, v.y);
          df_mac1(si, ci, a.x, a.y, v.y);
          df_mac1(si, ci, a.z, a.w, v.x);
        }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        float t, r;
        const float s2 = __shfl_xor_sync(0xffffffffu, sr, o), c2 = __shfl_xor_sync(0xffffffffu, cr, o);
        df_two_sum(sr, s2, t, r);
        cr = (cr + c2) + r;
        sr = t;
        const float s3 = __shfl_xor_sync(0xffffffffu, si, o), c3 = __shfl_xor_sync(0xffffffffu, ci, o);
        df_two_sum(si, s3, t, r);
        ci = (ci + c3) + r;
        si = t;
      }
      if (row < m && l16 == 0) x[at(row)] = make_float2(sr + cr, si + ci);
    }
    __syncthreads();
  }
  // ascent
  for (int l = nlev - 2; l >= 0; --l) {
    enter(l);
    const int Pc = Ls[l + 1].P, npc = DIM == 3 ? Pc * Pc * Pc : Pc * Pc;
    const float2* xcv = cgsm + s_base[l + 1] + npc;  // ghosts zero, and zeros before it (b's ghosts)
    float2 k0[CG_PT], x[CG_PT];
#pragma unroll
    for (int q = 0; q < CG_PT; ++q) {
      x[q] = make_float2(0.f, 0.f);
      if (!V.on[q]) continue;
      // odd i: coarse (i - 1) / 2; even i: the mean of i / 2 - 1 and i / 2
      const int X = V.cx[q] >> 1, Y = V.cy[q] >> 1, Z = V.cz[q] >> 1;
      const int dx = (V.cx[q] & 1) ? 0 : 1, dy = (V.cy[q] & 1) ? 0 : Pc, dz = (DIM == 3 && !(V.cz[q] & 1)) ? Pc * Pc : 0;
      const float2* f = xcv + ((DIM == 3 ? Z * Pc : 0) + Y) * Pc + X;
      float2 e = make_float2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < (DIM == 3 ? 2 : 1); ++c)
#pragma unroll
        for (int bq = 0; bq < 2; ++bq) {
          const float2 v0 = f[-(c ? dz : 0) - (bq ? dy : 0)], v1 = f[-(c ? dz : 0) - (bq ? dy : 0) - dx];
          e = cadd(e, cadd(v0, v1));
        }
      const float w = DIM == 3 ? 0.125f : 0.25f;
      x[q] = cadd(V.x[V.off[q]], make_float2(e.x * w, e.y * w));
    }
#pragma unroll
    for (int q = 0; q < CG_PT; ++q)
      if (V.on[q]) V.x[V.off[q]] = x[q];
    __syncthreads();
    if constexpr (S == 0) {
      if (nu2 > 0) {
        float2 b[CG_PT];
#pragma unroll
        for (int q = 0; q < CG_PT; ++q) b[q] = V.on[q] ? V.b[V.off[q]] : make_float2(0.f, 0.f);
        int tog = 1;  // V.x has just been written with x
        for (int sw = 0; sw < nu2; ++sw)
          cg_poly<S, DIM>(V, b, x, pw + 3 * ((size_t)prob * lev_stride + l), false, tog);
        __syncthreads();  // the last step's readers of V.x are done
#pragma unroll
        for (int q = 0; q < CG_PT; ++q)
          if (V.on[q]) V.x[V.off[q]] = x[q];
        __syncthreads();
      }
    } else if (nu2 > 0) {
      float2 z0 = make_float2(0.f, 0.f);
#pragma unroll
      for (int q = 0; q < CG_PT; ++q) {
        k0[q] = make_float2(0.f, 0.f);
        if (V.on[q]) {
          const float2 p = V.apply(V.x, x[q], q, z0);
          k0[q] = csub(V.b[V.off[q]], make_float2(p.x * V.it, p.y * V.it));
          V.r[V.off[q]] = k0[q];
        }
      }
      __syncthreads();
      for (int sw = 0; sw < nu2; ++sw) {
        float2 sg[S];
        const bool wide = WIDE && Ls[l].wide;
        gram_shifts<S>(Ls[l], false, wide, sg);
        cg_sweep<S, DIM>(V, V.r, k0, x, sg, wide, sh);
        if (sw + 1 < nu2) {
#pragma unroll
          for (int q = 0; q < CG_PT; ++q)
            if (V.on[q]) V.r[V.off[q]] = k0[q];
          __syncthreads();
        }
      }
#pragma unroll
      for (int q = 0; q < CG_PT; ++q)
        if (V.on[q]) V.x[V.off[q]] = x[q];
      __syncthreads();
    }
  }
  {  // the top level's result, ghosts included
    const int P = Ls[0].P, np = DIM == 3 ? P * P * P : P * P;
    const float2* x = cgsm + s_base[0] + np;
    float2* out = Ls[0].xb;
    for (int i = tid; i < np; i += CG_THREADS) out[i] = x[i];
  }
}

}  // namespace helm

// Layout conversions between the natural (n^d) and padded ((n+1)^d) layouts, the
// sampling of a phi field onto coarse levels, and a plain natural-layout operator
// apply used by helm_apply_operator.
#include "vcycle.cuh"
#include "../../include/helm.h"
#include <algorithm>
#include <cstring>

namespace helm {

static int grid_for(size_t npts) { return (int)std::min<size_t>((npts + 255) / 256, 8192); }

__global__ void k_dense_to_padded(int dim, int n, const double2* __restrict__ src, double2* __restrict__ dst) {
  const int P = n + 1;
  const size_t npts = dim == 3 ? (size_t)P * P * P : (size_t)P * P;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npts; i += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % P), y = (int)((i / P) % P), z = dim == 3 ? (int)(i / ((size_t)P * P)) : 0;
    dst[i] = inside(x, y, z, n) ? src[((size_t)z * n + y) * n + x] : make_double2(0, 0);
  }
}

__global__ void k_padded_to_dense(int dim, int n, const double2* __restrict__ src, double2* __restrict__ dst) {
  const int P = n + 1;
  const size_t npts = dim == 3 ? (size_t)n * n * n : (size_t)n * n;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npts; i += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % n), y = (int)((i / n) % n), z = dim == 3 ? (int)(i / ((size_t)n * n)) : 0;
    dst[i] = src[pidx(x, y, z, P)];
  }
}

// Level node x (0-based) sits on fine node (x + 1) * stride - 1.
__global__ void k_scatter_phi(int dim, int n, int stride, int nf, const float* __restrict__ phi_f,
                              float* __restrict__ dst) {
  const int P = n + 1;
  const size_t npts = dim == 3 ? (size_t)P * P * P : (size_t)P * P;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npts; i += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % P), y = (int)((i / P) % P), z = dim == 3 ? (int)(i / ((size_t)P * P)) : 0;
    float v = 0.0f;
    if (inside(x, y, z, n)) {
      const size_t fx = (size_t)(x + 1) * stride - 1, fy = (size_t)(y + 1) * stride - 1;
      const size_t fz = dim == 3 ? (size_t)(z + 1) * stride - 1 : 0;
      v = phi_f[(fz * nf + fy) * nf + fx];
    }
    dst[i] = v;
  }
}

// Largest and smallest finite value of a level's field: out[0] the largest as bits ordered like
// the values, out[1] the smallest as their complement (both zero before, and if there is none).
__global__ void __launch_bounds__(256) k_phi_range(int dim, int n, const float* __restrict__ phi, unsigned* out) {
  const int P = n + 1, rows = dim == 3 ? n * n : n;
  unsigned hi = 0u, lo = 0u;
  for (int row = blockIdx.x * 8 + (threadIdx.x >> 5); row < rows; row += gridDim.x * 8) {
    const float* r = phi + (dim == 3 ? ((size_t)(row / n) * P + row % n) * P : (size_t)row * P);
    for (int x = threadIdx.x & 31; x < n; x += 32) {
      const float v = r[x];
      if (!isfinite(v)) continue;
      const unsigned b = __float_as_uint(v), o = b & 0x80000000u ? ~b : b | 0x80000000u;
      hi = max(hi, o);
      lo = max(lo, ~o);
    }
  }
  hi = __reduce_max_sync(0xffffffffu, hi);
  lo = __reduce_max_sync(0xffffffffu, lo);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(out, hi);
    atomicMax(out + 1, lo);
  }
}

// w = A v in the natural layout.  A warp holds 32 neighbouring x positions of one row and
// marches along the last axis (z in 3D, y in 2D): its coefficients of the other axes and
// three values of the march stay in registers, the remaining neighbours come from L1.
//
// complex128 is bound by the FP64 pipe (one instruction per warp and 64 cycles, comparisons
// and predicated-off ones too): seven complex products, the diagonal's sums and phi's
// conversion are 34 instructions a point.  Outside the absorbing layers H's coefficients are
// real, and almost everywhere a node's two neighbours on an axis share one coefficient, so
// an axis takes four instructions (AX_REAL), six (AX_SAME: the neighbours are added first)
// or eight (AX_ANY), and three axes that share one coefficient fourteen (EVEN).  The cases
// are uniform over a warp; each is a body of its own behind a switch, as bodies of one axis
// would be predicated and all of them paid.  Coefficients are compared on their bits and phi
// is widened on the integer pipes.  H at 255^3: 961 -> 633 us, M 959 -> 760; 2047^2 H 168 -> 118.
//
// complex64 is bound by HBM (its coefficients are narrowed on the integer pipes, those of the
// march once for a warp's rows: converting six a point on the FP64 pipe bound it): 255^3 with
// a field 488 -> 158 us, 2047^2 88 -> 21.
__device__ __forceinline__ float narrow(double v) {  // round to nearest even
  const unsigned hi = __double2hiint(v), lo = __double2loint(v), e = (hi >> 20) & 0x7ffu;
  if (((hi << 1) | lo) == 0) return __uint_as_float(hi);  // +-0
  if (e - 897u >= 254u) return (float)v;                   // subnormal, huge, infinite, NaN
  unsigned u = (hi & 0x80000000u) | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  const unsigned rest = lo & 0x1fffffffu;
  u += rest > 0x10000000u || (rest == 0x10000000u && (u & 1u));  // a carry moves the exponent up
  return __uint_as_float(u);
}
template <typename C> __device__ __forceinline__ C dense_coef(const double2* p);
template <> __device__ __forceinline__ double2 dense_coef<double2>(const double2* p) { return __ldg(p); }
template <> __device__ __forceinline__ float2 dense_coef<float2>(const double2* p) {
  const double2 v = __ldg(p);
  return make_float2(narrow(v.x), narrow(v.y));
}
enum { AX_REAL, AX_SAME, AX_ANY };
enum { EVEN = 12, GENERAL = 13 };
// (The complex shift of M is in the diagonals alone: an axis with real off-diagonals and a
// complex diagonal is AX_SAME or AX_ANY.)
__device__ __forceinline__ int axis_case(double2 a, double2 d, double2 c) {
  const long long dx = __double_as_longlong(a.x) ^ __double_as_longlong(c.x);
  const long long dy = __double_as_longlong(a.y) ^ __double_as_longlong(c.y);
  if (((__double_as_longlong(a.y) | __double_as_longlong(d.y) | __double_as_longlong(c.y)) << 1) == 0) return AX_REAL;
  return (dx | dy) == 0 ? AX_SAME : AX_ANY;
}
template <int CASE, typename C>
__device__ __forceinline__ C axis_terms(C p, C a, C c, C vm, C vp) {
  if (CASE == AX_REAL) {
    p.x = fma(a.x, vm.x, p.x);
    p.y = fma(a.x, vm.y, p.y);
    p.x = fma(c.x, vp.x, p.x);
    p.y = fma(c.x, vp.y, p.y);
    return p;
  }
  if (CASE == AX_SAME) return cfma(a, cadd(vm, vp), p);
  return cfma(c, vp, cfma(a, vm, p));
}
// One value of w: axis terms by case, then the diagonal dxy + dz - f.
template <int CX, int CY, int CZ, int DIM, typename C, typename R>
__device__ __forceinline__ C dense_point(C ax, C qx, C ay, C qy, C az, C qz, C dxy, C dz, R f, C xm, C xp, C ym, C yp,
                                         C vm, C vp, C v0) {
  constexpr bool real = CX == AX_REAL && CY == AX_REAL && CZ == AX_REAL;
  C p = axis_terms<CX>(czero<C>(), ax, qx, xm, xp);
  if (DIM == 3) p = axis_terms<CY>(p, ay, qy, ym, yp);
  p = axis_terms<CZ>(p, az, qz, vm, vp);
  C d = dxy;
  d.x += dz.x;
  d.x -= f;
  if (real) {
    p.x = fma(d.x, v0.x, p.x);
    p.y = fma(d.x, v0.y, p.y);
    return p;
  }
  d.y += dz.y;
  return cfma(d, v0, p);
}

template <typename C, int DIM>
__global__ void __launch_bounds__(256, 3)
k_apply_dense(int n, int rows, const double2* __restrict__ ca, const double2* __restrict__ cd,
              const double2* __restrict__ cc, const float* __restrict__ phi, double phic,
              const C* __restrict__ v, C* __restrict__ w) {
  typedef typename CT<C>::R R;
  const int ntx = (n + 31) / 32, nty = DIM == 3 ? (n + 7) / 8 : 1;
  const int bx = blockIdx.x % ntx, by = (blockIdx.x / ntx) % nty, bz = blockIdx.x / (ntx * nty);
  const int x = bx * 32 + threadIdx.x;
  const int y = DIM == 3 ? by * 8 + threadIdx.y : 0;              // the middle axis (3D)
  const int m0 = (DIM == 3 ? bz : bz * 8 + threadIdx.y) * rows;   // the marched axis
  const int m1 = min(m0 + rows, n);
  const bool on = x < n && y < n;
  const C zero = czero<C>();
  auto coef = [&](const double2* p, int i) { return dense_coef<C>(p + i); };
  C ax = zero, qx = zero, ay = zero, qy = zero, dx0 = zero, dy0 = zero;
  if (on) {
    ax = coef(ca, x);
    qx = coef(cc, x);
    dx0 = coef(cd, x);
    if (DIM == 3) {
      ay = coef(ca, y);
      qy = coef(cc, y);
      dy0 = coef(cd, y);
    }
  }
  const C dxy = DIM == 3 ? cadd(dx0, dy0) : dx0;
  int cx = GENERAL, cy = 0;
  bool even = false;
  if constexpr (sizeof(C) == 16) {  // uniform over the warp: lanes past the edge agree with any case
    const unsigned full = 0xffffffffu;
    const int lx = on ? axis_case(ax, dx0, qx) : -1;
    cx = __all_sync(full, lx <= AX_REAL) ? AX_REAL : __all_sync(full, lx < 0 || lx == AX_SAME) ? AX_SAME : AX_ANY;
    if (DIM == 3) {
      const int ly = on ? axis_case(ay, dy0, qy) : -1;
      cy = __all_sync(full, ly <= AX_REAL) ? AX_REAL : __all_sync(full, ly < 0 || ly == AX_SAME) ? AX_SAME : AX_ANY;
      const long long dx = __double_as_longlong(ax.x) ^ __double_as_longlong(ay.x);
      const long long dy = __double_as_longlong(ax.y) ^ __double_as_longlong(ay.y);
      even = cx == AX_SAME && cy == AX_SAME && __all_sync(full, !on || (dx | dy) == 0);
    }
  }
  const size_t plane = DIM == 3 ? (size_t)n * n : (size_t)n;      // one step of the march
  const size_t col = (size_t)y * n + x;
  const C* vc = v + col;
  auto at = [&](int m) { return on && (unsigned)m < (unsigned)n ? vc[m * plane] : zero; };
  if (m0 >= n) return;
  C la = zero, ld = zero, lc = zero;  // complex64: lane i's are those of row m0 + i (rows <= 32)
  if (sizeof(C) == 8 && m0 + (int)threadIdx.x < m1) {
    la = coef(ca, m0 + threadIdx.x);
    ld = coef(cd, m0 + threadIdx.x);
    lc = coef(cc, m0 + threadIdx.x);
  }
  C vm = at(m0 - 1), v0 = at(m0);
  for (int m = m0; m < m1; ++m) {
    const C vp = at(m + 1);
    C az, qz, dz;
    if constexpr (sizeof(C) == 8) {
      auto row = [&](C c) {
        return make_float2(__shfl_sync(0xffffffffu, c.x, m - m0), __shfl_sync(0xffffffffu, c.y, m - m0));
      };
      az = row(la), qz = row(lc), dz = row(ld);
    } else {
      az = coef(ca, m), qz = coef(cc, m), dz = coef(cd, m);
    }
    if (on) {
      const C* q = vc + m * plane;
      const C xm = x > 0 ? q[-1] : zero, xp = x < n - 1 ? q[1] : zero;
      C ym = zero, yp = zero;
      if (DIM == 3) {
        ym = y > 0 ? q[-n] : zero;
        yp = y < n - 1 ? q[n] : zero;
      }
      const size_t pp = (DIM == 3 ? ((size_t)m * (n + 1) + y) : (size_t)m) * (n + 1) + x;  // padded
      R f;
      if constexpr (sizeof(C) == 16) f = phi ? widen(__ldg(phi + pp)) : phic;
      else f = phi ? __ldg(phi + pp) : (R)phic;
      C p;
#define DENSE(X, Y, Z) dense_point<X, Y, Z, DIM>(ax, qx, ay, qy, az, qz, dxy, dz, f, xm, xp, ym, yp, vm, vp, v0)
      if constexpr (sizeof(C) == 16) {
        const int cz = axis_case(az, dz, qz);  // of the row: uniform
        int mode = cy == AX_ANY || cz == AX_ANY ? GENERAL : (cx * 2 + cy) * 2 + cz;
        if (DIM == 3 && even && cz == AX_SAME) {
          const long long dx = __double_as_longlong(ax.x) ^ __double_as_longlong(az.x);
          const long long dy = __double_as_longlong(ax.y) ^ __double_as_longlong(az.y);
          if (__all_sync(__activemask(), (dx | dy) == 0)) mode = EVEN;
        }
        switch (mode) {
          case 0: p = DENSE(AX_REAL, AX_REAL, AX_REAL); break;
          case 1: p = DENSE(AX_REAL, AX_REAL, AX_SAME); break;
          case 4: p = DENSE(AX_SAME, AX_REAL, AX_REAL); break;
          case 5: p = DENSE(AX_SAME, AX_REAL, AX_SAME); break;
          case 8: p = DENSE(AX_ANY, AX_REAL, AX_REAL); break;
          case 9: p = DENSE(AX_ANY, AX_REAL, AX_SAME); break;
          case 2: if (DIM == 3) { p = DENSE(AX_REAL, AX_SAME, AX_REAL); break; }
          case 3: if (DIM == 3) { p = DENSE(AX_REAL, AX_SAME, AX_SAME); break; }
          case 6: if (DIM == 3) { p = DENSE(AX_SAME, AX_SAME, AX_REAL); break; }
          case 7: if (DIM == 3) { p = DENSE(AX_SAME, AX_SAME, AX_SAME); break; }
          case 10: if (DIM == 3) { p = DENSE(AX_ANY, AX_SAME, AX_REAL); break; }
          case 11: if (DIM == 3) { p = DENSE(AX_ANY, AX_SAME, AX_SAME); break; }
          case EVEN:
            if (DIM == 3) {
              const C s = cadd(cadd(cadd(xm, xp), cadd(ym, yp)), cadd(vm, vp));
              p = cmul(az, s);
              C d = cadd(dxy, dz);
              d.x -= f;
              p = cfma(d, v0, p);
              break;
            }
          default: p = DENSE(AX_ANY, AX_ANY, AX_ANY); break;
        }
      } else {
        p = DENSE(AX_ANY, AX_ANY, AX_ANY);
      }
#undef DENSE
      w[col + m * plane] = p;
    }
    vm = v0;
    v0 = vp;
  }
}

void convert_dense_to_padded_c128(int dim, int n, const double2* src, double2* dst, cudaStream_t st) {
  const size_t P = n + 1;
  k_dense_to_padded<<<grid_for(dim == 3 ? P * P * P : P * P), 256, 0, st>>>(dim, n, src, dst);
}
void convert_padded_to_dense_c128(int dim, int n, const double2* src, double2* dst, cudaStream_t st) {
  const size_t nn = n;
  k_padded_to_dense<<<grid_for(dim == 3 ? nn * nn * nn : nn * nn), 256, 0, st>>>(dim, n, src, dst);
}
void scatter_phi(int dim, int n_level, int stride, int n_fine, const float* phi_f, float* dst, cudaStream_t st) {
  const size_t P = n_level + 1;
  k_scatter_phi<<<grid_for(dim == 3 ? P * P * P : P * P), 256, 0, st>>>(dim, n_level, stride, n_fine, phi_f, dst);
}
void phi_range(int dim, int n, const float* phi_pad, unsigned* out, cudaStream_t st) {
  const int rows = dim == 3 ? n * n : n;
  k_phi_range<<<std::min((rows + 7) / 8, 1024), 256, 0, st>>>(dim, n, phi_pad, out);
}
void phi_range_values(const unsigned* bits, double* lo, double* hi) {
  auto value = [](unsigned o) {
    const unsigned b = o & 0x80000000u ? o & 0x7fffffffu : ~o;
    float v;
    std::memcpy(&v, &b, sizeof v);
    return (double)v;
  };
  *hi = bits[0] ? value(bits[0]) : 0.0;
  *lo = bits[1] ? value(~bits[1]) : 0.0;
}
void apply_operator_dense(int dim, int n, const double2* ca, const double2* cd, const double2* cc,
                          const float* phi_pad, double phic, const void* v, void* w, int prec, cudaStream_t st) {
  // rows per march: 8 (a plane is read from L2 1.25 times), fewer while that leaves fewer
  // than eight warps on each SM sub-partition
  const int ntx = (n + 31) / 32, lines = dim == 3 ? ntx * ((n + 7) / 8) * 8 : ntx;
  int rows = 8;
  while (rows > 1 && (long long)lines * ((n + rows - 1) / rows) < 32LL * GB300_SMS) rows /= 2;
  const int chunks = (n + rows - 1) / rows;
  const dim3 block(32, 8);
  const int grid = dim == 3 ? ntx * ((n + 7) / 8) * chunks : ntx * ((chunks + 7) / 8);
  if (dim == 3) {
    if (prec == HELM_C128)
      k_apply_dense<double2, 3><<<grid, block, 0, st>>>(n, rows, ca, cd, cc, phi_pad, phic, (const double2*)v, (double2*)w);
    else
      k_apply_dense<float2, 3><<<grid, block, 0, st>>>(n, rows, ca, cd, cc, phi_pad, phic, (const float2*)v, (float2*)w);
  } else if (prec == HELM_C128) {
    k_apply_dense<double2, 2><<<grid, block, 0, st>>>(n, rows, ca, cd, cc, phi_pad, phic, (const double2*)v, (double2*)w);
  } else {
    k_apply_dense<float2, 2><<<grid, block, 0, st>>>(n, rows, ca, cd, cc, phi_pad, phic, (const float2*)v, (float2*)w);
  }
}

}  // namespace helm

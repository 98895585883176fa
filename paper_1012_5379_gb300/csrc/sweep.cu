// Launchers of the complex64 sweep passes (sweep.cuh) and of the complex64 coarse sub-cycle
// (coarse.cuh).
#include "sweep_launch.cuh"
#include "poly.cuh"
#include "poly.h"

#include <algorithm>

namespace helm {

// 2D levels from this size on march: 639^2 20 us a sweep against 21.7 in register regions,
// 1023^2 25 against 37; at 511^2 and below a march of few rows is mostly halo.
constexpr int SWEEP2_MARCH_N = 600;
constexpr int SWEEP3_MARCH_N = 40;

bool fused2_size(int n) { return n < SWEEP2_MARCH_N; }

SweepCfg sweep_cfg(int dim, int n, int S, int sms, bool march) {
  SweepCfg c{0, 0, 1, 0, 1};
  if (dim == 2) {
    if (n < SWEEP2_MARCH_N || S > 3 || !march) {
      // rows per warp: the fewest rounds of resident CTAs, each a fixed latency and its rows
      // (511^2: one round at 6 rows; two at 4, 21 us against 12 on the way up)
      auto pick = [&](int H, int& geo, int& units) {
        int best = -1;
        for (int qy = 2; qy <= 6; qy += 2) {
          const int u = sw2_units(H, qy, n), slots = (qy == 2 ? 3 : 2) * sms;
          const int cost = (u + slots - 1) / slots * (4 + qy);
          if (best < 0 || cost < best) {
            best = cost;
            geo = qy;
            units = u;
          }
        }
      };
      pick(S, c.geo, c.units);
      pick(S + 1, c.geo_res, c.units_res);
      return c;
    }
    // rows per march: the fewest row steps of the SM that takes the most, four CTAs per SM
    c.march = 1;
    long long best = -1;
    for (int rows = 4; rows <= 256; ++rows) {
      const long long units = sv2_units(n, rows);
      const long long steps = (units + 4LL * sms - 1) / (4LL * sms) * (rows + 2 * S + 2);
      if (best < 0 || steps < best) {
        best = steps;
        c.geo = rows;
        c.units = (int)units;
      }
    }
    c.units_res = c.units;
    c.geo_res = c.geo;
    return c;
  }
  // 3D levels from this size on march: 47^3 12 us a sweep, 63^3 14.5 against 25 in regions, 95^3
  // 23 against 42; at 31^3 both take 10
  if (n < SWEEP3_MARCH_N || !march) {
    c.geo = 4;
    c.units_res = c.units = sw3_units(S, c.geo, n);
    c.geo_res = c.geo;
    return c;
  }
  // planes per march: the fewest plane steps of the CTA that takes the most, one CTA per SM
  c.march = 1;
  long long best = -1;
  for (int pieces = 1; pieces <= 32 && pieces <= n; ++pieces) {
    const int zc = ceil_div(n, pieces);
    const long long units = sm3_units(S, n, zc);
    const long long steps = (units + sms - 1) / sms * (zc + 2 * S + 2);
    if (best < 0 || steps < best) {
      best = steps;
      c.geo = zc;
      c.units = (int)units;
    }
  }
  c.geo_res = c.geo;
  c.units_res = c.units;
  return c;
}

template <int S>
static void launch_march3(const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg, int first, int store_last,
                          bool phi, cudaStream_t st) {
  const dim3 grid(nprob * cfg.units), block(32, SM3_NW);
  const size_t smem = sm3_smem(S, cfg.geo);
  if (phi) allow_smem<k_sweep3_march<S, true>>();
  else allow_smem<k_sweep3_march<S, false>>();
  if (phi) pdl_launch(k_sweep3_march<S, true>, grid, block, smem, st, levs, cfg.units, cfg.geo, first, store_last);
  else pdl_launch(k_sweep3_march<S, false>, grid, block, smem, st, levs, cfg.units, cfg.geo, first, store_last);
}
template <int S>
static void launch_march(int dim, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg, int first,
                         int store_last, bool phi, cudaStream_t st) {
  const dim3 grid(nprob * cfg.units);
  if (dim == 2) {
    const dim3 block(32, SV2_NW);
    const size_t smem = sv2_smem(S, cfg.geo);  // at most 256 rows: below 48 KB
    if (phi) pdl_launch(k_sweep2_march<S, true>, grid, block, smem, st, levs, cfg.units, cfg.geo, first, store_last);
    else pdl_launch(k_sweep2_march<S, false>, grid, block, smem, st, levs, cfg.units, cfg.geo, first, store_last);
    return;
  }
  launch_march3<S>(levs, nprob, cfg, first, store_last, phi, st);
}

void launch_sweep(int dim, int S, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg, bool first,
                  bool store_last, bool phi, bool wide, cudaStream_t st) {
  const int f = first ? 1 : 0, sl = store_last ? 1 : 0;
  if (!cfg.march) {
    if (wide) launch_regions_wide(dim, S, levs, nprob, cfg, f, sl, st);
    else launch_regions<W_NO>(dim, S, levs, nprob, cfg, f, sl, st);
    return;
  }
  switch (S) {
    case 1: launch_march<1>(dim, levs, nprob, cfg, f, sl, phi, st); break;
    case 2: launch_march<2>(dim, levs, nprob, cfg, f, sl, phi, st); break;
    case 3: launch_march<3>(dim, levs, nprob, cfg, f, sl, phi, st); break;
    default: launch_march3<4>(levs, nprob, cfg, f, sl, phi, st); break;  // (2D: sweep_cfg marches to S = 3)
  }
}

template <int S>
static void prolong2(const LevelDev<float2>* levs, int nprob, int n, bool xk, cudaStream_t st) {
  const int ntiles = ceil_div(n + 1, 64) * ceil_div(n + 1, 16);
  pdl_launch(k_prolong2_gram<S>, dim3(nprob * ntiles), dim3(32, SW2_NW), 0, st, levs, ntiles, xk ? 1 : 0);
}

void launch_fused2(int pass, int S, const LevelDev<float2>* levs, int nprob, int nwide, int n, const SweepCfg& cfg,
                   bool xk, cudaStream_t st) {
  if (pass != FUSED2_PROLONG) {
    if (nprob > nwide) launch_fused_regions<W_NO>(pass, S, levs, nprob - nwide, cfg, st);
    if (nwide > 0) launch_fused_regions_wide(pass, S, levs + (nprob - nwide), nwide, cfg, st);
    return;
  }
  switch (S) {
    case 1: prolong2<1>(levs, nprob, n, xk, st); break;
    case 2: prolong2<2>(levs, nprob, n, xk, st); break;
    case 3: prolong2<3>(levs, nprob, n, xk, st); break;
    default: prolong2<4>(levs, nprob, n, xk, st); break;
  }
}

void record_sweep(PassSeq& q, int S, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg, bool first,
                  bool store_last) {
  const int units = first ? cfg.units : cfg.units_res;
  seq_push(q, levs, PK_ARNOLDI, S, units, first ? cfg.geo : cfg.geo_res, first, store_last, 0, 0, nprob * units);
}

size_t coarse_gram_smem(int dim, int S, const int* sizes, int nlev, bool wide) {
  size_t total = 0;
  for (int l = 0; l < nlev; ++l) {
    const size_t P = sizes[l] + 1, np = dim == 3 ? P * P * P : P * P;
    total += np / P + cg_vectors(S, wide) * np;
  }
  return total * sizeof(float2);
}

void launch_coarse_gram(int dim, int S, const LevelDev<float2>* levs, int lev_stride, const CoarseLU* lus, int nprob,
                        int nwide, const float2* pw, int nu1, int nu2, bool from_res, size_t smem, cudaStream_t st) {
  const int m = nprob - nwide;
  const CoarseArgs a{lev_stride, pw, nu1, nu2, from_res ? 1 : 0, smem};
  if (m > 0) {
    if (S == 0) {
      if (dim == 2) launch_coarse_sd<0, 2, W_NO>(levs, lus, m, a, st);
      else launch_coarse_sd<0, 3, W_NO>(levs, lus, m, a, st);
    } else {
      launch_coarse_s<W_NO>(dim, S, levs, lus, m, a, st);
    }
  }
  if (nwide > 0) launch_coarse_wide(dim, S, levs + (size_t)m * lev_stride, lus + m, nwide, a, st);
}

template <int SRC, int END>
static void poly2(const LevelDev<float2>* levs, const float2* pw, int nprob, int n, int src, int dst, cudaStream_t st) {
  // regions of 16 rows while 32-row ones would leave SMs idle (1023^2: 1849 of the larger)
  if (n <= 300) {
    const int units = po_units(2, SRC, END, n);
    pdl_launch(k_poly2<2, SRC, END>, dim3(nprob * units), dim3(32, SW2_NW), 0, st, levs, pw, units, src, dst);
  } else {
    const int units = po_units(4, SRC, END, n);
    pdl_launch(k_poly2<4, SRC, END>, dim3(nprob * units), dim3(32, SW2_NW), 0, st, levs, pw, units, src, dst);
  }
}

void launch_poly2(const LevelDev<float2>* levs, const float2* pw, int nprob, int n, int from, int src, int dst,
                  bool restrict_end, cudaStream_t st) {
  if (from == POLY_FROM_COARSE) poly2<2, 0>(levs, pw, nprob, n, src, dst, st);
  else if (from == POLY_FROM_ZERO && restrict_end) poly2<0, 1>(levs, pw, nprob, n, src, dst, st);
  else if (from == POLY_FROM_ZERO) poly2<0, 0>(levs, pw, nprob, n, src, dst, st);
  else if (restrict_end) poly2<1, 1>(levs, pw, nprob, n, src, dst, st);
  else poly2<1, 0>(levs, pw, nprob, n, src, dst, st);
}

}  // namespace helm

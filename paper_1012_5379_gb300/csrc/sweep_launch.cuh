// Launchers of the complex64 sweep passes whose CTAs hold a region (sweep.cuh) and of the coarse
// sub-cycle (coarse.cuh), for levels of one kind W: sweep.cu instantiates them for ordinary
// levels, sweep_wide.cu for wide ones.
#pragma once
#include "sweep.cuh"
#include "coarse.cuh"
#include "launch.cuh"

namespace helm {

template <int S, int W>
static void launch_regions_s(int dim, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg, int first,
                             int store_last, cudaStream_t st) {
  const int units = first ? cfg.units : cfg.units_res, geo = first ? cfg.geo : cfg.geo_res;
  const dim3 grid(nprob * units), block(32, 8);
  static_assert(SW2_NW == 8 && SW3_NW == 8, "one block shape");
  if (dim == 2) {
    if (geo == 2) pdl_launch(k_sweep2<S, 2, W>, grid, block, 0, st, levs, units, first, store_last);
    else if (geo == 4) pdl_launch(k_sweep2<S, 4, W>, grid, block, 0, st, levs, units, first, store_last);
    else pdl_launch(k_sweep2<S, 6, W>, grid, block, 0, st, levs, units, first, store_last);
    return;
  }
  allow_smem<k_sweep3<S, 4, W>>();
  pdl_launch(k_sweep3<S, 4, W>, grid, block, sw3_smem(S, 4), st, levs, units, first, store_last);
}
template <int W>
static void launch_regions(int dim, int S, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg, int first,
                           int store_last, cudaStream_t st) {
  switch (S) {
    case 1: launch_regions_s<1, W>(dim, levs, nprob, cfg, first, store_last, st); break;
    case 2: launch_regions_s<2, W>(dim, levs, nprob, cfg, first, store_last, st); break;
    case 3: launch_regions_s<3, W>(dim, levs, nprob, cfg, first, store_last, st); break;
    default: launch_regions_s<4, W>(dim, levs, nprob, cfg, first, store_last, st); break;
  }
}

template <int S, int W>
static void launch_fused_regions_s(int pass, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg,
                                   cudaStream_t st) {
  const dim3 block(32, SW2_NW);
  if (pass == FUSED2_DOWN) {
    const dim3 grid(nprob * cfg.units);
    if (cfg.geo == 2) pdl_launch(k_sweep2_down<S, 2, W>, grid, block, 0, st, levs, cfg.units);
    else if (cfg.geo == 4) pdl_launch(k_sweep2_down<S, 4, W>, grid, block, 0, st, levs, cfg.units);
    else pdl_launch(k_sweep2_down<S, 6, W>, grid, block, 0, st, levs, cfg.units);
  } else {
    const dim3 grid(nprob * cfg.units_res);
    if (cfg.geo_res == 2) pdl_launch(k_sweep2_up<S, 2, W>, grid, block, 0, st, levs, cfg.units_res);
    else if (cfg.geo_res == 4) pdl_launch(k_sweep2_up<S, 4, W>, grid, block, 0, st, levs, cfg.units_res);
    else pdl_launch(k_sweep2_up<S, 6, W>, grid, block, 0, st, levs, cfg.units_res);
  }
}
template <int W>
static void launch_fused_regions(int pass, int S, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg,
                                 cudaStream_t st) {
  switch (S) {
    case 1: launch_fused_regions_s<1, W>(pass, levs, nprob, cfg, st); break;
    case 2: launch_fused_regions_s<2, W>(pass, levs, nprob, cfg, st); break;
    case 3: launch_fused_regions_s<3, W>(pass, levs, nprob, cfg, st); break;
    default: launch_fused_regions_s<4, W>(pass, levs, nprob, cfg, st); break;
  }
}

struct CoarseArgs {
  int lev_stride;
  const float2* pw;
  int nu1, nu2, from_res;
  size_t smem;
};
template <int S, int DIM, int W>
static void launch_coarse_sd(const LevelDev<float2>* levs, const CoarseLU* lus, int nprob, const CoarseArgs& a,
                             cudaStream_t st) {
  allow_smem<k_coarse_gram<S, DIM, W>>();
  pdl_launch(k_coarse_gram<S, DIM, W>, dim3(nprob), dim3(CG_THREADS), a.smem, st, levs, a.lev_stride, lus, a.pw, a.nu1,
             a.nu2, a.from_res);
}
template <int W>
static void launch_coarse_s(int dim, int S, const LevelDev<float2>* levs, const CoarseLU* lus, int nprob,
                            const CoarseArgs& a, cudaStream_t st) {
#define HELM_CG(SS)                                                      \
  case SS:                                                               \
    if (dim == 2) launch_coarse_sd<SS, 2, W>(levs, lus, nprob, a, st);   \
    else launch_coarse_sd<SS, 3, W>(levs, lus, nprob, a, st);            \
    break;
  switch (S) {
    HELM_CG(1)
    HELM_CG(2)
    HELM_CG(3)
    HELM_CG(4)
  }
#undef HELM_CG
}

// sweep_wide.cu
void launch_regions_wide(int dim, int S, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg, int first,
                         int store_last, cudaStream_t st);
void launch_fused_regions_wide(int pass, int S, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg,
                               cudaStream_t st);
void launch_coarse_wide(int dim, int S, const LevelDev<float2>* levs, const CoarseLU* lus, int nprob,
                        const CoarseArgs& a, cudaStream_t st);

}  // namespace helm

// Host launchers of the V-cycle kernels, instantiated once per precision in
// vcycle_c64.cu and vcycle_c128.cu (two translation units compile in parallel).
#pragma once
#include "tiles.cuh"
#include "launch.cuh"
#include <algorithm>
#include <type_traits>
#include "../../include/helm.h"
#include "poly.h"

namespace helm {

// Tiles per CTA of a 2D pass for one problem of `ntiles` tiles: each CTA pays a fixed
// cost (its reduction, the atomic, the ramp; about half a tile's time on GB300) plus
// the cost of its tiles, so t tiles per CTA take ceil(ntiles / (t slots)) rounds of
// (1/2 + t) tile times; the smallest such t up to 8 wins.  A function of the level size and of the kernel's
// residency on the device only (it fixes the order of the pass's partial sums).
template <typename K>
static int tiles_per_cta(K kernel, int ntiles, size_t smem = 0) {
  static thread_local K last_kernel = nullptr;
  static thread_local int slots = 0;
  if (kernel != last_kernel) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, smem) != cudaSuccess || per_sm < 1)
      per_sm = 1;
    slots = per_sm * sm_count();
    last_kernel = kernel;
  }
  int best = 1;
  long long best_cost = -1;
  for (int t = 1; t <= 8; t *= 2) {
    const long long rounds = (ntiles + (long long)t * slots - 1) / ((long long)t * slots);
    const long long cost = rounds * (1 + 2 * t);
    if (best_cost < 0 || cost < best_cost) { best = t; best_cost = cost; }
  }
  return best;
}

// The post-smoothing residual of a 3D complex64 level, x_b streamed by TMA.
template <int QY>
static void resid_tma3(const LevelDev<float2>* levs, int nprob, int P, const Tma3Params& tp, cudaStream_t st) {
  const size_t smem = tma3_smem(1, QY, tp.stages);
  thread_local int occ_stages = -1, occ = 1;  // per host thread: the residency of the last configuration
  allow_smem<k_resid_tma3<QY>>();
  if (occ_stages != tp.stages) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_resid_tma3<QY>, 256, smem) != cudaSuccess || occ < 1)
      occ = 1;
    occ_stages = tp.stages;
  }
  // shares of the level's (column, plane) sequence: column pieces, or one per resident CTA
  const long long cols = tma3_cols(P, QY);
  long long units = tp.pieces > 0 ? cols * std::min(tp.pieces, P) : (long long)occ * sm_count();
  units = std::max<long long>(1, std::min<long long>(units, std::min<long long>(TMA3_MAX_UNITS, cols * P)));
  pdl_launch(k_resid_tma3<QY>, dim3(nprob * (int)units), dim3(32, 8), smem, st, levs, (int)units, tp.stages);
}

// Coarse correction and post-smoothing residual of a 3D complex64 level in two passes:
// x_b = x_a + P e_c row by row, then r0 = b - M x_b with x_b streamed by TMA.
static void prolong_tma3(const LevelDev<float2>* levs, int nprob, int P, cudaStream_t st) {
  const Tma3Params tp = tma3_params(TP_PROLONG, P);
  const int nblk = std::max(1, std::min(8 * sm_count() / std::max(nprob, 1), (P / PR_ROWS) * P));
  if (P <= 256)
    pdl_launch(k_prolong3_rows<float2, 1>, dim3(nprob * nblk), dim3(256), 0, st, levs, nblk);
  else if (P <= 512)
    pdl_launch(k_prolong3_rows<float2, 2>, dim3(nprob * nblk), dim3(256), 0, st, levs, nblk);
  else
    pdl_launch(k_prolong3_rows<float2, 4>, dim3(nprob * nblk), dim3(256), 0, st, levs, nblk);
  if (tp.qy == 4)
    resid_tma3<4>(levs, nprob, P, tp, st);
  else
    resid_tma3<2>(levs, nprob, P, tp, st);
}

// Arnoldi steps one pass at a time (complex128; complex64 sweeps: sweep.cu).
template <typename C, int J>
static void arnoldi_J(int dim, const LevelDev<C>* levs, int grid, int ntiles, TileCfg cfg, bool r0_is_b,
                      bool store_p, cudaStream_t st) {
  if (dim == 2) {
    auto* const kern = tile2_q(cfg.P) == 1 ? k_arnoldi_t2<C, J, 1> : k_arnoldi_t2<C, J, 2>;
    const int t = tuned_tpc(TP_ARNOLDI, cfg.P, (int)sizeof(C), J, tiles_per_cta(kern, ntiles));
    pdl_launch(kern, dim3(grid / ntiles * ceil_div(ntiles, t)), dim3(dim3(32, 8)), 0, st, levs, ntiles, t, r0_is_b,
               store_p);
  }
  else
    pdl_launch(k_arnoldi_t3<C, J>, dim3(grid), dim3(dim3(32, 8)), 0, st, levs, ntiles, cfg.rows, r0_is_b, store_p);
}

template <typename C>
void launch_arnoldi(int dim, int J, const LevelDev<C>* levs, int nprob, int ntiles, TileCfg cfg, bool r0_is_b,
                    bool store_p, cudaStream_t st) {
  const int grid = nprob * ntiles;
  switch (J) {
    case 1: arnoldi_J<C, 1>(dim, levs, grid, ntiles, cfg, r0_is_b, store_p, st); break;
    case 2: arnoldi_J<C, 2>(dim, levs, grid, ntiles, cfg, r0_is_b, store_p, st); break;
    case 3: arnoldi_J<C, 3>(dim, levs, grid, ntiles, cfg, r0_is_b, store_p, st); break;
    default: arnoldi_J<C, 4>(dim, levs, grid, ntiles, cfg, r0_is_b, store_p, st); break;
  }
}

// The TMA-fed 3D restriction (complex64 levels of pitch 128..1024 with tensor maps).
static void restrict_tma3(const LevelDev<float2>* levs, int nprob, int P, bool r0_is_b, bool x_from_zero,
                          bool nosmooth, int nraw, cudaStream_t st) {
  const Tma3Params tp = tma3_params(TP_RESTRICT, P);
  const size_t smem = (size_t)tp.stages * nraw * tm3_box_stride(2);
  thread_local int occ_key = -1, occ = 1;
  allow_smem<k_restrict_tma3<SMAX>>();
  const int key = tp.stages * 16 + nraw;
  if (occ_key != key) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_restrict_tma3<SMAX>, 256, smem) != cudaSuccess || occ < 1)
      occ = 1;
    occ_key = key;
  }
  const long long cols = tma3_cols(P, 2);
  long long units = tp.pieces > 0 ? cols * std::min(tp.pieces, P) : (long long)occ * sm_count();
  units = std::max<long long>(1, std::min<long long>(units, std::min<long long>(TMA3_MAX_UNITS, cols * P)));
  pdl_launch(k_restrict_tma3<SMAX>, dim3(nprob * (int)units), dim3(32, 8), smem, st, levs, (int)units, tp.stages,
             r0_is_b ? 1 : 0, x_from_zero ? 1 : 0, nosmooth ? 1 : 0);
}

template <typename C>
void launch_restrict(int dim, const LevelDev<C>* levs, int nprob, int ntiles, TileCfg cfg, bool r0_is_b,
                     bool x_from_zero, bool nosmooth, cudaStream_t st, bool tma, int nraw) {
  if constexpr (std::is_same<C, float2>::value) {
    if (dim == 3 && tma && cfg.P >= TMA3_MIN_P && cfg.P <= TMA3_MAX_P && tma3_params(TP_RESTRICT, cfg.P).enabled) {
      restrict_tma3(levs, nprob, cfg.P, r0_is_b, x_from_zero, nosmooth, nraw, st);
      return;
    }
  }
  if (dim == 2) {
    auto* const kern = tile2_q(cfg.P) == 1 ? k_restrict_t2<C, 1> : k_restrict_t2<C, 2>;
    const int t = tuned_tpc(TP_RESTRICT, cfg.P, (int)sizeof(C), 0, tiles_per_cta(kern, ntiles));
    pdl_launch(kern, dim3(nprob * ceil_div(ntiles, t)), dim3(dim3(32, 8)), 0, st, levs, ntiles, t, r0_is_b,
               x_from_zero, nosmooth);
  } else
    pdl_launch(k_restrict_t3<C>, dim3(nprob * ntiles), dim3(dim3(32, 8)), 0, st, levs, ntiles, cfg.rows, r0_is_b, x_from_zero, nosmooth);
}

template <typename C>
void launch_update_flat(int dim, UpdateMode mode, const LevelDev<C>* levs, int nprob, int ntiles, bool r0_is_b,
                        int xsel, bool x_from_zero, cudaStream_t st) {
  pdl_launch(k_update_flat<C>, dim3(nprob * ntiles), dim3(256), 0, st, levs, ntiles, dim, (int)mode, r0_is_b, xsel, x_from_zero);
}

template <typename C>
void launch_prolong(int dim, bool with_residual, const LevelDev<C>* levs, int nprob, int ntiles, TileCfg cfg,
                    bool tma, cudaStream_t st) {
  if constexpr (std::is_same<C, float2>::value) {
    if (prolong_kernels(dim, with_residual, (int)sizeof(C), tma, cfg.P) == 2) {
      prolong_tma3(levs, nprob, cfg.P, st);
      return;
    }
  }
  if (!with_residual) {
    pdl_launch(k_prolong_flat<C>, dim3(nprob * ntiles), dim3(256), 0, st, levs, ntiles, dim);
  } else if (dim == 2) {
    auto* const kern = tile2_q(cfg.P) == 1 ? k_prolong_t2<C, 1> : k_prolong_t2<C, 2>;
    const int t = tuned_tpc(TP_PROLONG, cfg.P, (int)sizeof(C), 0, tiles_per_cta(kern, ntiles));
    pdl_launch(kern, dim3(nprob * ceil_div(ntiles, t)), dim3(dim3(32, 8)), 0, st, levs, ntiles, t);
  } else {
    pdl_launch(k_prolong_t3<C>, dim3(nprob * ntiles), dim3(dim3(32, 8)), 0, st, levs, ntiles, cfg.rows);
  }
}

template <typename C>
void launch_coarse(int dim, const LevelDev<C>* levs, int nlev, int lev_stride, const CoarseLU* lus, int nprob,
                   int nu1, int nu2, cudaStream_t st) {
  pdl_launch(k_coarse<C>, dim3(nprob), dim3(512), 0, st, levs, nlev, lev_stride, lus, nu1, nu2, dim);
}

template <typename C>
void launch_coarse_smem(int dim, const LevelDev<C>* levs, int nlev, int lev_stride, const CoarseLU* lus, int nprob,
                        int nu1, int nu2, size_t smem_bytes, cudaStream_t st) {
  allow_smem<k_coarse_smem<C>>();
  pdl_launch(k_coarse_smem<C>, dim3(nprob), dim3(512), smem_bytes, st, levs, nlev, lev_stride, lus, nu1, nu2, dim);
}

template <typename C>
void launch_load_input(int dim, const LevelDev<C>* levs, int ntiles, const void* src, int in_prec, cudaStream_t st) {
  if (in_prec == HELM_C128)
    pdl_launch(k_load_input<double2, C>, dim3(ntiles), dim3(256), 0, st, levs, ntiles, dim, (const double2*)src);
  else
    pdl_launch(k_load_input<float2, C>, dim3(ntiles), dim3(256), 0, st, levs, ntiles, dim, (const float2*)src);
}

template <typename C>
void launch_store_output(int dim, int n, const LevelDev<C>* levs, bool update, void* dst, int out_prec, cudaStream_t st) {
  const size_t items = (dim == 3 ? (size_t)n * n : (size_t)n) * ceil_div(n, 32 * IO_XPT);  // a warp's share
  const int grid = (int)std::min<size_t>((items + 7) / 8, (size_t)8 * sm_count());
  if (out_prec == HELM_C128)
    pdl_launch(k_store_output<C, double2>, dim3(grid), dim3(256), 0, st, levs, dim, update ? 1 : 0, (double2*)dst);
  else
    pdl_launch(k_store_output<C, float2>, dim3(grid), dim3(256), 0, st, levs, dim, update ? 1 : 0, (float2*)dst);
}

template <typename C>
void launch_poly_step(int dim, const LevelDev<C>* levs, const C* pw, int nprob, int nflat, int src, int dst,
                      int wsel, cudaStream_t st) {
  pdl_launch(k_poly_step<C>, dim3(nprob * nflat), dim3(256), 0, st, levs, pw, nflat, dim, src, dst, wsel);
}

template <typename C>
void launch_poly_restrict(int dim, const LevelDev<C>* levs, int nprob, int nflat, int src, cudaStream_t st) {
  pdl_launch(k_poly_residual<C>, dim3(nprob * nflat), dim3(256), 0, st, levs, nflat, dim, src);
  pdl_launch(k_poly_fw<C>, dim3(nprob * nflat), dim3(256), 0, st, levs, nflat, dim);
}

// ------------------------------------------------------------------ persistent segments
// The recorders append the pass an ordinary launch would run (the same launch
// parameters, so the same partial-sum order) to a pass list instead of launching it.
template <typename C, int J>
static void record_arnoldi_J(PassSeq& q, int dim, const LevelDev<C>* levs, int nprob, int ntiles, TileCfg cfg,
                             bool r0_is_b, bool store_p) {
  if (dim == 2) {
    const int t = tuned_tpc(TP_ARNOLDI, cfg.P, (int)sizeof(C), J, tiles_per_cta(k_arnoldi_t2<C, J, 1>, ntiles));
    seq_push(q, levs, PK_ARNOLDI, J, ntiles, t, r0_is_b, store_p, 0, 0, nprob * ceil_div(ntiles, t));
  } else {
    seq_push(q, levs, PK_ARNOLDI, J, ntiles, cfg.rows, r0_is_b, store_p, 0, 0, nprob * ntiles);
  }
}

template <typename C>
void record_arnoldi(PassSeq& q, int dim, int J, const LevelDev<C>* levs, int nprob, int ntiles, TileCfg cfg,
                    bool r0_is_b, bool store_p) {
  switch (J) {
    case 1: record_arnoldi_J<C, 1>(q, dim, levs, nprob, ntiles, cfg, r0_is_b, store_p); break;
    case 2: record_arnoldi_J<C, 2>(q, dim, levs, nprob, ntiles, cfg, r0_is_b, store_p); break;
    case 3: record_arnoldi_J<C, 3>(q, dim, levs, nprob, ntiles, cfg, r0_is_b, store_p); break;
    default: record_arnoldi_J<C, 4>(q, dim, levs, nprob, ntiles, cfg, r0_is_b, store_p); break;
  }
}

template <typename C>
void record_restrict(PassSeq& q, int dim, const LevelDev<C>* levs, int nprob, int ntiles, TileCfg cfg, bool r0_is_b,
                     bool x_from_zero, bool nosmooth) {
  if (dim == 2) {
    const int t = tuned_tpc(TP_RESTRICT, cfg.P, (int)sizeof(C), 0, tiles_per_cta(k_restrict_t2<C, 1>, ntiles));
    seq_push(q, levs, PK_RESTRICT, 0, ntiles, t, r0_is_b, x_from_zero, nosmooth, 0, nprob * ceil_div(ntiles, t));
  } else {
    seq_push(q, levs, PK_RESTRICT, 0, ntiles, cfg.rows, r0_is_b, x_from_zero, nosmooth, 0, nprob * ntiles);
  }
}

template <typename C>
void record_update(PassSeq& q, int dim, UpdateMode mode, const LevelDev<C>* levs, int nprob, int ntiles, bool r0_is_b,
                   int xsel, bool x_from_zero) {
  (void)dim;
  seq_push(q, levs, PK_UPDATE, 0, ntiles, 0, (int)mode, r0_is_b, xsel, x_from_zero, nprob * ntiles);
}

template <typename C>
void record_prolong(PassSeq& q, int dim, bool with_residual, const LevelDev<C>* levs, int nprob, int ntiles,
                    TileCfg cfg) {
  if (!with_residual) {
    seq_push(q, levs, PK_PROLONG_FLAT, 0, ntiles, 0, 0, 0, 0, 0, nprob * ntiles);
  } else if (dim == 2) {
    const int t = tuned_tpc(TP_PROLONG, cfg.P, (int)sizeof(C), 0, tiles_per_cta(k_prolong_t2<C, 1>, ntiles));
    seq_push(q, levs, PK_PROLONG, 0, ntiles, t, 0, 0, 0, 0, nprob * ceil_div(ntiles, t));
  } else {
    seq_push(q, levs, PK_PROLONG, 0, ntiles, cfg.rows, 0, 0, 0, 0, nprob * ntiles);
  }
}

// One cooperative launch of the pass list: every CTA resident (the grid barrier needs
// it), at most as many CTAs as the largest pass has virtual blocks.
template <typename C>
int launch_seq(int dim, const PassSeq& q, GridBar* gb, unsigned long long limit_ns, cudaStream_t st) {
  if (q.npass == 0) return 0;
  void (*kern)(const PassSeq, GridBar*, unsigned long long) = dim == 2 ? k_vcycle_seq<C, 2> : k_vcycle_seq<C, 3>;
  // shared memory of the complex64 sweep pass
  const size_t smem = sizeof(C) != 8 ? 0 : dim == 3 ? sw3_smem(SMAX, SEQ_O3) : sizeof(Sw2Shared<SMAX, 6>);
  thread_local void (*last)(const PassSeq, GridBar*, unsigned long long) = nullptr;
  thread_local int occ = 1;
  if (kern != last) {
    if (smem) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 256, smem) != cudaSuccess || occ < 1) occ = 1;
    last = kern;
  }
  int maxv = 1;
  for (int i = 0; i < q.npass; ++i) maxv = std::max(maxv, q.p[i].nvblk);
  const int grid = std::max(1, std::min(maxv, occ * sm_count()));
  cudaError_t e = cudaMemsetAsync(gb, 0, sizeof(GridBar), st);
  if (e != cudaSuccess) return (int)e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(32, 8);  // the tile passes' shape; the flat passes use the flat thread index
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, q, gb, limit_ns);
  return (int)e;
}

#define HELM_VCYCLE_INST(C)                                                                                   \
  template void launch_restrict<C>(int, const LevelDev<C>*, int, int, TileCfg, bool, bool, bool,           \
                                    cudaStream_t, bool, int);                                               \
  template void launch_update_flat<C>(int, UpdateMode, const LevelDev<C>*, int, int, bool, int, bool,         \
                                      cudaStream_t);                                                          \
  template void launch_prolong<C>(int, bool, const LevelDev<C>*, int, int, TileCfg, bool, cudaStream_t);      \
  template void launch_coarse<C>(int, const LevelDev<C>*, int, int, const CoarseLU*, int, int, int,           \
                                 cudaStream_t);                                                               \
  template void launch_load_input<C>(int, const LevelDev<C>*, int, const void*, int, cudaStream_t);           \
  template void launch_store_output<C>(int, int, const LevelDev<C>*, bool, void*, int, cudaStream_t);        \
  template void launch_poly_step<C>(int, const LevelDev<C>*, const C*, int, int, int, int, int, cudaStream_t); \
  template void launch_poly_restrict<C>(int, const LevelDev<C>*, int, int, int, cudaStream_t);                \
  template void record_restrict<C>(PassSeq&, int, const LevelDev<C>*, int, int, TileCfg, bool, bool, bool);    \
  template void record_update<C>(PassSeq&, int, UpdateMode, const LevelDev<C>*, int, int, bool, int, bool);    \
  template void record_prolong<C>(PassSeq&, int, bool, const LevelDev<C>*, int, int, TileCfg);                 \
  template int launch_seq<C>(int, const PassSeq&, GridBar*, unsigned long long, cudaStream_t);

}  // namespace helm

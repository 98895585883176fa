// The complex64 sweep passes and coarse sub-cycle of wide levels: double-float Gram sums
// (gram.cuh).  Beside the ordinary ones because the sums' registers would cost those their third
// CTA per SM (1023^2: 171 us a V-cycle with one kernel for both, 157 apart).
#include "sweep_launch.cuh"

namespace helm {

void launch_regions_wide(int dim, int S, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg, int first,
                         int store_last, cudaStream_t st) {
  launch_regions<W_YES>(dim, S, levs, nprob, cfg, first, store_last, st);
}
void launch_fused_regions_wide(int pass, int S, const LevelDev<float2>* levs, int nprob, const SweepCfg& cfg,
                               cudaStream_t st) {
  launch_fused_regions<W_YES>(pass, S, levs, nprob, cfg, st);
}
void launch_coarse_wide(int dim, int S, const LevelDev<float2>* levs, const CoarseLU* lus, int nprob,
                        const CoarseArgs& a, cudaStream_t st) {
  launch_coarse_s<W_YES>(dim, S, levs, lus, nprob, a, st);
}

}  // namespace helm

// Complex FP64 (HELM_C128) instantiation of the V-cycle kernels.
#include "vcycle_launch.cuh"
namespace helm {
HELM_VCYCLE_INST(double2)
template void launch_arnoldi<double2>(int, int, const LevelDev<double2>*, int, int, TileCfg, bool, bool, cudaStream_t);
template void record_arnoldi<double2>(PassSeq&, int, int, const LevelDev<double2>*, int, int, TileCfg, bool, bool);
template void launch_coarse_smem<double2>(int, const LevelDev<double2>*, int, int, const CoarseLU*, int, int, int,
                                          size_t, cudaStream_t);

// This translation unit's copy of the V-cycle error flag (the complex128 kernels'):
// read and clear.
int vcycle_take_error_c128() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_vcycle_error, sizeof(int)) != cudaSuccess) return 1;
  if (v) {
    const int z = 0;
    cudaMemcpyToSymbol(g_vcycle_error, &z, sizeof(int));
  }
  return v;
}
}

// Kernel launches with programmatic stream serialisation, and the SM count.
#pragma once
#include <cuda_runtime.h>
#include "helm_internal.h"

namespace helm {

// Launch with programmatic stream serialisation: the kernel may start while its
// predecessor finishes and synchronises with it through griddepcontrol.wait.  The
// passes that end in a grid reduction signal their dependents only after their main
// work, so waiting dependents never hold SM slots the predecessor's later waves need;
// the launch latency and the dependent's prologue then overlap the predecessor's
// reduction tail.
static inline int sm_count() {
  // initialised once, thread-safely (serving and callers' threads launch concurrently)
  static const int n = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 1;
    return v;
  }();
  return n;
}
// Allow a kernel the largest dynamic shared memory the device offers beside its static part,
// once per host thread.  The limit belongs to the kernel, not to the thread: every thread must
// set the same value, or one would take back what another counts on.
template <auto Kern>
static inline void allow_smem() {
  thread_local bool done = false;
  if (done) return;
  int dev = 0, optin = 0;
  cudaFuncAttributes fa;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (cudaFuncGetAttributes(&fa, Kern) == cudaSuccess && optin > (int)fa.sharedSizeBytes)
    cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
  done = true;
}
template <typename... KArgs, typename... Args>
static inline void pdl_launch(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// Append a pass to the list of a persistent segment.
static inline void seq_push(PassSeq& q, const void* levs, int kind, int J, int ntiles, int geo, int f0, int f1, int f2,
                            int f3, int nvblk) {
  if (q.npass >= SEQ_MAX) return;  // the caller sizes its lists (checked by the engine)
  PassDesc& d = q.p[q.npass++];
  d.levs = levs;
  d.kind = kind;
  d.J = J;
  d.ntiles = ntiles;
  d.geo = geo;
  d.f0 = f0;
  d.f1 = f1;
  d.f2 = f2;
  d.f3 = f3;
  d.nvblk = nvblk;
}

}  // namespace helm

// The tail kernels of the default steps, without and with the helix in a field (variants 0 and
// 8 of step_transport), for contexts with species kernels and, with the rounding of that form,
// with the fused one, and the launch of every variant's.
#include <cuda_runtime.h>

#include <algorithm>

#include "layout.h"
#include "tail.cuh"

namespace adept {

template <class R>
static const void* tail_fn(int variant, bool fused) {
  if (fused) return (variant & 8) ? (const void*)k_tail<R, 0, 24> : (const void*)k_tail<R, 0, 16>;
  if (variant & 5) return tail_variant_fn(sizeof(R) == 4, variant);
  return (variant & 8) ? (const void*)k_tail<R, 0, 8> : (const void*)k_tail<R, 0, 0>;
}

static void tail_config(const Params& P, cudaLaunchConfig_t& cfg, cudaLaunchAttribute& at, int blocks, cudaStream_t st) {
  cfg = {};
  cfg.dynamicSmemBytes = P.tail_shared;
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = blocks;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
}

static const void* tail_fn(const Params& P, int precision, bool fused) {
  return precision ? tail_fn<float>(transport_variant(P), fused) : tail_fn<double>(transport_variant(P), fused);
}

// The limit on dynamic shared memory belongs to the kernel, which every context of the process on
// this device launches, each with its own tables: it is set to the most there is, whatever this
// context needs, so that no context takes it from another and inits at the same time agree.
uint32_t tail_shared_bytes(const Params& P, int precision, bool fused) {
  uint32_t n = 0;
  for (int s = 0; s < 3; ++s) n = std::max(n, precision ? tail_units<float>(P, s) : tail_units<double>(P, s));
  const void* fn = tail_fn(P, precision, fused);
  cudaFuncAttributes fa;
  int dev = 0, most = 0;
  if (cudaFuncGetAttributes(&fa, fn) == cudaSuccess && cudaGetDevice(&dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
      16u * n + fa.sharedSizeBytes <= (size_t)most &&
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes) == cudaSuccess)
    return 16u * n;
  (void)cudaGetLastError();
  return 0;  // too many materials or volumes: read where they are
}

int tail_blocks(const Params& P, int precision, bool fused) {
  const void* fn = tail_fn(P, precision, fused);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  tail_config(P, cfg, at, 16, nullptr);
  int n = 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess && n > 0)
    return 16;
  (void)cudaGetLastError();
  return 8;
}

cudaError_t launch_tail(const Params& P, int precision, bool fused, int blocks, uint32_t max_gens, int b, cudaStream_t st) {
  void* args[] = {const_cast<Params*>(&P), &max_gens, &b};
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  tail_config(P, cfg, at, blocks, st);
  return cudaLaunchKernelExC(&cfg, tail_fn(P, precision, fused), args);
}

}  // namespace adept

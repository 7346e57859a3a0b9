// tile.cu -- instantiations of the register-tiled kernels (their own translation unit, compiled in
// parallel with hot.cu); see tile_kernels.cuh.
#include "tile.h"

#include <algorithm>

namespace hot_tile {

namespace {

// Raises the kernels' dynamic shared-memory limit to the device's (their blocks size themselves).
cudaError_t set_smem() {
  int dev = 0, most = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  auto raise = [&](auto *kernel) {
    cudaFuncAttributes f;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&f, kernel);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, at, most - (int)f.sharedSizeBytes);
  };
  raise(hot::gsw_tile_kernel<true, true, false>);
  raise(hot::gsw_tile_kernel<false, true, false>);
  raise(hot::gsw_tile_kernel<true, false, false>);
  raise(hot::gsw_tile_kernel<true, false, true>);
  raise(hot::gsw_tile_persistent_kernel);
  return e;
}

}  // namespace

cudaError_t occupancy(int M, int team, int pairs, int *per_sm) {
  int a = 0, b = 0;
  const int smem = hot::tile_smem_bytes(M, team, pairs);
  *per_sm = 0;
  cudaError_t e = set_smem();
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, hot::gsw_tile_kernel<true, true, false>, hot::kThreads, smem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, hot::gsw_tile_persistent_kernel, hot::kThreads, smem);
  *per_sm = std::min(a, b);
  return e;
}

cudaError_t launch(bool back, bool fwd, bool adj, cudaLaunchConfig_t cfg, const hot::TileArgs &a) {
  cfg.dynamicSmemBytes = hot::tile_smem_bytes(a.s.M, a.team, a.pairs);
  if (adj) return cudaLaunchKernelEx(&cfg, hot::gsw_tile_kernel<true, false, true>, a);
  if (back && fwd) return cudaLaunchKernelEx(&cfg, hot::gsw_tile_kernel<true, true, false>, a);
  if (back) return cudaLaunchKernelEx(&cfg, hot::gsw_tile_kernel<true, false, false>, a);
  return cudaLaunchKernelEx(&cfg, hot::gsw_tile_kernel<false, true, false>, a);
}

cudaError_t launch_persistent(cudaLaunchConfig_t cfg, const hot::TilePersistArgs &p) {
  cfg.dynamicSmemBytes = hot::tile_smem_bytes(p.step[0].s.M, p.step[0].team, p.step[0].pairs);
  return cudaLaunchKernelEx(&cfg, hot::gsw_tile_persistent_kernel, p);
}

}  // namespace hot_tile

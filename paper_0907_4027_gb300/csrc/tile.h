// tile.h -- host interface (internal to the library) of the register-tiled kernels
// (tile_kernels.cuh): tile.cu instantiates them, hot.cu drives them.
#pragma once
#include <cuda_runtime.h>

#include "tile_kernels.cuh"

namespace hot_tile {

// Blocks per SM that the step and the persistent kernel both keep resident (0: a block does not fit).
cudaError_t occupancy(int M, int team, int pairs, int *per_sm);

// One launch with the grid, block, stream and attributes of cfg (its dynamic shared memory is set
// here): the GSW step (back, fwd), the field of given phases (fwd), a superposition (back) or the
// adjoint (back, adj); and the persistent form.
cudaError_t launch(bool back, bool fwd, bool adj, cudaLaunchConfig_t cfg, const hot::TileArgs &a);
cudaError_t launch_persistent(cudaLaunchConfig_t cfg, const hot::TilePersistArgs &p);

}  // namespace hot_tile

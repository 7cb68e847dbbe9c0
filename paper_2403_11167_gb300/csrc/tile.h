// tile.h -- host side of the tile kernel (step_tile.cuh): its grid and its launch.
#pragma once
#include <cuda_runtime.h>

#include "lbm_kernels.cuh"
#include "step_tile.cuh"

namespace lbmk {

// Columns of a tile: nx in equal parts of at most a warp's columns, even in FP32.
inline int tile_columns(int nx, int cols, int per) {
    const int gx = (nx + cols - 1) / cols;
    return ((nx + gx - 1) / gx + per - 1) / per * per;
}
template <typename real>
inline int tile_columns(int model, int nx) {
    return model == 0   ? tile_columns(nx, Tile<real, 0>::kCols, Tile<real, 0>::kPer)
           : model == 1 ? tile_columns(nx, Tile<real, 1>::kCols, Tile<real, 1>::kPer)
                        : tile_columns(nx, Tile<real, 2>::kCols, Tile<real, 2>::kPer);
}

// One step of the tile kernel.  model: 0 pseudopotential, 1 free energy, 2 full free energy.  walls and drive (T.driven) exclude each other.
template <typename real>
cudaError_t launch_tile(int model, bool walls, const real* fin, real* fout, const StepParams<real>& P,
                        const TileArgs<real>& T, cudaStream_t s);

}  // namespace lbmk

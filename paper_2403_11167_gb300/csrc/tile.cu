// tile.cu -- instantiations and launches of the tile kernel.
#include "tile.h"

#include <algorithm>

namespace lbmk {
namespace {

template <typename real, int MODEL, bool WALLS, bool DRIVE>
cudaError_t launch(const real* fin, real* fout, const StepParams<real>& P, const TileArgs<real>& T, cudaStream_t s) {
    const int rows = T.rows, gy = WALLS && T.band > 0 ? 2 : (P.ny + rows - 1) / rows, gz = (gy + 65534) / 65535;
    const dim3 grid((P.nx + T.wb - 1) / T.wb, (gy + gz - 1) / gz, gz);
    using L = Tile<real, MODEL>;
    const int threads = 32 * (T.share ? L::LV + std::max(2 * rows, rows + L::LV) : rows + 2 * L::LV);
    constexpr bool f32 = std::is_same<real, float>::value;
    if (T.share)
        tile_step<real, MODEL, WALLS, DRIVE, false, false, L::kShared != 0><<<grid, threads, 0, s>>>(fin, fout, P, T);
    else if (!f32 || P.nx % 2 != 0)
        tile_step<real, MODEL, WALLS, DRIVE, false, false, false><<<grid, threads, 0, s>>>(fin, fout, P, T);
    else if (!near_buffer(P.pitch))
        tile_step<real, MODEL, WALLS, DRIVE, f32, false, false><<<grid, threads, 0, s>>>(fin, fout, P, T);
    else
        tile_step<real, MODEL, WALLS, DRIVE, f32, f32, false><<<grid, threads, 0, s>>>(fin, fout, P, T);
    return cudaGetLastError();
}

template <typename real, int MODEL>
cudaError_t launch_model(bool walls, const real* fin, real* fout, const StepParams<real>& P, const TileArgs<real>& T,
                         cudaStream_t s) {
    if (walls) return launch<real, MODEL, true, false>(fin, fout, P, T, s);
    if (T.driven) return launch<real, MODEL, false, true>(fin, fout, P, T, s);
    return launch<real, MODEL, false, false>(fin, fout, P, T, s);
}

}  // namespace

template <typename real>
cudaError_t launch_tile(int model, bool walls, const real* fin, real* fout, const StepParams<real>& P,
                        const TileArgs<real>& T, cudaStream_t s) {
    if (model == 0) return launch_model<real, 0>(walls, fin, fout, P, T, s);
    if (model == 1) return launch_model<real, 1>(walls, fin, fout, P, T, s);
    return launch_model<real, 2>(walls, fin, fout, P, T, s);
}
template cudaError_t launch_tile<float>(int, bool, const float*, float*, const StepParams<float>&,
                                        const TileArgs<float>&, cudaStream_t);
template cudaError_t launch_tile<double>(int, bool, const double*, double*, const StepParams<double>&,
                                         const TileArgs<double>&, cudaStream_t);

}  // namespace lbmk

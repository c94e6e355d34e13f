// Several 2D steps per launch: density form (order 2).
#include "step2d_tile_kernels.cuh"

namespace wave {

cudaError_t launch_tile2d_density(const Tile2DArgs& a, cudaStream_t s) {
  if (!a.acc) return launch_tile(tile2d_tmem_kernel<1, true, 1, 0>, 4, a, s, 32);
  if (a.nfields == 2)
    return a.comp ? launch_tile(tile2d_tmem_kernel<1, true, 2, 2>, 4, a, s, 32)
                  : launch_tile(tile2d_tmem_kernel<1, true, 2, 1>, 4, a, s, 32);
  return a.comp ? launch_tile(tile2d_tmem_kernel<1, true, 1, 2>, 4, a, s, 32)
                : launch_tile(tile2d_tmem_kernel<1, true, 1, 1>, 4, a, s, 32);
}

}  // namespace wave

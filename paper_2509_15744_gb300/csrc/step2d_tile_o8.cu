// Several 2D steps per launch: order 8.
#include "step2d_tile_kernels.cuh"

namespace wave {

cudaError_t launch_tile2d_o8(const Tile2DArgs& a, cudaStream_t s) { return launch_vel_r<4>(a, s); }

}  // namespace wave

// Several 2D steps per launch: order 6.
#include "step2d_tile_kernels.cuh"

namespace wave {

cudaError_t launch_tile2d_o6(const Tile2DArgs& a, cudaStream_t s) { return launch_vel_r<3>(a, s); }

}  // namespace wave

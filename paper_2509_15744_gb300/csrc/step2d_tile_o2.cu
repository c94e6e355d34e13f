// Several 2D steps per launch: order 2.
#include "step2d_tile_kernels.cuh"

namespace wave {

cudaError_t launch_tile2d_o2(const Tile2DArgs& a, cudaStream_t s) { return launch_vel_r<1>(a, s); }

}  // namespace wave

#include "fh_launch_warp.cuh"

int fh::launch_compress_warp_f32_random(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  return launch_compress_warp<kF32, 2>(pl, a, stream);
}

#include "fh_launch_warp.cuh"

int fh::launch_compress_warp_f32_plain(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  return launch_compress_warp<kF32, 0>(pl, a, stream);
}

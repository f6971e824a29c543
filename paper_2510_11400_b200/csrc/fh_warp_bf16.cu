#include "fh_launch_warp.cuh"

int fh::launch_compress_warp_bf16(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  return launch_compress_warp<kBF16, 1>(pl, a, stream);
}

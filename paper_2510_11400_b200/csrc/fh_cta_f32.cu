#include "fh_launch_cta.cuh"

int fh::launch_compress_cta_f32(const Plan& pl, const Variant& v, const CompressArgs& a, cudaStream_t stream) {
  return launch_compress_cta<kF32>(pl, v, a, stream);
}

#include "fh_launch_cta.cuh"

int fh::launch_compress_cta_bf16(const Plan& pl, const Variant& v, const CompressArgs& a, cudaStream_t stream) {
  return launch_compress_cta<kBF16>(pl, v, a, stream);
}

#include "fh_channel.cuh"
#include "fh_compress.cuh"
#include "fh_launch.cuh"

namespace fh {
namespace {

template <int DT, int BITS>
int launch_generic_t(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  int grid = 0;
  int rc = grid_for(compress_generic<DT, BITS>, pl.sm_total, pl.ntiles, &grid);
  if (rc != FH_OK) return rc;
  return launch_dependent(compress_generic<DT, BITS>, grid, kThreads, pl.sm_total, stream, pl, a) == cudaSuccess
             ? FH_OK : FH_ERR_CUDA;
}

template <int DT>
int launch_channel_passes_t(const Plan& pl, const ChannelArgs& ca, cudaStream_t stream) {
  const int sms = sm_count();
  if (sms < 1) return FH_ERR_CUDA;
  const uint64_t want = (pl.P + kWarps - 1) / kWarps, most = (uint64_t)sms * 8;
  const int grid = (int)(want < most ? want : most);
  if (cudaMemsetAsync(ca.chan, 0, pl.C * sizeof(ChanStat), stream) != cudaSuccess) return FH_ERR_CUDA;
  channel_pass<DT, 0><<<grid, kThreads, 0, stream>>>(pl, ca);
  channel_pass<DT, 1><<<grid, kThreads, 0, stream>>>(pl, ca);
  channel_pass<DT, 2><<<grid, kThreads, 0, stream>>>(pl, ca);
  if (cudaGetLastError() != cudaSuccess) return FH_ERR_CUDA;
  return FH_OK;
}

}  // namespace

int launch_compress_generic(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  if (pl.dtype == kF32)
    return pl.bits == 2   ? launch_generic_t<kF32, 2>(pl, a, stream)
           : pl.bits == 4 ? launch_generic_t<kF32, 4>(pl, a, stream)
                          : launch_generic_t<kF32, 8>(pl, a, stream);
  return pl.bits == 2   ? launch_generic_t<kBF16, 2>(pl, a, stream)
         : pl.bits == 4 ? launch_generic_t<kBF16, 4>(pl, a, stream)
                        : launch_generic_t<kBF16, 8>(pl, a, stream);
}

int launch_channel_passes(const Plan& pl, const ChannelArgs& ca, cudaStream_t stream) {
  return pl.dtype == kF32 ? launch_channel_passes_t<kF32>(pl, ca, stream) : launch_channel_passes_t<kBF16>(pl, ca, stream);
}

}  // namespace fh

#include "fh_channel.cuh"
#include "fh_compress.cuh"
#include "fh_launch.cuh"

namespace fh {
namespace {

template <int DT, int BITS, bool ROUND>
int launch_generic_t(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  int grid = 0;
  int rc = grid_for(compress_generic<DT, BITS, ROUND>, pl.sm_total, pl.ntiles, &grid);
  if (rc != FH_OK) return rc;
  return launch_dependent(compress_generic<DT, BITS, ROUND>, grid, kThreads, pl.sm_total, stream, pl, a) == cudaSuccess
             ? FH_OK : FH_ERR_CUDA;
}

template <int DT, bool ROUND>
int launch_generic_dt(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  return pl.bits == 2   ? launch_generic_t<DT, 2, ROUND>(pl, a, stream)
         : pl.bits == 4 ? launch_generic_t<DT, 4, ROUND>(pl, a, stream)
                        : launch_generic_t<DT, 8, ROUND>(pl, a, stream);
}

template <int DT, int PASS, bool VEC>
int launch_channel_pass(const Plan& pl, const ChannelArgs& ca, cudaStream_t stream) {
  int grid = 0;
  const uint64_t items = pl.P * ((pl.groups + kChanPiece - 1) / kChanPiece), per = kThreads / ca.team, want = (items + per - 1) / per;
  const auto kernel = VEC && ca.team == 32u ? channel_pass_runs<DT, PASS> : channel_pass<DT, PASS, VEC>;
  const int rc = grid_for(kernel, 0, (uint32_t)(want < 0x7FFFFFFFull ? want : 0x7FFFFFFFull), &grid);
  if (rc != FH_OK) return rc;
  return launch_dependent(kernel, grid, kThreads, 0, stream, pl, ca) == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

template <int DT, bool VEC>
int launch_channel_passes_t(const Plan& pl, const ChannelArgs& args, cudaStream_t stream) {
  ChannelArgs ca = args;  // a team takes four groups per lane at once: more lanes than that have nothing to do
  ca.team = 1;
  while (ca.team < 32u && ca.team * 4u < pl.groups) ca.team *= 2u;
  int rc = launch_channel_pass<DT, 0, VEC>(pl, ca, stream);
  if (rc == FH_OK) rc = launch_channel_pass<DT, 1, VEC>(pl, ca, stream);
  if (rc == FH_OK) rc = launch_channel_pass<DT, 2, VEC>(pl, ca, stream);
  return rc;
}

}  // namespace

int launch_compress_generic(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  if (pl.dtype == kF32) return pl.rounding ? launch_generic_dt<kF32, true>(pl, a, stream) : launch_generic_dt<kF32, false>(pl, a, stream);
  return pl.rounding ? launch_generic_dt<kBF16, true>(pl, a, stream) : launch_generic_dt<kBF16, false>(pl, a, stream);
}

int launch_channel_passes(const Plan& pl, const ChannelArgs& ca, cudaStream_t stream) {
  const bool vec = pl.HW % 4 == 0;
  if (pl.dtype == kF32) return vec ? launch_channel_passes_t<kF32, true>(pl, ca, stream) : launch_channel_passes_t<kF32, false>(pl, ca, stream);
  return vec ? launch_channel_passes_t<kBF16, true>(pl, ca, stream) : launch_channel_passes_t<kBF16, false>(pl, ca, stream);
}

}  // namespace fh

// Launches of the warp-team compress kernels for one element type.
#pragma once

#include "fh_compress.cuh"
#include "fh_launch.cuh"

namespace fh {

template <int DT, int SIGMA, int TT, bool FULLVEC>
int launch_warp_t(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  int grid = 0;
  int rc = grid_for(compress_warp<DT, SIGMA, TT, FULLVEC>, pl.sm_total, pl.ntiles, &grid, kWarpKernelThreads);
  if (rc != FH_OK) return rc;
  grid = spread_grid(grid, pl.ntiles);
  return launch_dependent(compress_warp<DT, SIGMA, TT, FULLVEC>, grid, kWarpKernelThreads, pl.sm_total, stream,
                          with_first_request(pl, grid, 1), a) == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

template <int DT, int SIGMA, bool FULLVEC>
int launch_warp_tt(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  switch (pl.team) {
    case 1: return launch_warp_t<DT, SIGMA, 1, FULLVEC>(pl, a, stream);
    case 2: return launch_warp_t<DT, SIGMA, 2, FULLVEC>(pl, a, stream);
    case 4: return launch_warp_t<DT, SIGMA, 4, FULLVEC>(pl, a, stream);
    case 8: return launch_warp_t<DT, SIGMA, 8, FULLVEC>(pl, a, stream);
    case 16: return launch_warp_t<DT, SIGMA, 16, FULLVEC>(pl, a, stream);
    case 32: return launch_warp_t<DT, SIGMA, 32, FULLVEC>(pl, a, stream);
  }
  return FH_ERR_UNSUPPORTED;
}

template <int DT, int SIGMA>
int launch_warp_s(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  const bool fullvec = pl.plane_bytes % 16 == 0 && pl.HW % 4 == 0 && pl.groups == 8u * pl.team;
  return fullvec ? launch_warp_tt<DT, SIGMA, true>(pl, a, stream) : launch_warp_tt<DT, SIGMA, false>(pl, a, stream);
}

template <int DT>
int launch_compress_warp(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  if (pl.mode != FH_SALIENT_AUTO) return launch_warp_s<DT, 0>(pl, a, stream);
  return pl.rounding ? launch_warp_s<DT, 2>(pl, a, stream) : launch_warp_s<DT, 1>(pl, a, stream);
}

}  // namespace fh

// Launches of the warp-team compress kernels for one element type.
#pragma once

#include "fh_compress.cuh"
#include "fh_launch.cuh"

namespace fh {

template <int DT, int SIGMA, int TT, int K, int EDGE>
int launch_warp_t(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  int grid = 0;
  int rc = grid_for(compress_warp<DT, SIGMA, TT, K, EDGE>, pl.sm_total, pl.ntiles, &grid, kWarpKernelThreads);
  if (rc != FH_OK) return rc;
  grid = spread_grid(grid, pl.ntiles);
  Plan q = with_first_request(pl, grid, 1);
  q.nstage = pl.nstage;  // (the ring has all its stages, however many tiles the first request is for)
  return launch_dependent(compress_warp<DT, SIGMA, TT, K, EDGE>, grid, kWarpKernelThreads, pl.sm_total, stream, q, a) == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

// Slots per lane: the team is the smallest that holds the plane, so (teams of two and more) at least four are whole;
// seven with three of them masked (7 x 7, 14 x 14 and 28 x 28 take seven), eight with one, or exactly eight (8 x 8,
// 16 x 16, 32 x 32).
template <int DT, int SIGMA, int TT>
int launch_warp_k(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  if constexpr (TT == 1) {
    if (pl.HW == 16u) return launch_warp_t<DT, SIGMA, 1, 4, 0>(pl, a, stream);
    return pl.groups <= 4u ? launch_warp_t<DT, SIGMA, 1, 4, 4>(pl, a, stream) : launch_warp_t<DT, SIGMA, 1, 8, 4>(pl, a, stream);
  } else {
    if (pl.HW == 32u * TT) return launch_warp_t<DT, SIGMA, TT, 8, 0>(pl, a, stream);
    return pl.groups <= 7u * TT ? launch_warp_t<DT, SIGMA, TT, 7, 3>(pl, a, stream) : launch_warp_t<DT, SIGMA, TT, 8, 1>(pl, a, stream);
  }
}

template <int DT, int SIGMA>
int launch_warp_s(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  switch (pl.team) {
    case 1: return launch_warp_k<DT, SIGMA, 1>(pl, a, stream);
    case 2: return launch_warp_k<DT, SIGMA, 2>(pl, a, stream);
    case 4: return launch_warp_k<DT, SIGMA, 4>(pl, a, stream);
    case 8: return launch_warp_k<DT, SIGMA, 8>(pl, a, stream);
    case 16: return launch_warp_k<DT, SIGMA, 16>(pl, a, stream);
    case 32: return launch_warp_k<DT, SIGMA, 32>(pl, a, stream);
  }
  return FH_ERR_UNSUPPORTED;
}

template <int DT>
int launch_compress_warp(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  if (pl.mode != FH_SALIENT_AUTO) return launch_warp_s<DT, 0>(pl, a, stream);
  return pl.rounding ? launch_warp_s<DT, 2>(pl, a, stream) : launch_warp_s<DT, 1>(pl, a, stream);
}

}  // namespace fh

// Launches of the warp-team compress kernels for one element type.
#pragma once

#include "fh_compress.cuh"
#include "fh_launch.cuh"

namespace fh {

template <int DT, int SIGMA, int TT, int K, int EDGE>
int launch_warp_t(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  // (the first K - EDGE slots are not masked: a smaller plane's team would read past it)
  if (pl.groups < (uint32_t)(TT * (K - EDGE)) || pl.groups > (uint32_t)(TT * K)) return FH_ERR_UNSUPPORTED;
  int grid = 0;
  int rc = grid_for(compress_warp<DT, SIGMA, TT, K, EDGE>, pl.sm_total, pl.ntiles, &grid, kWarpKernelThreads);
  if (rc != FH_OK) return rc;
  grid = spread_grid(grid, pl.ntiles);
  // Outlier-rich planes of tiles that are no longer in a stage are fetched again, into a warp's part of the stages, which has to hold
  // them: four planes of a block each, or one.  Where tiles have been made small for the Huffman stage it does not, but then a CTA gets no
  // more tiles than it has stages, and nothing is fetched.
  const size_t part = (pl.sm_sal / (uint32_t)kWarps) & ~15u, fetched = (pl.nblk == 1u ? 4u : 1u) * A16(pl.plane_bytes + 16);
  if (pl.mode != kModeOff && part < fetched && pl.ntiles > (uint64_t)pl.nstage * (uint32_t)grid) return FH_ERR_UNSUPPORTED;
  Plan q = with_first_request(pl, grid, 1);
  q.nstage = pl.nstage;  // (the ring has all its stages, however many tiles the first request is for)
  return launch_dependent(compress_warp<DT, SIGMA, TT, K, EDGE>, grid, kWarpKernelThreads, pl.sm_total, stream, q, a) == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

// Slots per lane.  The team is the smallest that holds the plane in eight slots, so teams of two and more need five to eight: as
// many as the plane needs, of which all but the last are whole.  (Seven slots, three of them masked, for whatever needs five to
// seven took 112 us for 2,048 x 64 fp32 planes of 24 x 24, five take 100; 28 x 28, seven with one masked: 58.9 -> 55.8 us for
// 1,024 x 64 planes; bf16: 97.8 -> 83.5 and 57.7 -> 54.3.)
template <int DT, int SIGMA, int TT>
int launch_warp_k(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  if constexpr (TT == 1) {
    if (pl.HW == 16u) return launch_warp_t<DT, SIGMA, 1, 4, 0>(pl, a, stream);
    return pl.groups <= 4u ? launch_warp_t<DT, SIGMA, 1, 4, 4>(pl, a, stream) : launch_warp_t<DT, SIGMA, 1, 8, 4>(pl, a, stream);
  } else {
    if (pl.HW == 32u * TT) return launch_warp_t<DT, SIGMA, TT, 8, 0>(pl, a, stream);  // (8 x 8, 16 x 16, 32 x 32)
    switch ((pl.groups + TT - 1u) / TT) {
      case 5: return launch_warp_t<DT, SIGMA, TT, 5, 1>(pl, a, stream);
      case 6: return launch_warp_t<DT, SIGMA, TT, 6, 1>(pl, a, stream);
      case 7: return launch_warp_t<DT, SIGMA, TT, 7, 1>(pl, a, stream);  // (7 x 7, 14 x 14, 28 x 28)
      default: return launch_warp_t<DT, SIGMA, TT, 8, 1>(pl, a, stream);
    }
  }
}

template <int DT, int SIGMA>
int launch_compress_warp(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
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

}  // namespace fh

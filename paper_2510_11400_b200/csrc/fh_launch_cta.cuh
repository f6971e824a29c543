// Launches of the CTA-team compress kernels for one element type.
#pragma once

#include "fh_compress.cuh"
#include "fh_launch.cuh"

namespace fh {

template <bool SIGMA>
int launch_cta_t(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  int grid = 0;
  int rc = grid_for(compress_cta<SIGMA>, pl.sm_total, pl.ntiles, &grid, kSweepThreads);
  if (rc != FH_OK) return rc;
  grid = spread_grid(grid, pl.ntiles);
  return launch_dependent(compress_cta<SIGMA>, grid, kSweepThreads, pl.sm_total, stream, with_first_request(pl, grid, 2), a) == cudaSuccess
             ? FH_OK : FH_ERR_CUDA;
}

template <int DT, int SIGMA, int K, int EDGE, bool PARTS, bool WORDS>
int launch_cta_regs_p(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  int grid = 0;
  int rc = grid_for(compress_cta_regs<DT, SIGMA, K, EDGE, PARTS, WORDS>, pl.sm_total, pl.ntiles, &grid, (int)pl.team);
  if (rc != FH_OK) return rc;
  grid = spread_grid(grid, pl.ntiles);
  return launch_dependent(compress_cta_regs<DT, SIGMA, K, EDGE, PARTS, WORDS>, grid, (int)pl.team, pl.sm_total, stream,
                          with_first_request(pl, grid, 1), a) == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}
template <int DT, int SIGMA, int K, int EDGE, bool WORDS = false>
int launch_cta_regs_t(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  return pl.seg > 1u ? launch_cta_regs_p<DT, SIGMA, K, EDGE, true, WORDS>(pl, a, stream)
                     : launch_cta_regs_p<DT, SIGMA, K, EDGE, false, WORDS>(pl, a, stream);
}

// Slots per lane; as the CTA has as few warps as hold the plane, a warp's share is 225 to 448 groups (8 to 14 slots).
template <int DT, int SIGMA>
int launch_cta_regs(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  const uint32_t nw = pl.team / 32u, slots = ((pl.groups + nw - 1u) / nw + 31u) / 32u;
  const bool whole = pl.HW == nw * 4u * kCtaGroups;  // (112 x 112)
  if constexpr (DT == kBF16) {
    if (nw == 7u || nw == 11u || nw == 12u) {  // (see Held; a warp's share is at least 385 groups)
      if (whole) return launch_cta_regs_t<DT, SIGMA, 14, 0, true>(pl, a, stream);
      if (slots <= 13u) return launch_cta_regs_t<DT, SIGMA, 13, 1, true>(pl, a, stream);
      return launch_cta_regs_t<DT, SIGMA, 14, 1, true>(pl, a, stream);
    }
  }
  if (whole) return launch_cta_regs_t<DT, SIGMA, 14, 0>(pl, a, stream);
  if (slots <= 10u) return launch_cta_regs_t<DT, SIGMA, 10, 3>(pl, a, stream);
  if (slots <= 12u) return launch_cta_regs_t<DT, SIGMA, 12, 2>(pl, a, stream);
  if (slots <= 13u) return launch_cta_regs_t<DT, SIGMA, 13, 1>(pl, a, stream);
  return launch_cta_regs_t<DT, SIGMA, 14, 1>(pl, a, stream);
}

template <int DT>
int launch_compress_cta(const Plan& pl, const Variant& v, const CompressArgs& a, cudaStream_t stream) {
  const bool sigma = pl.mode == FH_SALIENT_AUTO;
  if (!v.regs) {
    if constexpr (DT == kBF16) return sigma ? launch_cta_t<true>(pl, a, stream) : launch_cta_t<false>(pl, a, stream);
    return FH_ERR_UNSUPPORTED;  // (make_plan sends them elsewhere)
  }
  if (!sigma) return launch_cta_regs<DT, 0>(pl, a, stream);
  return pl.rounding ? launch_cta_regs<DT, 2>(pl, a, stream) : launch_cta_regs<DT, 1>(pl, a, stream);
}

}  // namespace fh

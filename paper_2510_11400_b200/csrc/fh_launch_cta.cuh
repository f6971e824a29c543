// Launches of the CTA-team compress kernels for one element type.
#pragma once

#include "fh_compress.cuh"
#include "fh_launch.cuh"

namespace fh {

template <int DT, bool SIGMA, int NT>
int launch_cta_t(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  int grid = 0;
  int rc = grid_for(compress_cta<DT, SIGMA, NT>, pl.sm_total, pl.ntiles, &grid, NT);
  if (rc != FH_OK) return rc;
  grid = spread_grid(grid, pl.ntiles);
  return launch_dependent(compress_cta<DT, SIGMA, NT>, grid, NT, pl.sm_total, stream, with_first_request(pl, grid, 2), a) == cudaSuccess
             ? FH_OK : FH_ERR_CUDA;
}

template <int DT, bool SIGMA, int NT, int G>
int launch_cta_regs_t(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  int grid = 0;
  if (pl.groups == (uint32_t)(NT * G)) {
    int rc = grid_for(compress_cta_regs<DT, SIGMA, NT, G, true>, pl.sm_total, pl.ntiles, &grid, NT);
    if (rc != FH_OK) return rc;
    grid = spread_grid(grid, pl.ntiles);
    return launch_dependent(compress_cta_regs<DT, SIGMA, NT, G, true>, grid, NT, pl.sm_total, stream,
                            with_first_request(pl, grid, 2), a) == cudaSuccess ? FH_OK : FH_ERR_CUDA;
  }
  int rc = grid_for(compress_cta_regs<DT, SIGMA, NT, G, false>, pl.sm_total, pl.ntiles, &grid, NT);
  if (rc != FH_OK) return rc;
  grid = spread_grid(grid, pl.ntiles);
  return launch_dependent(compress_cta_regs<DT, SIGMA, NT, G, false>, grid, NT, pl.sm_total, stream,
                          with_first_request(pl, grid, 2), a) == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

template <int DT, bool SIGMA>
int launch_cta_g(const Plan& pl, const Variant& v, const CompressArgs& a, cudaStream_t stream) {
  if (v.G) {
    switch (pl.team * 16 + v.G) {
      case 128 * 16 + 7: return launch_cta_regs_t<DT, SIGMA, 128, 7>(pl, a, stream);
      case 128 * 16 + 8: return launch_cta_regs_t<DT, SIGMA, 128, 8>(pl, a, stream);
      case 256 * 16 + 7: return launch_cta_regs_t<DT, SIGMA, 256, 7>(pl, a, stream);
      case 256 * 16 + 8: return launch_cta_regs_t<DT, SIGMA, 256, 8>(pl, a, stream);
      case 448 * 16 + 7: return launch_cta_regs_t<DT, SIGMA, 448, 7>(pl, a, stream);
      case 512 * 16 + 8: return launch_cta_regs_t<DT, SIGMA, 512, 8>(pl, a, stream);
    }
    return FH_ERR_UNSUPPORTED;
  }
  switch (pl.team) {
    case 128: return launch_cta_t<DT, SIGMA, 128>(pl, a, stream);
    case 256: return launch_cta_t<DT, SIGMA, 256>(pl, a, stream);
    case 512: return launch_cta_t<DT, SIGMA, 512>(pl, a, stream);
  }
  return FH_ERR_UNSUPPORTED;
}

template <int DT>
int launch_compress_cta(const Plan& pl, const Variant& v, const CompressArgs& a, cudaStream_t stream) {
  return pl.mode == FH_SALIENT_AUTO ? launch_cta_g<DT, true>(pl, v, a, stream) : launch_cta_g<DT, false>(pl, v, a, stream);
}

}  // namespace fh

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
  // (the first K - EDGE slots are not masked: a warp that has fewer groups would read past its run)
  if (pl.groups / (pl.team / 32u) < 32u * (K - EDGE)) return FH_ERR_UNSUPPORTED;
  return pl.seg > 1u ? launch_cta_regs_p<DT, SIGMA, K, EDGE, true, WORDS>(pl, a, stream)
                     : launch_cta_regs_p<DT, SIGMA, K, EDGE, false, WORDS>(pl, a, stream);
}

// Whether the planes of a bf16 tensor are held as words (see Held): CTAs of 7, 11 and 12 warps, by how many planes there are.  A plane
// alone takes longer so, by 0.3 us; it pays where more CTAs have one at once than could otherwise, and where there are so many that it
// makes no difference how full the last ones are.  us a call, 4 bits, 112 x 112, as fp32 / as words: 296 planes 8.0 / 9.4, 444
// 10.2 / 9.8, 480 10.4 / 13.0, 960 15.0 / 18.4, 1,480 20.4 / 20.0, 2,000 25.5 / 24.8, 6,000 61.9 / 57.8; 134 x 134 (11 warps): 148 7.0 / 7.3,
// 296 11.9 / 9.6, 400 12.6 / 13.9, 592 17.1 / 18.1, 740 19.7 / 19.2, 2,000 44.5 / 36.3; 146 x 146 (12): 400 13.4 / 15.3, 740 20.9 / 22.0, 900
// 24.1 / 23.0.  With random rounding they gain wherever there are more of them: 112 x 112, 296 12.0 / 11.9, 592 24.4 / 17.5, 2,000 56.3 / 48.1
// (but 700 26.1 / 28.9).
inline bool word_runs(uint32_t nw, int sigma, uint32_t planes) {
  if (nw != 7u && nw != 11u && nw != 12u) return false;
  const uint32_t sms = (uint32_t)sm_count(), at_once = sms * (20u / nw), as_words = sms * ((sigma == 1 ? 24u : 28u) / nw);
  return planes > at_once && (sigma == 2 || planes <= as_words || planes > 5u * at_once);
}

// Slots per lane; as the CTA has as few warps as hold the plane, a warp's share is 224 to 448 groups (7 to 14 slots).  Shares differ by
// one group at most, so that with `slots` slots in the largest the smallest fills all but the last (224, 320, 384 and 416 groups at
// least: just what the instances below leave unmasked).
template <int DT, int SIGMA>
int launch_cta_regs(const Plan& pl, const CompressArgs& a, cudaStream_t stream) {
  const uint32_t nw = pl.team / 32u, slots = ((pl.groups + nw - 1u) / nw + 31u) / 32u;
  const bool whole = pl.HW == nw * 4u * kCtaGroups;  // (112 x 112)
  if constexpr (DT == kBF16) {
    if (word_runs(nw, SIGMA, pl.ntiles)) {
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

#include "fh_decompress.cuh"
#include "fh_launch.cuh"

#include <algorithm>

namespace fh {
namespace {

template <int DT, bool ALIGNED>
int launch_decompress_t(const Plan& pl, const DecompressArgs& a, cudaStream_t stream) {
  int grid = 0;
  const uint32_t lines = chunk_lines(pl.HW, Chunk<DT>::VE, ALIGNED), chunks = (lines + Chunk<DT>::kLines - 1) / Chunk<DT>::kLines;
  const uint64_t ctas = (pl.P * chunks + kWarps - 1) / kWarps;
  int rc = grid_for(decompress_kernel<DT, ALIGNED>, pl.sm_total, (uint32_t)std::min<uint64_t>(ctas, 0x7FFFFFFFu), &grid);
  if (rc != FH_OK) return rc;
  DecompressArgs b = a;
  b.team_stride = prime_at_most((uint64_t)grid * kWarps);
  b.cta_stride = prime_at_most((uint64_t)grid);
  return launch_dependent(decompress_kernel<DT, ALIGNED>, grid, kThreads, pl.sm_total, stream, pl, b) == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

// Planes of at most 128 groups: tiles of 256 / team planes restored in shared memory, one bulk store per tile.
template <int DT>
int launch_decompress_small(const Plan& pl0, const DecompressArgs& a, cudaStream_t stream) {
  Plan pl = pl0;
  // eight groups to a lane; fewer, and smaller tiles, while there are not enough of them for every SM to have one (the
  // Huffman-coded 8 x 512 planes of 7 x 7: 32 tiles, 42.6 us; half the size for all tensors: 32,768 planes 9.2 -> 10.5 us)
  pl.team = team_of_groups(pl.groups);
  while (pl.team < 32u && pl.P * pl.team < (uint64_t)sm_count() * kThreads) pl.team *= 2u;
  pl.ppt = kThreads / pl.team;
  if (pl.ppt > pl.P) pl.ppt = (uint32_t)pl.P;
  pl.stage_bytes = (uint32_t)((pl.ppt * pl.plane_bytes + 127) & ~(uint64_t)127);
  pl.ntiles = (uint32_t)((pl.P + pl.ppt - 1) / pl.ppt);
  // two tile buffers (where the second is, the warps' Huffman tables have room too), then per warp: the block-wise path's
  // scratch (planes of this kernel have so few blocks that a warp restores them) with room behind it for a payload, or for
  // four of one-block planes.  (With tables of their own, 24 KB, one CTA fewer fits an SM: 233,569 planes of 8 x 8, fp32, took
  // 33.3 us, now 24.1.)
  pl.sm_sal = pl.stage_bytes + std::max(pl.stage_bytes, (uint32_t)A16(kWarps * sizeof(HufDecode)));
  pl.sal_stride -= pl.pay_bytes + (uint32_t)A16(sizeof(HufDecode));
  pl.pay_bytes = (pl.nblk == 1u ? 4u : 1u) * ((uint32_t)A16(pl.plane_bytes) + 16u);
  pl.sal_stride = (uint32_t)A16(pl.sal_stride + pl.pay_bytes);
  pl.sm_total = pl.sm_sal + (uint32_t)kWarps * pl.sal_stride;
  if (pl.sm_total > kSmemLimit) return FH_ERR_UNSUPPORTED;
  // Tensors with room for all their tiles at once: no more CTAs to an SM than an even spread puts there (more of them pile up
  // on some SMs, as the kernel before still holds most of the others when they are placed), so room beyond that is asked for
  // as shared memory.  256 tiles of 7 x 7, fp32: three to an SM 7.8 us, two 7.0.
  const uint32_t even = (pl.ntiles + (uint32_t)sm_count() - 1u) / (uint32_t)std::max(sm_count(), 1);
  if (even < 4u) pl.sm_total = std::max(pl.sm_total, (kSmemPerSm / (even + 1u)) & ~15u);
  int grid = 0;
  int rc = grid_for(decompress_small<DT>, pl.sm_total, pl.ntiles, &grid);
  if (rc != FH_OK) return rc;
  if (launch_dependent(decompress_small<DT>, grid, kThreads, pl.sm_total, stream, pl, a) != cudaSuccess)
    return FH_ERR_CUDA;
  return FH_OK;
}

// (see decompress_large, where both sides of the line are measured)
constexpr uint64_t kLargeBytes = 128ull << 20;
int launch_decompress_large(const Plan& pl, const DecompressArgs& a, cudaStream_t stream) {
  int grid = 0;
  const uint64_t ctas = (pl.P * ((pl.HW + 3 + 1023) / 1024) + kWarps - 1) / kWarps;
  int rc = grid_for(decompress_large, pl.sm_total, (uint32_t)std::min<uint64_t>(ctas, 0x7FFFFFFFu), &grid);
  if (rc != FH_OK) return rc;
  DecompressArgs b = a;
  b.team_stride = prime_at_most((uint64_t)grid * kWarps);
  b.cta_stride = prime_at_most((uint64_t)grid);
  return launch_dependent(decompress_large, grid, kThreads, pl.sm_total, stream, pl, b) == cudaSuccess ? FH_OK : FH_ERR_CUDA;
}

template <int DT>
int launch_decompress_dt(const Plan& pl, const DecompressArgs& a, cudaStream_t stream) {
  if (pl.groups <= 128 && pl.team == 32u) return launch_decompress_small<DT>(pl, a, stream);
  if constexpr (DT == kF32) {
    if (pl.dense_bytes > kLargeBytes) return launch_decompress_large(pl, a, stream);
  }
  return pl.plane_bytes % 16 == 0 ? launch_decompress_t<DT, true>(pl, a, stream) : launch_decompress_t<DT, false>(pl, a, stream);
}

}  // namespace

int launch_decompress(const Plan& pl, const DecompressArgs& a, cudaStream_t stream) {
  return pl.dtype == kF32 ? launch_decompress_dt<kF32>(pl, a, stream) : launch_decompress_dt<kBF16>(pl, a, stream);
}

}  // namespace fh

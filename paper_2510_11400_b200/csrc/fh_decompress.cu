#include "fh_decompress.cuh"
#include "fh_launch.cuh"

namespace fh {
namespace {

// Largest prime <= n (n >= 2), or 1.
uint64_t prime_at_most(uint64_t n) {
  static std::map<uint64_t, uint64_t> cache;  // guarded by the library's mutex
  auto it = cache.find(n);
  if (it != cache.end()) return it->second;
  for (uint64_t c = n; c >= 2; --c) {
    bool prime = true;
    for (uint64_t f = 2; f * f <= c; ++f)
      if (c % f == 0) {
        prime = false;
        break;
      }
    if (prime) return cache[n] = c;
  }
  return cache[n] = 1;
}

template <int DT, int TT, bool DEFER = false>
int launch_decompress_t(const Plan& pl, const DecompressArgs& a, cudaStream_t stream) {
  if (TT == 32 && !DEFER && pl.nblk >= kDeferBlocks) return launch_decompress_t<DT, TT, TT == 32>(pl, a, stream);
  int grid = 0;
  int rc = grid_for(decompress_kernel<DT, TT, DEFER>, pl.sm_total, pl.ntiles, &grid);
  if (rc != FH_OK) return rc;
  DecompressArgs b = a;
  b.team_stride = prime_at_most((uint64_t)grid * (kThreads / TT));
  if (launch_dependent(decompress_kernel<DT, TT, DEFER>, grid, kThreads, pl.sm_total, stream, pl, b) != cudaSuccess)
    return FH_ERR_CUDA;
  return FH_OK;
}

// Planes of at most 128 groups: tiles of 256 / team planes restored in shared memory, one bulk store per tile.
template <int DT>
int launch_decompress_small(const Plan& pl0, const DecompressArgs& a, cudaStream_t stream) {
  Plan pl = pl0;
  pl.ppt = kThreads / pl.team;
  if (pl.ppt > pl.P) pl.ppt = (uint32_t)pl.P;
  pl.stage_bytes = (uint32_t)((pl.ppt * pl.plane_bytes + 127) & ~(uint64_t)127);
  pl.ntiles = (uint32_t)((pl.P + pl.ppt - 1) / pl.ppt);
  // two tile buffers, then per warp: scratch for a small plane's payload, or the general path's scratch
  const uint32_t pay = (uint32_t)A16(pl.plane_bytes) + 16u;
  if (pl.sal_stride < pay) pl.sal_stride = pay;
  pl.sm_total = 2u * pl.stage_bytes + (uint32_t)kWarps * pl.sal_stride;
  if (pl.sm_total > kSmemLimit) return FH_ERR_UNSUPPORTED;
  int grid = 0;
  int rc = grid_for(decompress_small<DT>, pl.sm_total, pl.ntiles, &grid);
  if (rc != FH_OK) return rc;
  if (launch_dependent(decompress_small<DT>, grid, kThreads, pl.sm_total, stream, pl, a) != cudaSuccess)
    return FH_ERR_CUDA;
  return FH_OK;
}

template <int DT>
int launch_decompress_dt(const Plan& pl, const DecompressArgs& a, cudaStream_t stream) {
  if (pl.groups <= 128 && pl.P <= 0x7FFFFFFFull) return launch_decompress_small<DT>(pl, a, stream);
  switch (pl.team) {
    case 1: return launch_decompress_t<DT, 1>(pl, a, stream);
    case 2: return launch_decompress_t<DT, 2>(pl, a, stream);
    case 4: return launch_decompress_t<DT, 4>(pl, a, stream);
    case 8: return launch_decompress_t<DT, 8>(pl, a, stream);
    case 16: return launch_decompress_t<DT, 16>(pl, a, stream);
    case 32: return launch_decompress_t<DT, 32>(pl, a, stream);
  }
  return FH_ERR_UNSUPPORTED;
}

}  // namespace

int launch_decompress(const Plan& pl, const DecompressArgs& a, cudaStream_t stream) {
  return pl.dtype == kF32 ? launch_decompress_dt<kF32>(pl, a, stream) : launch_decompress_dt<kBF16>(pl, a, stream);
}

}  // namespace fh

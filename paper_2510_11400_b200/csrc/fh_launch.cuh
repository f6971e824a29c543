// Launching: what the host side (fh.cu) and the files that instantiate the kernels share.  The kernels are compiled in
// several translation units, so that they build in parallel.
#pragma once

#include "../../include/fh.h"

#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <tuple>

#include "fh_device.cuh"

namespace fh {

constexpr size_t kSmemLimit = 227 * 1024 - 4096;  // dynamic shared memory a CTA may ask for
constexpr uint32_t kSmemPerSm = 228 * 1024;       // shared memory of an SM

inline size_t A16(size_t x) { return (x + 15) & ~(size_t)15; }

// Lanes of the team that works on a plane of so many groups, eight groups to a lane: a power of two, at most a warp.
inline uint32_t team_of_groups(uint32_t groups) {
  uint32_t t = 1;
  while (t < 32u && t * 8u < groups) t *= 2u;
  return t;
}

// Which kernel a plan runs on.
struct Variant {
  bool fast = false;  // compress_warp / compress_cta (bulk-copy pipeline) instead of compress_generic
  bool cta = false;   // fast: a plane per CTA instead of compress_warp (a plane per team of lanes)
  bool regs = false;  // cta: compress_cta_regs instead of compress_cta
};

// SMs of the current device (0: none).
int sm_count();

// Largest prime <= n (n >= 2), or 1.  The caller holds the library's mutex.
uint64_t prime_at_most(uint64_t n);

// All of these enqueue on `stream` and return an fh_status; the caller holds the library's mutex.
// (Warp-team kernels: with the plane-wise three-sigma rule, without it, and with it and random rounding.)
int launch_compress_warp_f32(const Plan& pl, const CompressArgs& a, cudaStream_t stream);
int launch_compress_warp_f32_plain(const Plan& pl, const CompressArgs& a, cudaStream_t stream);
int launch_compress_warp_f32_random(const Plan& pl, const CompressArgs& a, cudaStream_t stream);
int launch_compress_warp_bf16(const Plan& pl, const CompressArgs& a, cudaStream_t stream);
int launch_compress_warp_bf16_plain(const Plan& pl, const CompressArgs& a, cudaStream_t stream);
int launch_compress_warp_bf16_random(const Plan& pl, const CompressArgs& a, cudaStream_t stream);
int launch_compress_cta_f32(const Plan& pl, const Variant& v, const CompressArgs& a, cudaStream_t stream);
int launch_compress_cta_bf16(const Plan& pl, const Variant& v, const CompressArgs& a, cudaStream_t stream);
int launch_compress_generic(const Plan& pl, const CompressArgs& a, cudaStream_t stream);
int launch_channel_passes(const Plan& pl, const ChannelArgs& ca, cudaStream_t stream);
int launch_decompress(const Plan& pl, const DecompressArgs& a, cudaStream_t stream);

template <typename K>
int grid_for(K kernel, size_t smem, uint32_t ntiles, int* grid, int threads = fh::kThreads) {
  static std::map<std::tuple<int, const void*, size_t>, int> cache;  // guarded by the library's mutex; per device: the attribute is
  int dev = 0;                                                        // set once for every device that runs the kernel
  if (cudaGetDevice(&dev) != cudaSuccess) return FH_ERR_CUDA;
  const auto key = std::make_tuple(dev, (const void*)kernel, (smem << 12) | (size_t)threads);
  auto it = cache.find(key);
  int per_sm;
  if (it == cache.end()) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit) != cudaSuccess)
      return FH_ERR_CUDA;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess)
      return FH_ERR_CUDA;
    if (per_sm < 1) return FH_ERR_UNSUPPORTED;
    cache[key] = per_sm;
  } else {
    per_sm = it->second;
  }
  const int sms = sm_count();
  if (sms < 1) return FH_ERR_CUDA;
  const uint64_t g = (uint64_t)per_sm * sms;
  *grid = (int)(ntiles < g ? ntiles : g);
  return FH_OK;
}

// Grid of a compress kernel that hands out tiles in order: when every CTA gets several, a prime number of CTAs.  Equally
// fast CTAs then take tiles c, c + grid, ..., and a periodic pattern of outlier-rich planes -- every eighth channel, say --
// spreads over all of them instead of landing on the few whose index shares a factor with the period (with 296 CTAs and
// period 8, 37 CTAs got every such plane of the bf16 112 x 112 tensor).
inline int spread_grid(int grid, uint32_t ntiles) {
  return ntiles >= 2u * (uint32_t)grid && grid >= 2 ? (int)prime_at_most((uint64_t)grid) : grid;
}

// Tiles a CTA requests at once when it starts: all its stages when every CTA of the grid gets that many, fewer
// when the tensor is small, so that the tiles spread over all CTAs before any CTA takes a second one.
inline Plan with_first_request(const Plan& pl, int grid, uint32_t least) {
  Plan q = pl;
  const uint32_t each = pl.ntiles / (uint32_t)(grid > 0 ? grid : 1);
  q.nstage = q.first_req = each < least ? least : (each > pl.nstage ? pl.nstage : each);
  return q;
}

// Launch that may overlap the tail of the previous kernel on the stream (see dep_wait for what keeps the order).
template <typename K, typename A>
cudaError_t launch_dependent(K kernel, int grid, int threads, size_t smem, cudaStream_t stream, const Plan& pl,
                             const A& a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, pl, a);
}

}  // namespace fh

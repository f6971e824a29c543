// Device-side building blocks shared by the compress and decompress kernels (sm_100a).
//
// Terminology: a "plane" is one (n, c) feature map of H x W elements; a "group" is four consecutive
// elements of a plane; a "tile" is a run of consecutive planes that one CTA stages in shared memory;
// a "team" is the set of threads that works on one plane: a power-of-two slice of a warp for small
// planes, the whole CTA for large ones.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace fh {

constexpr int kThreads = 256;             // CTA size, but for the CTA-team kernels' and the warp-team kernel's producer warp
constexpr int kWarps = kThreads / 32;
constexpr int kMaxWarps = 20;            // largest CTA of any kernel: 640 threads
constexpr int kCtaMaxWarps = 20;         // CTA-team kernel, register variant: warps of a CTA at most ...
constexpr int kCtaGroups = 14 * 32;      // ... and groups of a warp (112 x 112: seven warps exactly)
constexpr uint32_t kMagic = 0x31434846u;  // "FHC1"
constexpr uint32_t kClsNormal = 0, kClsSalient = 1, kClsRaw = 2;
constexpr int kModeAuto = 0, kModeOff = 1, kModeAll = 2, kModeChannel = 3, kModeTensor = 4;
constexpr int kF32 = 0, kBF16 = 1;
constexpr int kMaxStages = 4;
constexpr float kMagicF = 12582912.0f;    // 1.5 * 2^23: fma(v, c, kMagicF) leaves rne(v*c) in the mantissa
constexpr uint32_t kMagicBits = 0x4B400000u;

// Device-side error codes (positive, ordered by priority; status_word() maps them to fh_status).
constexpr uint32_t kErrNone = 0, kErrNonfinite = 1, kErrCapacity = 2, kErrCorrupt = 3, kErrTimeout = 4;

// Everything a kernel needs to know about the tensor, the parameters and the tiling.
struct Plan {
  int32_t dtype, esize, H, W;
  uint32_t N, C;
  uint32_t HW;
  uint32_t groups;       // ceil(HW / 4)
  uint64_t P;            // planes
  uint64_t plane_bytes;  // HW * esize
  uint64_t dense_bytes;  // P * plane_bytes
  double inv_hw;         // 1 / HW in fp64
  int32_t bits, mode;
  int32_t rounding;      // 0: round half to even; 1: random rounding (Philox draws)
  int32_t entropy;       // 1: Huffman stage on the dense-block codes of outlier-rich planes (container version 2)
  uint64_t seed;
  uint32_t rho_num, rho_den, tau_num, tau_den;
  float eps;
  uint64_t tensor_id;
  uint32_t npay;         // slot size: A16(bytes of a normal payload)
  uint64_t slots_off;    // 64 + 16 P
  uint64_t ovf_off;      // slots_off + P * npay: start of the overflow region
  uint32_t nbx, nby, nblk, nbm;  // 8x8 blocks per row / column / plane, bitmap words
  uint32_t qs, nsr;              // block-wise path: log2 of the blocks side by side in a step of four, (parts of) rows of steps
  uint32_t seg, segb;            // ... parts of a row of steps, block columns of a part
  // tiling
  uint32_t ppt;          // planes per tile
  uint32_t ntiles;
  uint32_t team;         // threads per plane: 1..32 (power of two) or kThreads
  uint32_t nstage;       // fast kernels: tiles in flight per CTA
  uint32_t first_req;    // warp-team kernel: tiles a CTA requests at once when it starts
  uint32_t stage_bytes;  // fast kernels: bytes of one stage buffer (ppt * plane_bytes)
  // shared-memory layout (byte offsets into dynamic shared memory)
  uint32_t sm_tile, sm_out, sm_rec, sm_total;
  // block-wise path (outlier-rich planes): measuring scratch of one unit (a warp, or the whole CTA)
  uint32_t sm_sal;          // byte offset of the first measuring area in dynamic shared memory
  uint32_t sal_stride;      // bytes between the areas of consecutive units
  uint32_t pay_bytes;       // decompress: bytes at the end of an area that hold payloads
};

// Book-keeping scratch, one per stream: a header of counters and three arrays for the plane-ordered
// placement of overflow parts (see "Placement scan" below).  Everything in the header that a call changes
// is returned to zero by the last CTA of its kernel.
struct Scratch {
  unsigned long long ticket[2];  // next tile (low half; high half, CTA-team kernels: CTAs that have started); consecutive
                                 // compress calls on a stream alternate between the two
  unsigned long long exited;     // CTAs that have left the running kernel
  unsigned long long status;     // device error code (atomicMax)
  unsigned long long nsal, nraw; // outlier-rich planes of either kind (see cta_exit)
  unsigned long long reserved;
  unsigned long long queue;      // CTA-team kernels: planes put off, entries claimed (high half, low half)
  unsigned long long done;       // ... CTAs that have finished phase 1 and either work on the queue or have an error to report
};
static_assert(sizeof(Scratch) == 72, "Scratch layout");
constexpr uint32_t kScratchHeadBytes = 256;  // the header, padded

// (uint64)(int64) fh_status of a device error code.
__device__ __forceinline__ unsigned long long status_word(uint32_t code) {
  const long long st = code == kErrNonfinite ? -4 : code == kErrCapacity ? -3 : code == kErrCorrupt ? -5
                       : code == kErrTimeout ? -6 : 0;
  return (unsigned long long)st;
}

// Lines of 32 output vectors (of `ve` elements) that a plane spans; off the 16-byte grid it may begin anywhere in its first.
__host__ __device__ __forceinline__ uint32_t chunk_lines(uint32_t HW, uint32_t ve, bool aligned) {
  return ((HW + (aligned ? 0u : ve - 1u) + ve - 1u) / ve + 31u) / 32u;
}

__device__ __forceinline__ uint32_t a4(uint32_t x) { return (x + 3u) & ~3u; }
__device__ __forceinline__ uint32_t a16(uint32_t x) { return (x + 15u) & ~15u; }
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ uint32_t ld_relaxed32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed32(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// ---- programmatic dependent launch: a kernel launched with the programmatic-serialisation attribute may become resident when
// every CTA of its predecessor on the stream has called dep_trigger() or ended.  What the library's kernels rely on:
//  - None has completed before all earlier ones on the stream have: dep_wait() returns when they have, and in every kernel threads
//    that write pass it.  So whatever passes dep_wait() sees all that the stream's earlier kernels have written.
//  - Compress kernels trigger behind their wait.  So when a kernel behind a compress kernel starts, everything before that compress
//    kernel has completed.  The others trigger first: any number of them may be resident and waiting.
//  - Ahead of its wait a kernel touches global memory in two cases.  A compress kernel's first request for tiles (early_ticket):
//    its ticket counter was returned to zero by the compress call before the last one on the stream, which had completed when the
//    last one let anything start.  Loads of the input and further requests (early_load): the schedule runner's second and later
//    compress kernels, whose inputs were complete before its first one started and are written by none of them; they are whole
//    16-byte pieces, so that all these loads are bulk copies, which go to the L2 cache, where completed kernels' writes are.
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- shared-memory barriers and bulk (TMA) copies -------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Bulk copy global -> shared; src, dst and bytes are multiples of 16.  Completion is signalled on `bar`.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// Bulk copy shared -> global (same alignment rules), tracked by bulk async-groups.
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
// ... until all but the N most recent groups are complete (their writes performed).
template <int N>
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory"); }
// One wait attempt: the hardware may suspend the thread for up to about `kSuspendNs` nanoseconds
// while the phase is incomplete, so that waiting warps do not burn issue slots polling.
constexpr uint32_t kSuspendNs = 2000;
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3; selp.u32 %0, 1, 0, p; }"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendNs)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait that also gives up when *abort becomes non-zero (looked at every eighth attempt: an attempt
// ends early whenever anything arrives at the barrier, so a waiting warp makes many of them).
__device__ __forceinline__ bool mbar_wait_abortable(uint64_t* bar, uint32_t parity, uint32_t limit,
                                                    const volatile uint32_t* abort) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 7u) == 7u && *abort) return false;
  }
  return false;
}
// Bounded wait: false when the phase did not complete within `limit` polls.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t limit) {
  for (uint32_t i = 0; i < limit; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// ---- arithmetic helpers --------------------------------------------------------------------------
// min / max that return NaN when any operand is NaN, so that a NaN anywhere in a plane surfaces in
// its minimum and maximum.
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float min3_nan(float a, float b, float c) {
  float r;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ float bf16_bits_to_f32(uint32_t h) { return __uint_as_float(h << 16); }
// fp32 -> bf16, round to nearest even (the hardware conversion; the values converted here are never NaN).
__device__ __forceinline__ uint32_t f32_to_bf16_bits(float f) {
  uint16_t r;
  asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(r) : "f"(f));
  return r;
}
// Two at once: `lo` lands in the low half of the word.
__device__ __forceinline__ uint32_t f32x2_to_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

template <int DT>
__device__ __forceinline__ float load_elem(const uint8_t* plane, uint32_t i) {
  if (DT == kF32) return reinterpret_cast<const float*>(plane)[i];
  return bf16_bits_to_f32(reinterpret_cast<const uint16_t*>(plane)[i]);
}

// Group g of a plane, elements past HW read as 0.  `vec` says that the plane starts on a 16-byte
// (fp32) / 8-byte (bf16) boundary so that a full group is one load.
template <int DT>
__device__ __forceinline__ void load_group(const uint8_t* plane, uint32_t g, uint32_t HW, bool vec, float v[4]) {
  const uint32_t i0 = g * 4u;
  if (vec && i0 + 3u < HW) {
    if (DT == kF32) {
      const float4 t = reinterpret_cast<const float4*>(plane)[g];
      v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
      const uint2 t = reinterpret_cast<const uint2*>(plane)[g];
      v[0] = __uint_as_float(t.x << 16); v[1] = __uint_as_float(t.x & 0xFFFF0000u);
      v[2] = __uint_as_float(t.y << 16); v[3] = __uint_as_float(t.y & 0xFFFF0000u);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = (i0 + k < HW) ? load_elem<DT>(plane, i0 + k) : 0.0f;
  }
}

// ---- packed fp32 pairs (sm_100: one instruction, two independent IEEE round-to-nearest results) ----
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ void unpack2u(f32x2 v, uint32_t& a, uint32_t& b) { asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Three-sigma rule: integer moment sums of the distances d = x - lo from the smallest element, scaled by
// the exponent e of the range (2^e <= range < 2^(e+1)): a group of four contributes rne(s * 2^(18-e)) and
// rne(q * 2^(16-2e)), both below 2^22.  The rule is applied for -40 <= e <= 60 only (no product can over-
// or underflow there); a constant plane (range 0, exponent field 0) falls outside like any other.
struct SigmaScale {
  float cs, cq;   // 2^(18-e), 2^(16-2e)
  int32_t e;
  bool applies;
};
__device__ __forceinline__ SigmaScale sigma_scale(float range) {
  SigmaScale s;
  s.e = (int)((__float_as_uint(range) >> 23) & 255u) - 127;
  s.applies = s.e >= -40 && s.e <= 60;
  const int32_t e = s.applies ? s.e : 0;
  s.cs = __uint_as_float((uint32_t)(18 - e + 127) << 23);
  s.cq = __uint_as_float((uint32_t)(16 - 2 * e + 127) << 23);
  return s;
}
// Raw mantissa images of the two addends of one group of distances (d0, d1, d2, d3); the caller sums them
// with wrap-around arithmetic and subtracts kMagicBits once per group at the end.  The group's two pairs
// (d0, d1) and (d2, d3) are combined position by position, s = (d0 + d2) + (d1 + d3) and
// q = fma(d2, d2, d0 * d0) + fma(d3, d3, d1 * d1): with packed two-wide instructions that is one add, one
// multiply and one multiply-add on the pairs as they come out of a 16-byte load, then one add of the halves each.
__device__ __forceinline__ void sigma_addends2(f32x2 p, f32x2 q, const SigmaScale& sc, uint32_t& as, uint32_t& aq) {
  float sa, sb, qa, qb;
  unpack2(add2(p, q), sa, sb);                 // d0 + d2, d1 + d3
  unpack2(fma2(q, q, mul2(p, p)), qa, qb);     // fma(d2, d2, d0 * d0), fma(d3, d3, d1 * d1)
  const f32x2 fixed = fma2(pack2(__fadd_rn(sa, sb), __fadd_rn(qa, qb)), pack2(sc.cs, sc.cq), pack2(kMagicF, kMagicF));
  uint32_t is, iq;
  unpack2u(fixed, is, iq);
  as += is;
  aq += iq;
}
__device__ __forceinline__ void sigma_addends4(float d0, float d1, float d2, float d3, const SigmaScale& sc,
                                               uint32_t& as, uint32_t& aq) {
  sigma_addends2(pack2(d0, d1), pack2(d2, d3), sc, as, aq);
}
__device__ __forceinline__ void sigma_addends(const float d[4], const SigmaScale& sc, uint32_t& as, uint32_t& aq) {
  sigma_addends2(pack2(d[0], d[1]), pack2(d[2], d[3]), sc, as, aq);
}
// Thresholds, as distances from lo, from the exact integer sums: m1 +- 3 sigma.
template <typename I>
__device__ __forceinline__ void sigma_thresholds(I Is, I Iq, const SigmaScale& sc, double inv_count, float& dlo,
                                                 float& dhi) {
  const double ps = __hiloint2double((1023 + sc.e - 18) << 20, 0);      // 2^(e-18)
  const double pq = __hiloint2double((1023 + 2 * sc.e - 16) << 20, 0);  // 2^(2e-16)
  const double m1 = __dmul_rn(__dmul_rn((double)Is, ps), inv_count);
  const double m2 = __dmul_rn(__dmul_rn((double)Iq, pq), inv_count);
  double var = __dsub_rn(m2, __dmul_rn(m1, m1));
  if (!(var > 0.0)) var = 0.0;
  const float m_f = __double2float_rn(m1);
  const float sigma_f = __fsqrt_rn(__double2float_rn(var));
  dhi = __fmaf_rn(3.0f, sigma_f, m_f);
  dlo = __fmaf_rn(-3.0f, sigma_f, m_f);
}

// Quantiser parameters of a normal plane.
__device__ __forceinline__ void quant_params(float range, uint32_t L, float& inv, float& scale) {
  inv = __fdiv_rn((float)L, range);
  scale = __fdiv_rn(range, (float)L);
  if (range == 0.0f || !(fabsf(inv) <= 3.402823466e38f)) {
    inv = 0.0f;
    scale = 0.0f;
  }
}
// Code of one element from its distance d = x - lo: rne of the exact product d * inv, as an integer in the
// mantissa.
__device__ __forceinline__ uint32_t quant_code(float d, float inv, uint32_t L) {
  const float r = __fmaf_rn(d, inv, kMagicF);
  return (__float_as_uint(r) - kMagicBits) & L;
}

// ---- random rounding (rounding = 1) ------------------------------------------------------------------
// Philox-4x32 with 10 rounds (Salmon et al., SC'11): counter-based, so a draw is a pure function of the
// key (seed) and the counter (group within the plane, plane, tensor id).
__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1,
                                              uint32_t (&out)[4]) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t h0 = __umulhi(0xD2511F53u, c0), l0 = 0xD2511F53u * c0;
    const uint32_t h1 = __umulhi(0xCD9E8D57u, c2), l1 = 0xCD9E8D57u * c2;
    c0 = h1 ^ c1 ^ k0;
    c1 = l1;
    c2 = h0 ^ c3 ^ k1;
    c3 = l0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  out[0] = c0;
  out[1] = c1;
  out[2] = c2;
  out[3] = c3;
}
// Codes of a group under random rounding, packed: t = fp32 product d * inv of a distance d = x - lo, n = floor(t), and the code
// goes up iff floor(frac(t) * 2^24) + r reaches 2^24, r = word >> 8.  As n * 2^24 is an integer, floor(frac(t) * 2^24) are the low
// 24 bits of floor(t * 2^24) -- a scaling that is exact, and at most 255 * 2^24 -- and the code is the top byte of that plus r,
// which cannot overflow.  t may come out a little above the last code L; such a position carries L whatever the draw.
// One conversion and about four other instructions an element (a conversion takes a scheduler eight cycles, but on another
// pipe than the generator's products, which take it four each).
template <int BITS>
__device__ __forceinline__ uint32_t quant4_random(const float (&d)[4], float inv, const uint32_t (&rnd)[4]) {
  constexpr float L = (float)((1u << BITS) - 1u);
  const f32x2 inv2 = pack2(inv, inv), one2 = pack2(16777216.0f, 16777216.0f);
  float t[4];
  uint32_t u[4];
  unpack2(mul2(pack2(d[0], d[1]), inv2), t[0], t[1]);
  unpack2(mul2(pack2(d[2], d[3]), inv2), t[2], t[3]);
#pragma unroll
  for (int e = 0; e < 4; ++e) t[e] = fminf(t[e], L);
  unpack2(mul2(pack2(t[0], t[1]), one2), t[0], t[1]);
  unpack2(mul2(pack2(t[2], t[3]), one2), t[2], t[3]);
#pragma unroll
  for (int e = 0; e < 4; ++e) u[e] = __float2uint_rz(t[e]) + (rnd[e] >> 8);
  const uint32_t q = __byte_perm(__byte_perm(u[0], u[1], 0x0073u), __byte_perm(u[2], u[3], 0x0073u), 0x5410u);  // a code to a byte
  if (BITS == 8) return q;
  if (BITS == 4) {
    const uint32_t y = q | (q >> 4);
    return (y & 0xFFu) | ((y >> 8) & 0xFF00u);
  }
  return ((q * 0x00041041u) >> 18) & 0xFFu;  // (the partial products' fields do not overlap)
}

// ------------------------------------------------------------------------------------------------
// Teams
// ------------------------------------------------------------------------------------------------
struct Team {
  uint32_t size;   // threads in the team
  uint32_t lane;   // this thread's index inside the team
  uint32_t mask;   // warp member mask of the team (sub-warp teams)
  bool block;      // the team is the whole CTA
  uint32_t nwarps; // warps of a CTA team
  double* red;     // shared scratch for CTA-wide reductions: kMaxWarps * 4 doubles (see red_half)
};

__device__ __forceinline__ Team make_team(uint32_t team_size, double* red) {
  Team t;
  t.size = team_size;
  t.red = red;
  t.nwarps = team_size >> 5;
  if (team_size > 32u) {
    t.block = true;
    t.lane = threadIdx.x;
    t.mask = 0xFFFFFFFFu;
  } else {
    t.block = false;
    t.lane = threadIdx.x & (team_size - 1u);
    const uint32_t wl = threadIdx.x & 31u;
    t.mask = (team_size == 32u) ? 0xFFFFFFFFu : (((1u << team_size) - 1u) << (wl & ~(team_size - 1u)));
  }
  return t;
}
// The whole CTA as a team, also when it is one warp (make_team would take that for a warp among others).
__device__ __forceinline__ Team make_cta_team(uint32_t threads, double* red) {
  Team t;
  t.size = threads;
  t.red = red;
  t.nwarps = threads >> 5;
  t.block = true;
  t.lane = threadIdx.x;
  t.mask = 0xFFFFFFFFu;
  return t;
}
// The warp of this thread as a team (used for the block-wise path of the warp-team kernels).
__device__ __forceinline__ Team make_warp_team(double* red) {
  Team t;
  t.size = 32;
  t.nwarps = 1;
  t.red = red;
  t.block = false;
  t.lane = threadIdx.x & 31u;
  t.mask = 0xFFFFFFFFu;
  return t;
}

__device__ __forceinline__ void team_sync(const Team& t) {
  if (t.block) __syncthreads();
  else __syncwarp(t.mask);
}

// CTA-wide reductions exchange per-warp partials through t.red, which is split in two halves used
// alternately (`rp` counts the reductions of this thread), so that one barrier per reduction
// suffices: a half is rewritten only after the barrier of the reduction in between.
__device__ __forceinline__ double* red_half(const Team& t, uint32_t& rp) {
  double* r = t.red + ((rp++) & 1u) * (kMaxWarps * 2);
  return r;
}

// min / max over the team with NaN propagation (hardware warp reduction for fp32; teams of a few lanes by butterflies:
// a reduction instruction whose member mask differs within the warp is executed mask by mask, and leaves the warp's
// teams running one after the other -- 2,870 instructions for a warp's sixteen 7 x 7 planes).
__device__ __forceinline__ void team_minmax(const Team& t, float& lo, float& hi, uint32_t& rp) {
  if (!t.block && t.size < 32u) {
    for (uint32_t o = t.size >> 1; o > 0; o >>= 1) {
      lo = min_nan(lo, __shfl_xor_sync(t.mask, lo, o));
      hi = max_nan(hi, __shfl_xor_sync(t.mask, hi, o));
    }
    return;
  }
  asm volatile("redux.sync.min.NaN.f32 %0, %0, %1;" : "+f"(lo) : "r"(0xFFFFFFFFu));
  asm volatile("redux.sync.max.NaN.f32 %0, %0, %1;" : "+f"(hi) : "r"(0xFFFFFFFFu));
  if (t.block) {
    float* r = reinterpret_cast<float*>(red_half(t, rp));
    const uint32_t warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31u) == 0) {
      r[warp * 2] = lo;
      r[warp * 2 + 1] = hi;
    }
    __syncthreads();
    // second stage, lane k takes warp k's pair (a CTA has at most 32 warps): two more warp reductions
    // instead of a walk over all pairs by every thread
    const uint32_t k = min(threadIdx.x & 31u, t.nwarps - 1u);
    const float2 pr = reinterpret_cast<const float2*>(r)[k];
    lo = pr.x;
    hi = pr.y;
    asm volatile("redux.sync.min.NaN.f32 %0, %0, %1;" : "+f"(lo) : "r"(0xFFFFFFFFu));
    asm volatile("redux.sync.max.NaN.f32 %0, %0, %1;" : "+f"(hi) : "r"(0xFFFFFFFFu));
  }
}

// Exact 64-bit sum over the warp of one int32 per lane: high and low halves are summed apart (neither sum
// can overflow 32 bits) and put together again.
__device__ __forceinline__ long long warp_sum_s32_wide(int32_t v) {
  int32_t h = v >> 16;
  uint32_t l = (uint32_t)v & 0xFFFFu;
  asm volatile("redux.sync.add.s32 %0, %0, %1;" : "+r"(h) : "r"(0xFFFFFFFFu));
  asm volatile("redux.sync.add.u32 %0, %0, %1;" : "+r"(l) : "r"(0xFFFFFFFFu));
  return (long long)h * 65536ll + (long long)l;
}

// Sum of two int32 per thread over the team, returned as 64-bit integers.  The sums over one warp
// must fit 32 bits (at most 512 groups per warp, see sigma_addends); warps are combined in 64 bits.
__device__ __forceinline__ void team_sum2(const Team& t, int32_t a, int32_t b, long long& A, long long& B,
                                          uint32_t& rp) {
  if (!t.block && t.size < 32u) {
    for (uint32_t o = t.size >> 1; o > 0; o >>= 1) {
      a += __shfl_xor_sync(t.mask, a, o);
      b += __shfl_xor_sync(t.mask, b, o);
    }
    A = a;
    B = b;
    return;
  }
  asm volatile("redux.sync.add.s32 %0, %0, %1;" : "+r"(a) : "r"(0xFFFFFFFFu));
  asm volatile("redux.sync.add.s32 %0, %0, %1;" : "+r"(b) : "r"(0xFFFFFFFFu));
  A = a;
  B = b;
  if (t.block) {
    int2* r = reinterpret_cast<int2*>(red_half(t, rp));
    const uint32_t warp = threadIdx.x >> 5, wl = threadIdx.x & 31u;
    if (wl == 0) r[warp] = make_int2(a, b);
    __syncthreads();
    // second stage: lane k takes warp k's pair, the warp adds them up in 64 bits
    const int2 pr = wl < t.nwarps ? r[wl] : make_int2(0, 0);
    A = warp_sum_s32_wide(pr.x);
    B = warp_sum_s32_wide(pr.y);
  }
}

// The same for per-thread partial sums that may exceed 32 bits once added over a warp (CTA teams on
// very large planes): 64-bit shuffles inside the warp.
__device__ __forceinline__ void team_sum2_wide(const Team& t, long long a, long long b, long long& A, long long& B,
                                               uint32_t& rp) {
  for (uint32_t o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xFFFFFFFFu, a, o);
    b += __shfl_xor_sync(0xFFFFFFFFu, b, o);
  }
  long long* r = reinterpret_cast<long long*>(red_half(t, rp));
  const uint32_t warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31u) == 0) {
    r[warp * 2] = a;
    r[warp * 2 + 1] = b;
  }
  __syncthreads();
  A = 0;
  B = 0;
  for (uint32_t k = 0; k < t.nwarps; ++k) {
    A += r[k * 2];
    B += r[k * 2 + 1];
  }
}

__device__ __forceinline__ uint32_t team_sum_u32(const Team& t, uint32_t v, uint32_t& rp) {
  if (!t.block && t.size < 32u) {
    for (uint32_t o = t.size >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(t.mask, v, o);
    return v;
  }
  asm volatile("redux.sync.add.u32 %0, %0, %1;" : "+r"(v) : "r"(0xFFFFFFFFu));
  if (t.block) {
    uint32_t* r = reinterpret_cast<uint32_t*>(red_half(t, rp));
    const uint32_t warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31u) == 0) r[warp] = v;
    __syncthreads();
    v = (threadIdx.x & 31u) < t.nwarps ? r[threadIdx.x & 31u] : 0u;  // second stage: lane k takes warp k's sum
    asm volatile("redux.sync.add.u32 %0, %0, %1;" : "+r"(v) : "r"(0xFFFFFFFFu));
  }
  return v;
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
  for (uint32_t o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// ------------------------------------------------------------------------------------------------
// Huffman stage on the residual code bytes of an outlier-rich plane's dense blocks (entropy = 1)
// ------------------------------------------------------------------------------------------------
// One code per plane from the plane's own 256-bin histogram; classical merge of the two least nodes, nodes
// ordered by (weight, id), a leaf's id its symbol, a merged node's 256 + its order of creation; canonical
// code values by (length, symbol); every dense block a chunk of its own that starts on a byte boundary, bits
// most significant first.  Section: u8 len(0) | u8 smin | u8 smax | u8 0 | u8 len(smin..smax) (pad 4) |
// u8 bytes of each chunk (pad 4) | chunks (pad 4).  Lengths stay below 25 (a plane has fewer than 2^17 codes).
constexpr uint32_t kHufMaxLen = 24;
constexpr uint32_t kHufLutBits = 10;     // decoder: with 60 symbols about one code in a hundred is longer
constexpr uint32_t kHufStageWords = 48;  // a chunk has at most 64 * 24 / 8 = 192 bytes

// Encoder scratch of one unit (shared memory, 16-byte aligned).
struct HufEncode {
  uint32_t hist[256];                // once it has been read: the nodes' parents (merged nodes), 256 sorted leaves and 256 merged nodes
  uint32_t code[256];                // by symbol: length << 24 | code value; 0: does not occur
  uint32_t used[256 + 4];            // symbols that occur, ascending, weight << 8 | symbol; four sentinels behind them
  uint8_t sorted[256];               // index into `used` of the sorted leaves
  uint32_t cnt[32], first[32];       // symbols of a length, then running rank; a length's first code value
  uint32_t smin, smax, maxlen, nlens;
  union {
    // weights of the sorted leaves and a sentinel, then of the merged nodes in order of creation (kHufNone: not there yet);
    // done with once the code is built
    uint32_t weight[2 * 260];
    uint32_t stage[1][4 * kHufStageWords];  // chunks' bits while a warp assembles four of them; one per warp of the team
  };
};
constexpr uint32_t kHufNone = 0xFFFFFFu, kHufMerged = 260;
// Words set aside for it and for its alignment: a fixed figure, since which planes are too large for the Huffman stage follows
// from it and must not move with the tables.
constexpr uint32_t kHufEncodeWords = 1542;
static_assert(sizeof(HufEncode) / 4 + 3 <= kHufEncodeWords, "the encoder's tables do not fit");

// First code value of length `lane`, from the number `n` of symbols of that length (0 for length 0), for codes that do not
// oversubscribe: the sum over the shorter lengths k of n_k 2^(length - k), by a prefix sum in units of 2^-31.
__device__ __forceinline__ uint32_t huffman_first(uint32_t n) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t sum = lane ? n << (31u - lane) : 0u;
  const uint32_t own = sum;
#pragma unroll
  for (uint32_t o = 1; o < 32u; o <<= 1) {
    const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, sum, o);
    if (lane >= o) sum += up;
  }
  return (sum - own) >> (31u - lane);
}

// A whole warp: code lengths and canonical codes from h->hist.  Symbols are ranked by comparison with all others (a few
// dozen occur); one lane merges the two queues with the heads of both in registers, the next elements already on
// their way from shared memory, without a branch; depths are walks up the tree, a lane per leaf; code values are
// first-of-length plus rank among the length's symbols, over the symbols that occur.
static __device__ __noinline__ void huffman_build(HufEncode* h) {
  const uint32_t lane = threadIdx.x & 31u, full = 0xFFFFFFFFu, lt = (1u << lane) - 1u;
  uint16_t* parent = reinterpret_cast<uint16_t*>(h->hist);
  uint32_t n = 0;
#pragma unroll
  for (uint32_t i = 0; i < 8u; ++i) {
    const uint32_t sym = i * 32u + lane, w = h->hist[sym], m = __ballot_sync(full, w != 0u);
    if (w) h->used[n + __popc(m & lt)] = w << 8 | sym;  // (weights stay below 2^24)
    n += __popc(m);
    h->code[sym] = 0;
  }
  if (lane < 4u) h->used[n + lane] = 0xFFFFFFFFu;
  h->cnt[lane] = 0;
  __syncwarp();
  for (uint32_t i = lane; i < n; i += 32u) {
    const uint32_t k = h->used[i];
    uint32_t rank = 0;
#pragma unroll 2
    for (uint32_t j = 0; j < n; j += 4u) {
      const uint4 u = *reinterpret_cast<const uint4*>(&h->used[j]);
      rank += (u.x < k ? 1u : 0u) + (u.y < k ? 1u : 0u) + (u.z < k ? 1u : 0u) + (u.w < k ? 1u : 0u);
    }
    h->weight[rank] = k >> 8;
    h->sorted[rank] = (uint8_t)i;
  }
  for (uint32_t i = lane; i < n; i += 32u) h->weight[kHufMerged + i] = kHufNone;
  if (lane < 2u) h->weight[n + lane] = kHufNone;
  __syncwarp();
  if (lane == 0 && n > 1u) {
    uint32_t li = 0, mi = 0, a0 = h->weight[0], a1 = h->weight[1], b0 = kHufNone, b1 = kHufNone;
    for (uint32_t mn = 0; mn + 1u < n; ++mn) {
      uint32_t sum = 0;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const bool leaf = a0 <= b0;  // equal weights: the leaf has the smaller id
        sum += leaf ? a0 : b0;
        parent[leaf ? li : 256u + mi] = (uint16_t)mn;
        li += leaf ? 1u : 0u;
        mi += leaf ? 0u : 1u;
        const uint32_t next = h->weight[leaf ? li + 1u : kHufMerged + mi + 1u];
        a0 = leaf ? a1 : a0;
        b0 = leaf ? b0 : b1;
        a1 = leaf ? next : a1;
        b1 = leaf ? b1 : next;
      }
      h->weight[kHufMerged + mn] = sum;
      if (mi == mn) b0 = sum;
      else if (mi + 1u == mn) b1 = sum;
    }
  }
  __syncwarp();
  uint32_t deepest = 0;
  for (uint32_t i = lane; i < n; i += 32u) {
    uint32_t d = 1;
    if (n > 1u)
      for (uint32_t v = parent[i]; v + 2u != n; v = parent[256u + v]) ++d;  // (the root is merged node n - 2)
    d = min(d, 31u);
    h->code[h->used[h->sorted[i]] & 255u] = d << 24;
    atomicAdd(&h->cnt[d], 1u);
    deepest = max(deepest, d);
  }
  asm volatile("redux.sync.max.u32 %0, %0, %1;" : "+r"(deepest) : "r"(full));
  __syncwarp();
  const uint32_t first = huffman_first(h->cnt[lane]);
  __syncwarp();
  h->first[lane] = first;
  h->cnt[lane] = 0;
  __syncwarp();
  for (uint32_t i = 0; i < n; i += 32u) {
    const uint32_t sym = h->used[min(i + lane, n - 1u)] & 255u, len = i + lane < n ? h->code[sym] >> 24 : 0u;
    const uint32_t same = __match_any_sync(full, len), before = h->cnt[len];
    __syncwarp();
    if (len) h->code[sym] = len << 24 | ((h->first[len] + before + __popc(same & lt)) & 0xFFFFFFu);
    if ((same & lt) == 0u) h->cnt[len] = before + __popc(same);
    __syncwarp();
  }
  if (lane == 0) {  // (symbol 0 is not among those whose lengths are stored as a run)
    uint32_t smin = 1, smax = 1;
    const uint32_t least = n && (h->used[0] & 255u) == 0u ? 1u : 0u;
    if (n > least) {
      smin = h->used[least] & 255u;
      smax = h->used[n - 1u] & 255u;
    }
    h->smin = smin;
    h->smax = smax;
    h->maxlen = deepest;
    h->nlens = smax - smin + 1u;
  }
  __syncwarp();
}

// Decoder tables of one unit (shared memory), from the lengths stored in a section.
struct HufDecode {
  uint32_t count[32];   // symbols of every length
  uint32_t limit[32];   // end of a length's codes, left-aligned (2^32, the end of the longest's, as all ones)
  uint32_t base[32];    // index of a length's first symbol in `sorted`, less the length's first code value
  uint16_t lut[1 << kHufLutBits];  // by the next bits: length << 8 | symbol of a code of at most so many bits, 0 otherwise
  uint8_t sorted[256];  // symbols by (length, symbol)
  uint8_t len[256];
  uint32_t maxlen, ok;
};
// A whole warp: tables from t->len; t->ok = 0 unless the lengths form a complete prefix code (or a single code of any length).
static __device__ __noinline__ void huffman_tables(HufDecode* t) {
  const uint32_t lane = threadIdx.x & 31u, full = 0xFFFFFFFFu, lt = (1u << lane) - 1u;
  bool bad = false;
  t->count[lane] = 0;
  __syncwarp();
  uint32_t rank[8];  // of the lane's symbols among those of the same length
#pragma unroll
  for (uint32_t i = 0; i < 8u; ++i) {
    const uint32_t l = t->len[i * 32u + lane];
    bad |= l > kHufMaxLen;
    const uint32_t lc = min(l, 31u), same = __match_any_sync(full, lc), used = t->count[lc];
    rank[i] = used + __popc(same & lt);
    __syncwarp();
    if ((same & lt) == 0u) t->count[lc] = used + __popc(same);
    __syncwarp();
  }
  bad = __any_sync(full, bad);
  const uint32_t n = lane >= 1u && lane <= kHufMaxLen ? t->count[lane] : 0u;
  uint32_t incl = n;
#pragma unroll
  for (uint32_t o = 1; o < 32u; o <<= 1) {
    const uint32_t up = __shfl_up_sync(full, incl, o);
    if (lane >= o) incl += up;
  }
  const uint32_t nsym = __shfl_sync(full, incl, 31);
  const unsigned long long kraft = warp_sum_u64((unsigned long long)n << (32u - min(lane, 32u)));  // in units of 2^-32
  if (nsym == 0u || kraft > (1ull << 32) || (nsym > 1u && kraft != (1ull << 32))) bad = true;
  __syncwarp();
  if (lane == 0) {
    t->count[0] = 0;
    t->ok = bad ? 0u : 1u;
  }
  const uint32_t longest = __ballot_sync(full, n != 0u);
  __syncwarp();
  const uint32_t first = huffman_first(n);
  const uint32_t index = incl - n;
  t->base[lane] = index - first;
  const unsigned long long lim = (unsigned long long)(first + n) << (32u - min(max(lane, 1u), 31u));
  t->limit[lane] = lim > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)lim;
  if (lane == 0) t->maxlen = longest ? 31u - (uint32_t)__clz((int)longest) : 0u;
  if (!bad) {
#pragma unroll
    for (uint32_t i = 0; i < 8u; ++i) {
      const uint32_t l = t->len[i * 32u + lane];
      const uint32_t at = __shfl_sync(full, index, (int)(l & 31u)) + rank[i];
      if (l) t->sorted[at] = (uint8_t)(i * 32u + lane);
    }
  }
  __syncwarp();
}
// The look-up table, by all `n` threads of the team (this is thread `i`), once huffman_tables is through.
__device__ __forceinline__ void huffman_lut(HufDecode* t, uint32_t i, uint32_t n) {
  for (uint32_t bits = i; bits < (1u << kHufLutBits); bits += n) {
    const uint32_t hi = bits << (32 - kHufLutBits);
    uint32_t len = 1;
#pragma unroll
    for (uint32_t l = 1; l < kHufLutBits; ++l) len += hi >= t->limit[l] ? 1u : 0u;  // (limits ascend with the length)
    const uint32_t at = (hi >> (32u - len)) + t->base[len];
    t->lut[bits] = hi < t->limit[len] ? (uint16_t)(len << 8 | t->sorted[at & 255u]) : (uint16_t)0;
  }
}

// ------------------------------------------------------------------------------------------------
// Placement scan
// ------------------------------------------------------------------------------------------------
// The overflow parts of outlier-rich and raw planes lie in plane order, so a plane's place is the sum of
// the overflow sizes of all planes before it.  A tile (a run of consecutive planes, handed out in order by
// a ticket) publishes the total U of its planes' overflow sizes as soon as it has measured them -- before
// it waits for anything -- and a tile with U > 0 then needs the sum over all earlier tiles.  Two levels
// keep that look-back short (sizes in units of 16 bytes):
//   tile[t] = epoch << 32 | U_t          written once per call; an entry of another epoch reads as "not yet"
//   grp[g]  = count << 40 | sum of U     over the tiles of group g = t >> 5 that have published (atomic adds).
//                                        Two sets alternate between consecutive calls on a scratch; a call's last
//                                        CTA returns the set of the call BEFORE it to zero (grp_clear): every add
//                                        of that call was performed when its kernel completed, so no fence is
//                                        needed between a tile's add and the clearing store.
//   gpre[g] = epoch << 32 | sum of U     over all tiles of groups 0..g, published by whoever has worked it out
// Progress: tiles are taken in ticket order by CTAs that are running, and a CTA publishes all its tiles before it waits for
// another's; so nobody who waits holds up a tile.  Every wait is bounded all the same and reports a time-out instead of hanging.
struct Scan {
  unsigned long long* tile;
  unsigned long long* grp;
  unsigned long long* gpre;
  unsigned long long* grp_clear;  // group sums the call's last CTA returns to zero (see above)
  uint32_t clear_groups;          // ... and how many
  uint32_t epoch;      // of this call (never 0)
  uint32_t polls;      // limit of every wait, in polls of about 0.1 us
  uint32_t skip_tile;  // this tile never publishes (fault injection for the time-out test; 0xFFFFFFFF: none)
};

// One thread: tile t has measured its planes.
__device__ __forceinline__ void scan_publish(const Scan& s, uint32_t t, uint32_t U) {
  if (t == s.skip_tile) return;
  st_relaxed(&s.tile[t], ((unsigned long long)s.epoch << 32) | U);
  atomicAdd(&s.grp[t >> 5], (1ull << 40) | (unsigned long long)U);
}

// A whole warp: sum of U over the tiles before t.  False when a wait ran out.
static __device__ __noinline__ bool scan_prefix(const Scan& s, uint32_t t, uint32_t& prefix) {
  const uint32_t lane = threadIdx.x & 31u, full = 0xFFFFFFFFu;
  const uint32_t g = t >> 5, within = t & 31u;
  // tiles of the own group before t, and at the same time earlier groups, the nearest first, 32 at a time, until a group
  // whose prefix somebody has published
  unsigned long long own = 0, gsum = 0;
  bool mine = lane >= within;
  if (g > 0u) {  // usually that prefix is there: one word, where the search below has every waiting warp read 64
    const unsigned long long vp = ld_relaxed(&s.gpre[g - 1u]);
    const unsigned long long vt = mine ? 0ull : ld_relaxed(&s.tile[g * 32u + lane]);
    if (!mine && (uint32_t)(vt >> 32) == s.epoch) {
      own = vt & 0xFFFFFFFFull;
      mine = true;
    }
    // (one vote of all lanes on the whole condition: another CTA may store the word between two lanes' loads of it)
    if (__all_sync(full, mine && (uint32_t)(vp >> 32) == s.epoch)) {
      prefix = (uint32_t)((vp & 0xFFFFFFFFull) + warp_sum_u64(own));
      return true;
    }
  }
  for (uint32_t hi = g;;) {
    const bool act = lane < hi;
    const uint32_t j = act ? hi - 1u - lane : 0u;
    bool have_pre = false, done = !act;
    unsigned long long val = 0;
    uint32_t first = 32;
    bool all = false;
    for (uint32_t k = 0; k < s.polls; ++k) {
      unsigned long long vt = 0, vp = 0, vg = 0;
      if (!mine) vt = ld_relaxed(&s.tile[g * 32u + lane]);
      if (act && !have_pre) vp = ld_relaxed(&s.gpre[j]);
      if (!done) vg = ld_relaxed(&s.grp[j]);
      if (!mine && (uint32_t)(vt >> 32) == s.epoch) {
        own = vt & 0xFFFFFFFFull;
        mine = true;
      }
      if (act && !have_pre && (uint32_t)(vp >> 32) == s.epoch) {
        have_pre = true;
        done = true;
        val = vp & 0xFFFFFFFFull;
      }
      if (!done && (vg >> 40) == 32ull) {  // every group before another one is a whole group of 32 tiles
        done = true;
        val = vg & ((1ull << 40) - 1ull);
      }
      const uint32_t pm = __ballot_sync(full, have_pre);
      first = pm ? (uint32_t)__ffs((int)pm) - 1u : 32u;
      const uint32_t need = first >= 31u ? full : ((2u << first) - 1u);  // lanes 0..first
      const uint32_t dm = __ballot_sync(full, done);
      all = (dm & need) == need && __all_sync(full, mine);
      if (all) break;
      __nanosleep(k < 4u ? 100u : 500u);
    }
    if (!all) return false;
    gsum += warp_sum_u64(lane <= first ? val : 0ull);
    if (first < 32u || hi <= 32u) break;
    hi -= 32u;
  }
  if (g > 0 && lane == 0) st_relaxed(&s.gpre[g - 1u], ((unsigned long long)s.epoch << 32) | (gsum & 0xFFFFFFFFull));
  prefix = (uint32_t)(gsum + warp_sum_u64(own));
  return true;
}

// The same for up to 32 tiles at once by one warp: lane i < n asks for tile t (with t in no particular order) and gets the sum
// before it.  One warp to a CTA asks, and the group sums are read once for all its tiles: with a warp to a tile, 128 x 192 bf16
// planes of 28 x 28 (3,072 tiles, every one with an outlier-rich plane) had 3,100 warps reading the same dozen lines, which held
// up the publications they waited for: 8 to 35 us from the last publication to the last place.
static __device__ __noinline__ bool scan_places(const Scan& s, uint32_t t, uint32_t n, uint32_t& prefix) {
  constexpr uint32_t kAhead = 4;
  const uint32_t lane = threadIdx.x & 31u, full = 0xFFFFFFFFu, g = t >> 5;
  const bool asks = lane < n;
  // tiles of the own groups: the first few tiles' words are on their way while the group prefixes are looked up
  unsigned long long own[kAhead];
#pragma unroll
  for (uint32_t i = 0; i < kAhead; ++i) {
    const uint32_t ti = __shfl_sync(full, t, (int)i);
    own[i] = i < n && lane < (ti & 31u) ? ld_relaxed(&s.tile[(ti & ~31u) + lane]) : 0ull;
  }
  // prefixes of the groups: those that somebody has published, then the lowest of the others by walking back, then forward
  bool have = !asks || g == 0u;
  unsigned long long pre = 0;
  uint32_t polls = 0;
  while (!__all_sync(full, have)) {
    uint32_t low = have ? 0xFFFFFFFFu : g, high = have ? 0u : g;
    asm volatile("redux.sync.min.u32 %0, %0, %1;" : "+r"(low) : "r"(full));
    asm volatile("redux.sync.max.u32 %0, %0, %1;" : "+r"(high) : "r"(full));
    const unsigned long long v = have ? 0ull : ld_relaxed(&s.gpre[g - 1u]);
    unsigned long long sum = 0;
    bool found = true;
    for (uint32_t hi = low;;) {
      const bool act = lane < hi;
      const uint32_t j = act ? hi - 1u - lane : 0u;
      const unsigned long long vp = act ? ld_relaxed(&s.gpre[j]) : 0ull, vg = act ? ld_relaxed(&s.grp[j]) : 0ull;
      const bool known = act && (uint32_t)(vp >> 32) == s.epoch;
      const uint32_t pm = __ballot_sync(full, known), first = pm ? (uint32_t)__ffs((int)pm) - 1u : 32u;
      // (every group before another one is a whole group of 32 tiles)
      found = __all_sync(full, lane > first || !act || known || (vg >> 40) == 32ull);
      if (!found) break;
      sum += warp_sum_u64(lane > first || !act ? 0ull : (known ? vp & 0xFFFFFFFFull : vg & ((1ull << 40) - 1ull)));
      if (first < 32u || hi <= 32u) break;
      hi -= 32u;
    }
    if (!have && (uint32_t)(v >> 32) == s.epoch) {
      have = true;
      pre = v & 0xFFFFFFFFull;
    }
    if (found) {
      // groups low - 1 (whose prefix is `sum`), low, low + 1, ... as far as they are complete and somebody here asks
      const uint32_t j = low + lane - 1u;
      const unsigned long long vg = lane > 0u && j < high ? ld_relaxed(&s.grp[j]) : 0ull;  // (none when one group is asked for)
      const uint32_t not_done = ~__ballot_sync(full, lane == 0u || (vg >> 40) == 32ull);
      const uint32_t upto = not_done ? (uint32_t)__ffs((int)not_done) - 1u : 32u;
      unsigned long long incl = lane == 0u ? sum : (vg & ((1ull << 40) - 1ull));
#pragma unroll
      for (uint32_t o = 1; o < 32u; o <<= 1) {
        const unsigned long long up = __shfl_up_sync(full, incl, o);
        if (lane >= o) incl += up;
      }
      if (lane < upto) st_relaxed(&s.gpre[j], ((unsigned long long)s.epoch << 32) | (incl & 0xFFFFFFFFull));
      const uint32_t at = have ? 0u : g - low;  // (the lane that holds the prefix this one wants)
      const unsigned long long mine = __shfl_sync(full, incl, (int)min(at, 31u));
      if (!have && at < upto) {
        have = true;
        pre = mine;
      }
    } else {
      if (++polls >= s.polls) return false;
      __nanosleep(polls < 4u ? 100u : 500u);
    }
  }
  // the own groups
  for (uint32_t i0 = 0; i0 < n; i0 += kAhead) {
    if (i0) {
#pragma unroll
      for (uint32_t i = 0; i < kAhead; ++i) {
        const uint32_t ti = __shfl_sync(full, t, (int)min(i0 + i, 31u));
        own[i] = i0 + i < n && lane < (ti & 31u) ? ld_relaxed(&s.tile[(ti & ~31u) + lane]) : 0ull;
      }
    }
#pragma unroll
    for (uint32_t i = 0; i < kAhead; ++i) {
      if (i0 + i >= n) break;
      const uint32_t ti = __shfl_sync(full, t, (int)(i0 + i));
      const bool act = lane < (ti & 31u);
      while (!__all_sync(full, !act || (uint32_t)(own[i] >> 32) == s.epoch)) {
        if (++polls >= s.polls) return false;
        __nanosleep(polls < 4u ? 100u : 500u);
        if (act) own[i] = ld_relaxed(&s.tile[(ti & ~31u) + lane]);
      }
      const unsigned long long sum = warp_sum_u64(act ? own[i] & 0xFFFFFFFFull : 0ull);
      if (lane == i0 + i) pre += sum;
    }
  }
  prefix = (uint32_t)pre;
  return true;
}

// ------------------------------------------------------------------------------------------------
// Arguments of the kernels beside the plan
// ------------------------------------------------------------------------------------------------
struct CompressArgs {
  const uint8_t* src;
  uint8_t* dst_base;
  unsigned long long capacity;          // bytes available at dst_base (minus the offset below)
  const unsigned long long* d_off_in;   // optional: byte offset of the container in dst_base
  unsigned long long* d_off_out;        // optional: offset for the next container
  unsigned long long* out2;             // optional: {total bytes, status}
  Scratch* sc;
  Scan scan;                            // placement of overflow parts (unused with salient_mode OFF)
  uint32_t* defer_next;                 // one word per tile, zero between calls: tiles put off (see BlockCtl)
  uint32_t parity;                      // which of the two ticket counters this call uses
  uint32_t early_ticket;                // 1: tiles may be requested before the previous kernel on the stream has completed
  uint32_t early_load;                  // 1: ... and loaded: the input was complete before that kernel started
  // channel- and tensor-wide three-sigma modes: the statistics passes' results per channel (ChanStat, four words each),
  // the words that the call's last CTA returns to zero, and outlier counts per plane
  unsigned long long* chan_stats;
  uint32_t chan_words;
  const uint32_t* plane_nout;
};

struct DecompressArgs {
  const uint8_t* src_base;
  unsigned long long src_bytes;
  const unsigned long long* d_off_in;  // optional: byte offset of the container in src_base
  uint8_t* dst;
  unsigned long long* d_status;        // optional
  Scratch* sc;
  unsigned long long team_stride;      // a prime, at most the number of warps of the grid (see decompress_kernel)
  unsigned long long cta_stride;       // ... of CTAs
};

struct ChanStat {
  unsigned int lo_inv;       // ~key(minimum): atomicMax
  unsigned int hi_key;       // key(maximum): atomicMax
  unsigned long long Is, Iq;  // fixed-point moment sums (two's complement)
  unsigned long long nout;    // three-sigma outliers of the channel
};
static_assert(sizeof(ChanStat) == 32, "ChanStat layout");

struct ChannelArgs {
  const uint8_t* src;
  ChanStat* chan;        // C entries (one in the tensor-wide mode), zero ahead of pass 0
  uint32_t team;         // lanes per plane: a power of two, at most a warp
  uint32_t* plane_nout;  // P entries, zeroed by pass 0, written by pass 2
  double inv_nhw;        // 1 / (N * HW); tensor-wide: 1 / (N * C * HW)
};

}  // namespace fh

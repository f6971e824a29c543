// Block-wise path of an outlier-rich plane, encoder side (Section 4.4.1): pooled non-zero mask, CSR of the sparse
// blocks, residual codes of the dense ones, optional Huffman stage.
//
// A warp takes four 8x8 blocks per step.  Lane l holds one block row, eight consecutive elements in registers: row
// r = l >> 2 of block q = l & 3.  Two of the three Lorenzo neighbours then lie in the lane itself and the upper row's
// differences come from lane l - 4, one shuffle per eight elements' column; a block's sums are three shuffles over the
// lanes of its column of the warp, a plane row's running count is carried in the lanes that own the row.  The blocks of
// a step lie side by side (planes of three block columns and more), in 2 x 2 (two columns) or below one another (one).
// Warps take the plane's block rows ("step rows") in turn, a CTA's warps parts of them (PARTS) where there are fewer rows
// than warps; only their sums -- CSR row lengths, dense blocks, verbatim
// elements, chunk bytes per step row -- go through shared memory, and one pass of scans turns them into places.
// What bounds it: instruction issue (about 25 instructions per element and pass); a 112 x 112 plane measured in
// 13 us and written in 14 us with a warp per block and a lane per two elements, see the figures at the kernels.
#pragma once

#include "fh_device.cuh"

namespace fh {

struct SalientInfo {
  uint32_t nnz_s, n_dense, n_out_d, size;
  uint32_t coded;  // bytes of the Huffman-coded section that replaces the dense blocks' code bytes; 0: plain codes
};

// Where the bytes of a salient / raw payload go: offsets below npay land in the plane's slot, the
// rest in its overflow part.  Offsets and npay are multiples of the access size.
struct SplitOut {
  uint8_t* slot;
  uint8_t* ovf;
  uint32_t npay;
  __device__ __forceinline__ uint8_t* at(uint32_t o) const { return o < npay ? slot + o : ovf + (o - npay); }
  __device__ __forceinline__ void st32(uint32_t o, uint32_t v) const { *reinterpret_cast<uint32_t*>(at(o)) = v; }
  __device__ __forceinline__ void st16(uint32_t o, uint32_t v) const { *reinterpret_cast<uint16_t*>(at(o)) = (uint16_t)v; }
  __device__ __forceinline__ void st8(uint32_t o, uint32_t v) const { *at(o) = (uint8_t)v; }
};

// What the block-wise path needs to know of the plan, in registers: the outlined functions get the plan by address, and
// a field read through it would be read again after every store.
struct Geometry {
  uint32_t H, W, HW, nbx, nby, nblk, nbm, nsr, qs, esize;
  __device__ __forceinline__ explicit Geometry(const Plan& pl)
      : H((uint32_t)pl.H), W((uint32_t)pl.W), HW(pl.HW), nbx(pl.nbx), nby(pl.nby), nblk(pl.nblk), nbm(pl.nbm), nsr(pl.nsr),
        qs(pl.qs), esize((uint32_t)pl.esize) {}
};

// Shared scratch of one measured plane: words of rowp[H * seg + 1] (a row's entries part by part), dense[nsr + 1],
// outl[nsr + 1], bitmap[nbm] and, with the Huffman stage, chunks[nsr + 1] and a HufEncode.
struct SalScratch {
  uint32_t *rowp, *dense, *outl, *bitmap, *chunks;
  HufEncode* huf;
};
__device__ __forceinline__ SalScratch sal_scratch(const Geometry& pl, uint32_t* sal, uint32_t seg) {
  SalScratch s;
  s.rowp = sal;
  s.dense = s.rowp + pl.H * seg + 1u;
  s.outl = s.dense + pl.nsr + 1u;
  s.bitmap = s.outl + pl.nsr + 1u;
  s.chunks = s.bitmap + pl.nbm;
  s.huf = reinterpret_cast<HufEncode*>(sal + (((uint32_t)(s.chunks - sal) + pl.nsr + 1u + 3u) & ~3u));  // (`sal` is 16-byte aligned)
  return s;
}

// Parts of a step row, block columns of a part.  (Fixed where a row is one part: the streaming kernels' sweeps lose 5 % to the
// registers that these take in the outlined functions.)
template <bool PARTS>
struct Split {
  uint32_t seg, segb;
  __device__ __forceinline__ explicit Split(const Plan& pl) : seg(PARTS ? pl.seg : 1u), segb(PARTS ? pl.segb : pl.nbx) {}
};
// The `unit`-th part: its step row, its number within the row, its block columns.
struct StepUnit {
  uint32_t sr, part, bx0, bx1;
};
template <bool PARTS>
__device__ __forceinline__ StepUnit step_unit(const Geometry& g, const Split<PARTS>& sp, uint32_t unit) {
  if (!PARTS) return StepUnit{unit, 0u, 0u, g.nbx};
  StepUnit u;
  u.sr = sp.seg == 1u ? unit : unit / sp.seg;
  u.part = unit - u.sr * sp.seg;
  u.bx0 = u.part * sp.segb;
  u.bx1 = min(g.nbx, u.bx0 + sp.segb);
  return u;
}
// This lane's place in a step.
struct StepLane {
  uint32_t r, q;    // row within the block, block within the step
  uint32_t qm;      // blocks side by side in a step, less one
  uint32_t qrow;    // the block's row of blocks within the step
};
__device__ __forceinline__ StepLane step_lane(const Geometry& pl) {
  StepLane s;
  const uint32_t lane = threadIdx.x & 31u;
  s.r = lane >> 2;
  s.q = lane & 3u;
  s.qm = (1u << pl.qs) - 1u;
  s.qrow = s.q >> pl.qs;
  return s;
}

// Eight elements of row y from column x0 (positions outside the plane read as 0).  `vec`: rows are whole aligned
// groups of four.
template <int DT>
__device__ __forceinline__ void load_seg(const uint8_t* plane, uint32_t W, uint32_t y, uint32_t x0, uint32_t nin, bool vec,
                                         float (&v)[8]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = 0.0f;
  const uint32_t i = y * W + x0;
  if (vec) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (nin > 4u * h) {
        if (DT == kF32) {
          const float4 t = *reinterpret_cast<const float4*>(plane + 4ull * (i + 4u * h));
          v[4 * h] = t.x; v[4 * h + 1] = t.y; v[4 * h + 2] = t.z; v[4 * h + 3] = t.w;
        } else {
          const uint2 t = *reinterpret_cast<const uint2*>(plane + 2ull * (i + 4u * h));
          v[4 * h] = __uint_as_float(t.x << 16); v[4 * h + 1] = __uint_as_float(t.x & 0xFFFF0000u);
          v[4 * h + 2] = __uint_as_float(t.y << 16); v[4 * h + 3] = __uint_as_float(t.y & 0xFFFF0000u);
        }
      }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if ((uint32_t)j < nin) v[j] = load_elem<DT>(plane, i + j);
  }
}
template <int DT>
__device__ __forceinline__ bool seg_vec(const uint8_t* plane, uint32_t W) {
  return (W & 3u) == 0u && ((uint32_t)(uintptr_t)plane & (DT == kF32 ? 15u : 7u)) == 0u;
}
// Elements of the segment that lie inside the plane.
__device__ __forceinline__ uint32_t seg_in(const Geometry& g, bool valid, uint32_t y, uint32_t x0) {
  return valid && y < g.H ? min(8u, g.W - x0) : 0u;
}
__device__ __forceinline__ uint32_t nonzero_mask(const float (&v)[8]) {
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) m |= (v[j] != 0.0f ? 1u : 0u) << j;
  return m;
}
// Sum over the eight rows of the lane's block.
__device__ __forceinline__ uint32_t block_sum(uint32_t v) {
  v += __shfl_xor_sync(0xFFFFFFFFu, v, 4);
  v += __shfl_xor_sync(0xFFFFFFFFu, v, 8);
  return v + __shfl_xor_sync(0xFFFFFFFFu, v, 16);
}
// Inclusive prefix sum over the rows of the lane's block.
__device__ __forceinline__ uint32_t block_prefix(uint32_t v) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (uint32_t o = 4; o < 32u; o <<= 1) {
    const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, v, o);
    if (lane >= o) v += up;
  }
  return v;
}
// From inclusive row prefixes: sum over the step's blocks before this lane's (`before`) and over all four.
__device__ __forceinline__ void across_blocks(uint32_t incl, uint32_t q, uint32_t& before, uint32_t& all) {
  const uint32_t full = 0xFFFFFFFFu;
  const uint32_t t0 = __shfl_sync(full, incl, 28), t1 = __shfl_sync(full, incl, 29), t2 = __shfl_sync(full, incl, 30),
                 t3 = __shfl_sync(full, incl, 31);
  before = (q > 0u ? t0 : 0u) + (q > 1u ? t1 : 0u) + (q > 2u ? t2 : 0u);
  all = t0 + t1 + t2 + t3;
}

// Residual codes of the lane's block row (Eq. 7-9): first-order Lorenzo prediction on the pre-quantised integers
// k = rne(fp32(x / 2 eps)), neighbours outside the block count as 0.  The second difference of k is the residual:
// e[j] = k[j] - k[j-1] in the row, less the same of the row above.  ca, cb: eight code bytes; vm: verbatim elements.
__device__ __forceinline__ void seg_codes(const float (&v)[8], uint32_t nin, float inv2e, uint32_t& ca, uint32_t& cb,
                                          uint32_t& vm) {
  const uint32_t lane = threadIdx.x & 31u;
  // rounding to an integer by adding 1.5 * 2^23, which holds up to 2^22; beyond (rare) by conversion, at an eighth of the
  // issue rate
  float most = 0.0f;
  int32_t kk[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float x = __fmul_rn(v[j], inv2e);
    most = fmaxf(most, fabsf(x));
    kk[j] = (int32_t)(__float_as_uint(__fadd_rn(x, kMagicF)) - kMagicBits);
  }
  const bool far = !(most < 4194304.0f);
  if (__any_sync(0xFFFFFFFFu, far) && far) {
#pragma unroll
    for (int j = 0; j < 8; ++j) kk[j] = max(min(__float2int_rn(__fmul_rn(v[j], inv2e)), 1 << 24), -(1 << 24));
  }
  int32_t left = 0;
  uint32_t w[2] = {0, 0};
  vm = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int32_t k = kk[j];
    const bool big = k == (1 << 24) || k == -(1 << 24);
    const int32_t e = k - left;
    left = k;
    const int32_t up = __shfl_up_sync(0xFFFFFFFFu, e, 4);
    const int32_t d = e - (lane < 4u ? 0 : up);
    const bool verb = big || (uint32_t)(d + 127) > 254u;
    const bool in = (uint32_t)j < nin;
    const uint32_t code = !in ? 128u : (verb ? 0u : (uint32_t)(d + 128));
    w[j >> 2] |= code << (8 * (j & 3));
    vm |= (in && verb ? 1u : 0u) << j;
  }
  ca = w[0];
  cb = w[1];
}

// In-place exclusive prefix sum of arr[0..n) in shared memory by one warp.
__device__ __forceinline__ void warp_excl_scan(uint32_t* arr, uint32_t n) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t run = 0;
  for (uint32_t b = 0; b < n; b += 32u) {
    const uint32_t v = b + lane < n ? arr[b + lane] : 0u;
    uint32_t incl = v;
#pragma unroll
    for (uint32_t o = 1; o < 32u; o <<= 1) {
      const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += up;
    }
    if (b + lane < n) arr[b + lane] = run + incl - v;
    run += __shfl_sync(0xFFFFFFFFu, incl, 31);
  }
}

// Measuring part: block classes, CSR row lengths, sizes.  The team is a whole warp or a whole CTA.  Leaves rowp, dense
// and outl (and chunks) as exclusive prefix sums with the total behind the last entry, the bitmap and the code.
template <int DT, bool PARTS, bool ENTROPY>
__device__ __noinline__ SalientInfo salient_measure_as(const Team t, const Plan& pl, const uint8_t* plane, uint32_t* sal) {
  const Geometry g(pl);
  const Split<PARTS> sp(pl);
  const SalScratch sc = sal_scratch(g, sal, sp.seg);
  const uint32_t H = g.H, W = g.W, nsr = g.nsr, tau_den = pl.tau_den, full = 0xFFFFFFFFu;
  const uint32_t nw = t.block ? t.nwarps : 1u, wid = t.block ? threadIdx.x >> 5 : 0u, lane = threadIdx.x & 31u;
  const float inv2e = __fdiv_rn(1.0f, __fmul_rn(2.0f, pl.eps));
  const StepLane sl = step_lane(g);
  const bool vec = seg_vec<DT>(plane, W);
  const uint32_t least = pl.tau_num * 64u;  // (at most 2^22)
  for (uint32_t i = t.lane; i < g.nbm; i += t.size) sc.bitmap[i] = 0;
  if (ENTROPY)
    for (uint32_t i = t.lane; i < 256u; i += t.size) sc.huf->hist[i] = 0;
  if (t.lane == 0) sc.rowp[H * sp.seg] = sc.dense[nsr] = sc.outl[nsr] = 0;
  team_sync(t);
  for (uint32_t sr = wid; sr < nsr; sr += nw) {
    const StepUnit un = step_unit(g, sp, sr);
    const uint32_t by = un.sr * (4u >> g.qs) + sl.qrow, y = by * 8u + sl.r;
    uint32_t row = 0, n_dense = 0, n_out = 0, n_zero = 0;
    for (uint32_t bx0 = un.bx0; bx0 < un.bx1; bx0 += sl.qm + 1u) {
      const uint32_t bx = bx0 + (sl.q & sl.qm), x0 = bx * 8u;
      const bool valid = by < g.nby && bx < g.nbx;
      const uint32_t nin = seg_in(g, valid, y, x0);
      float v[8];
      load_seg<DT>(plane, W, y, x0, nin, vec, v);
      const uint32_t cnt = __popc(nonzero_mask(v));
      const bool dense = block_sum(cnt) * tau_den >= least && valid;
      const uint32_t dm = __ballot_sync(full, dense) & 15u;  // (row 0 of every block)
      if (dm) {
        uint32_t ca, cb, vm;
        seg_codes(v, nin, inv2e, ca, cb, vm);
        if (dense) {
          n_out += __popc(vm);
          if (ENTROPY) {  // (residuals of 0 are by far the most frequent: counted apart, their bin is not fought over)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint32_t code = ((j < 4 ? ca : cb) >> (8 * (j & 3))) & 255u;
              if (code == 128u) ++n_zero;
              else atomicAdd(&sc.huf->hist[code], 1u);
            }
          }
          if (sl.r == 0) {
            const uint32_t b = by * g.nbx + bx;
            atomicOr(&sc.bitmap[b >> 5], 1u << (b & 31u));
          }
        }
        n_dense += __popc(dm);
      }
      if (!dense) row += cnt;
    }
    if (g.qs > 0) row += __shfl_xor_sync(full, row, 1);
    if (g.qs > 1) row += __shfl_xor_sync(full, row, 2);
    if ((sl.q & sl.qm) == 0u && y < H) sc.rowp[y * sp.seg + un.part] = row;
    asm volatile("redux.sync.add.u32 %0, %0, %1;" : "+r"(n_out) : "r"(full));
    if (ENTROPY) asm volatile("redux.sync.add.u32 %0, %0, %1;" : "+r"(n_zero) : "r"(full));
    if (lane == 0) {
      sc.dense[sr] = n_dense;
      sc.outl[sr] = n_out;
      if (n_zero) atomicAdd(&sc.huf->hist[128], n_zero);
    }
  }
  team_sync(t);
  if (wid == 0) warp_excl_scan(sc.rowp, H * sp.seg + 1u);
  if (wid == min(1u, nw - 1u)) {
    warp_excl_scan(sc.dense, nsr + 1u);
    warp_excl_scan(sc.outl, nsr + 1u);
  }
  team_sync(t);
  SalientInfo info;
  info.n_dense = sc.dense[nsr];
  info.nnz_s = sc.rowp[H * sp.seg];
  info.n_out_d = sc.outl[nsr];
  info.coded = 0;
  if (ENTROPY && info.n_dense) {
    // Huffman stage (Section 4.4.1): the code from the histogram, then the size of every dense block's chunk
    HufEncode* h = sc.huf;
    if (wid == 0) huffman_build(h);
    if (t.lane == 0) sc.chunks[nsr] = 0;
    team_sync(t);
    if (h->maxlen <= kHufMaxLen) {
      for (uint32_t sr = wid; sr < nsr; sr += nw) {
        const StepUnit un = step_unit(g, sp, sr);
        const uint32_t by = un.sr * (4u >> g.qs) + sl.qrow, y = by * 8u + sl.r;
        uint32_t bytes = 0;
        for (uint32_t bx0 = un.bx0; bx0 < un.bx1; bx0 += sl.qm + 1u) {
          const uint32_t bx = bx0 + (sl.q & sl.qm), x0 = bx * 8u, b = by * g.nbx + bx;
          const bool valid = by < g.nby && bx < g.nbx;
          const bool dense = valid && ((sc.bitmap[b >> 5] >> (b & 31u)) & 1u);
          if (!__any_sync(full, dense)) continue;
          const uint32_t nin = seg_in(g, valid, y, x0);
          float v[8];
          load_seg<DT>(plane, W, y, x0, nin, vec, v);
          uint32_t ca, cb, vm, bits = 0;
          seg_codes(v, nin, inv2e, ca, cb, vm);
#pragma unroll
          for (int j = 0; j < 8; ++j) bits += h->code[((j < 4 ? ca : cb) >> (8 * (j & 3))) & 255u] >> 24;
          bits = block_sum(bits);
          if (dense && sl.r == 0) bytes += (bits + 7u) >> 3;
        }
        asm volatile("redux.sync.add.u32 %0, %0, %1;" : "+r"(bytes) : "r"(full));
        if (lane == 0) sc.chunks[sr] = bytes;
      }
      team_sync(t);
      if (wid == 0) warp_excl_scan(sc.chunks, nsr + 1u);
      team_sync(t);
      const uint32_t section = a4(4u + a4(h->nlens) + a4(info.n_dense) + sc.chunks[nsr]);
      if (section < 64u * info.n_dense) info.coded = section;
    }
  }
  const uint32_t e = g.esize;
  info.size = 16u + 4u * g.nbm + 4u * (H + 1u) + a4(2u * info.nnz_s) + a4(e * info.nnz_s) +
              (info.coded ? info.coded : 64u * info.n_dense) + a4(e * info.n_out_d);
  return info;
}
// With the Huffman stage and without: its counts take registers that the others' loop lacks.
template <int DT, bool PARTS>
__device__ __forceinline__ SalientInfo salient_measure(const Team& t, const Plan& pl, const uint8_t* plane, uint32_t* sal) {
  return pl.entropy ? salient_measure_as<DT, PARTS, true>(t, pl, plane, sal) : salient_measure_as<DT, PARTS, false>(t, pl, plane, sal);
}
// The same as one call, for the general-purpose kernel, whose registers two calls in its loop displace (fp32, random rounding,
// statistics per channel, 190 x 513 planes of 4 x 4 without outliers: 54 -> 61 us).
template <int DT, bool PARTS>
__device__ __noinline__ SalientInfo salient_measure_outlined(const Team t, const Plan& pl, const uint8_t* plane, uint32_t* sal) {
  return salient_measure<DT, PARTS>(t, pl, plane, sal);
}

// Writing part; `sal` holds what salient_measure left.  Every lane recomputes the codes of its block rows and stores
// them (and the CSR entries and verbatim values) straight to their places.
template <int DT, bool PARTS>
__device__ __noinline__ void salient_write(const Team t, const Plan& pl, const uint8_t* plane, const SalientInfo info,
                                           uint32_t* sal, const SplitOut out) {
  const Geometry g(pl);
  const Split<PARTS> sp(pl);
  const SalScratch sc = sal_scratch(g, sal, sp.seg);
  const uint32_t H = g.H, W = g.W, nsr = g.nsr, e = g.esize, full = 0xFFFFFFFFu;
  const uint32_t nw = t.block ? t.nwarps : 1u, wid = t.block ? threadIdx.x >> 5 : 0u, lane = threadIdx.x & 31u;
  const uint32_t o_bm = 16u, o_rp = o_bm + 4u * g.nbm, o_col = o_rp + 4u * (H + 1u);
  const uint32_t o_val = o_col + a4(2u * info.nnz_s), o_codes = o_val + a4(e * info.nnz_s);
  const uint32_t o_outl = o_codes + (info.coded ? info.coded : 64u * info.n_dense);
  if (t.lane == 0) {
    out.st32(0, info.nnz_s);
    out.st32(4, info.n_dense);
    out.st32(8, info.n_out_d);
    out.st32(12, info.coded);
    // pads the section writers leave: col (2 bytes), val / verbatim values (bf16: 2 bytes)
    if (info.nnz_s & 1u) out.st16(o_col + 2u * info.nnz_s, 0);
    if (DT == kBF16 && (info.nnz_s & 1u)) out.st16(o_val + 2u * info.nnz_s, 0);
    if (DT == kBF16 && (info.n_out_d & 1u)) out.st16(o_outl + 2u * info.n_out_d, 0);
  }
  // zero padding up to the end of the slot / of the 16-byte padded overflow part
  const uint32_t end = max(out.npay, a16(info.size));
  for (uint32_t o = info.size + 4u * t.lane; o < end; o += 4u * t.size) out.st32(o, 0);
  for (uint32_t w = t.lane; w < g.nbm; w += t.size) out.st32(o_bm + 4u * w, sc.bitmap[w]);
  for (uint32_t y = t.lane; y <= H; y += t.size) out.st32(o_rp + 4u * y, sc.rowp[y * sp.seg]);
  const HufEncode* h = sc.huf;  // (only looked at when info.coded)
  uint32_t o_cb = 0, o_chunks = 0;
  if (info.coded) {  // the section's head: code lengths, then the bytes of every chunk; pads are zero
    const uint32_t nl = h->nlens;
    o_cb = o_codes + 4u + a4(nl);
    o_chunks = o_cb + a4(info.n_dense);
    if (t.lane == 0) {
      out.st8(o_codes, h->code[0] >> 24);
      out.st8(o_codes + 1u, h->smin);
      out.st8(o_codes + 2u, h->smax);
      out.st8(o_codes + 3u, 0);
      for (uint32_t o = o_codes + 4u + nl; o < o_cb; ++o) out.st8(o, 0);
      for (uint32_t o = o_cb + info.n_dense; o < o_chunks; ++o) out.st8(o, 0);
      for (uint32_t o = o_chunks + sc.chunks[nsr]; o < o_codes + info.coded; ++o) out.st8(o, 0);
    }
    for (uint32_t i = t.lane; i < nl; i += t.size) out.st8(o_codes + 4u + i, h->code[h->smin + i] >> 24);
  }
  const float inv2e = __fdiv_rn(1.0f, __fmul_rn(2.0f, pl.eps));
  const StepLane sl = step_lane(g);
  const bool vec = seg_vec<DT>(plane, W);
  for (uint32_t sr = wid; sr < nsr; sr += nw) {
    const StepUnit un = step_unit(g, sp, sr);
    const uint32_t by = un.sr * (4u >> g.qs) + sl.qrow, y = by * 8u + sl.r;
    uint32_t rank0 = sc.dense[sr], outl0 = sc.outl[sr], chunk0 = info.coded ? sc.chunks[sr] : 0u;
    uint32_t csr = y < H ? sc.rowp[y * sp.seg + un.part] : 0u;
    for (uint32_t bx0 = un.bx0; bx0 < un.bx1; bx0 += sl.qm + 1u) {
      const uint32_t bx = bx0 + (sl.q & sl.qm), x0 = bx * 8u, b = by * g.nbx + bx;
      const bool valid = by < g.nby && bx < g.nbx;
      const uint32_t nin = seg_in(g, valid, y, x0);
      float v[8];
      load_seg<DT>(plane, W, y, x0, nin, vec, v);
      const bool dense = valid && ((sc.bitmap[b >> 5] >> (b & 31u)) & 1u);
      const uint32_t dm = __ballot_sync(full, dense) & 15u;
      if (dm) {
        uint32_t ca, cb, vm;
        seg_codes(v, nin, inv2e, ca, cb, vm);
        if (!dense) vm = 0;
        const uint32_t rank = rank0 + __popc(dm & ((1u << sl.q) - 1u));
        rank0 += __popc(dm);
        if (__any_sync(full, vm != 0u)) {  // verbatim values, in raster order within a block
          const uint32_t c = __popc(vm), incl = block_prefix(c);
          uint32_t before, all;
          across_blocks(incl, sl.q, before, all);
          uint32_t o = o_outl + e * (outl0 + before + incl - c);
          outl0 += all;
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if ((vm >> j) & 1u) {
              if (DT == kF32) out.st32(o, __float_as_uint(v[j]));
              else out.st16(o, __float_as_uint(v[j]) >> 16);
              o += e;
            }
        }
        if (!info.coded) {
          if (dense) {
            const uint32_t oc = o_codes + 64u * rank + 8u * sl.r;
            out.st32(oc, ca);
            out.st32(oc + 4u, cb);
          }
        } else {
          // the chunks' bits are assembled in shared memory (a code goes in most significant bit first, the words
          // hold the stream big-endian) and leave byte by byte
          uint32_t* stg = sc.huf->stage[wid];
#pragma unroll
          for (uint32_t i = 0; i < 4u * kHufStageWords / 32u; ++i) stg[i * 32u + lane] = 0;
          __syncwarp();
          uint32_t bits = 0;
#pragma unroll
          for (int j = 0; j < 8; ++j) bits += h->code[((j < 4 ? ca : cb) >> (8 * (j & 3))) & 255u] >> 24;
          const uint32_t incl = block_prefix(bits), total = __shfl_sync(full, incl, 28u + sl.q);
          const uint32_t bytes = dense ? (total + 7u) >> 3 : 0u;
          uint32_t before, all;
          across_blocks(bytes, sl.q, before, all);
          if (dense) {
            uint32_t at = incl - bits;
            uint32_t* sw = stg + sl.q * kHufStageWords;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint32_t hc = h->code[((j < 4 ? ca : cb) >> (8 * (j & 3))) & 255u], len = hc >> 24, cv = hc & 0xFFFFFFu;
              const uint32_t wi = at >> 5;
              const int shift = 32 - (int)(at & 31u) - (int)len;
              if (shift >= 0) {
                atomicOr(&sw[wi], cv << shift);
              } else {
                atomicOr(&sw[wi], cv >> (-shift));
                atomicOr(&sw[wi + 1u], cv << (32 + shift));
              }
              at += len;
            }
          }
          __syncwarp();
          if (dense) {
            const uint32_t* sw = stg + sl.q * kHufStageWords;
            if (sl.r == 0) out.st8(o_cb + rank, bytes);
            for (uint32_t j = sl.r; j < bytes; j += 8u)
              out.st8(o_chunks + chunk0 + before + j, (sw[j >> 2] >> (24u - 8u * (j & 3u))) & 0xFFu);
          }
          chunk0 += all;
          __syncwarp();
        }
      }
      if (info.nnz_s) {  // CSR entries of the sparse blocks
        const uint32_t nz = dense ? 0u : nonzero_mask(v), c = __popc(nz);
        uint32_t incl = c;
        if (g.qs > 0) {
          const uint32_t up = __shfl_up_sync(full, incl, 1);
          if ((sl.q & sl.qm) >= 1u) incl += up;
        }
        if (g.qs > 1) {
          const uint32_t up = __shfl_up_sync(full, incl, 2);
          if (sl.q >= 2u) incl += up;
        }
        uint32_t pos = csr + incl - c;
        csr += __shfl_sync(full, incl, lane | sl.qm);
        if (nz) {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if ((nz >> j) & 1u) {
              out.st16(o_col + 2u * pos, x0 + j);
              if (DT == kF32) out.st32(o_val + 4u * pos, __float_as_uint(v[j]));
              else out.st16(o_val + 2u * pos, __float_as_uint(v[j]) >> 16);
              ++pos;
            }
        }
      }
    }
  }
}

}  // namespace fh

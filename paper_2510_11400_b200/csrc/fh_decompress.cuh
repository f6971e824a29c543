// Decompress kernel: container -> dense tensor, one pass.
//
// Planes are independent and their slots sit at closed-form offsets, so the kernels need no hand-out.  Normal planes
// are the fused unpack-and-dequantise: codes are read straight from the slot (they are 1/16 to 1/4 of the output) and
// leave as 16-byte stores.  Raw planes are copied; outlier-rich planes are restored a lane per dense block (decode_salient),
// small ones four blocks per warp and step (decode_few).  Every read of the container is bounds-checked against src_bytes; a plane whose table entry or
// payload is inconsistent reports FH_ERR_CORRUPT.
#pragma once

#include "fh_blocks.cuh"

namespace fh {

// Reads of a salient / raw payload: offsets below npay come from the plane's slot, the rest from its
// overflow part.
struct SplitIn {
  const uint8_t* slot;
  const uint8_t* ovf;
  uint32_t npay;
  __device__ __forceinline__ const uint8_t* at(uint32_t o) const { return o < npay ? slot + o : ovf + (o - npay); }
  __device__ __forceinline__ uint32_t ld32(uint32_t o) const { return __ldg(reinterpret_cast<const uint32_t*>(at(o))); }
  __device__ __forceinline__ uint32_t ld16(uint32_t o) const { return __ldg(reinterpret_cast<const uint16_t*>(at(o))); }
  __device__ __forceinline__ uint32_t ld8(uint32_t o) const { return __ldg(at(o)); }
};

// A payload copied to shared memory as one piece.
struct FlatIn {
  const uint8_t* p;
  uint32_t npay;  // (kept for the size check: bytes of the payload that came from the slot)
  __device__ __forceinline__ uint32_t ld32(uint32_t o) const { return *reinterpret_cast<const uint32_t*>(p + o); }
  __device__ __forceinline__ uint32_t ld16(uint32_t o) const { return *reinterpret_cast<const uint16_t*>(p + o); }
  __device__ __forceinline__ uint32_t ld8(uint32_t o) const { return p[o]; }
};

// One thread decodes a dense block's chunk of the Huffman-coded section (`nbytes` bytes at payload offset
// `o_chunk`; `end`: bytes of the payload) into the block's 64 code bytes, four to a word.  False when the chunk is
// inconsistent.  The chain of a symbol is a table look-up and a shift; the 64-bit window on the stream is fetched anew
// for every group of symbols that surely fits it (four of at most 16 bits, two otherwise), without a branch, so that
// the lanes' chunks stay in step.
template <typename In>
__device__ __forceinline__ bool huffman_decode_chunk(const In& in, uint32_t o_chunk, uint32_t nbytes, uint32_t end,
                                                     const HufDecode* hd, uint32_t (&codes)[16]) {
  uint32_t pos = o_chunk * 8u;  // in bits from the start of the payload
  bool ok = true;
  const uint32_t longest = hd->maxlen;
  const bool four = longest <= 16u;
  auto symbol = [&](uint32_t& hi, uint32_t& lo) -> uint32_t {
    uint32_t en = hd->lut[hi >> (32 - kHufLutBits)];
    if (en == 0u) {  // a longer code: the first length whose codes, left-aligned, reach beyond the window
      uint32_t l = kHufLutBits + 1;
      while (l < longest && hi >= hd->limit[l]) ++l;
      const uint32_t at = (hi >> (32u - l)) + hd->base[l];
      if (l > longest) ok = false;  // (a lone symbol's code leaves half of the windows without a meaning)
      en = l << 8 | hd->sorted[at & 255u];
    }
    const uint32_t l = en >> 8;
    pos += l;
    hi = __funnelshift_l(lo, hi, l);
    lo <<= l;
    return en & 255u;
  };
  auto window = [&](uint32_t& hi, uint32_t& lo) {
    const uint32_t o = (pos >> 5) << 2;
    const uint32_t w0 = o + 4u <= end ? in.ld32(o) : 0u, w1 = o + 8u <= end ? in.ld32(o + 4u) : 0u, w2 = o + 12u <= end ? in.ld32(o + 8u) : 0u;
    const uint32_t b0 = __byte_perm(w0, 0u, 0x0123), b1 = __byte_perm(w1, 0u, 0x0123), b2 = __byte_perm(w2, 0u, 0x0123);
    hi = __funnelshift_l(b1, b0, pos & 31u);
    lo = __funnelshift_l(b2, b1, pos & 31u);
  };
#pragma unroll 1
  for (uint32_t i = 0; i < 16u; ++i) {
    uint32_t hi, lo;
    window(hi, lo);
    uint32_t word = symbol(hi, lo);
    word |= symbol(hi, lo) << 8;
    if (!four) window(hi, lo);
    word |= symbol(hi, lo) << 16;
    word |= symbol(hi, lo) << 24;
    // (the words move up by one and the new one comes in last: registers need static indexes)
#pragma unroll
    for (int k = 0; k < 15; ++k) codes[k] = codes[k + 1];
    codes[15] = word;
  }
  return ok && pos <= (o_chunk + nbytes) * 8u;
}

template <int DT>
__device__ __forceinline__ void store_elem(uint8_t* plane, uint32_t i, float v) {
  if (DT == kF32) reinterpret_cast<float*>(plane)[i] = v;
  else reinterpret_cast<uint16_t*>(plane)[i] = (uint16_t)f32_to_bf16_bits(v);
}

// x = fma(q, scale, lo); q < 2^23 is turned into a float through its bit pattern.
__device__ __forceinline__ float dequant(uint32_t q, float scale, float lo) {
  const float qf = __fsub_rn(__uint_as_float(0x4B000000u | q), 8388608.0f);
  return __fmaf_rn(qf, scale, lo);
}

// Eight restored values of row y from column x0 on, `nin` of them inside the plane.  `vec`: rows are whole aligned
// groups of four.
template <int DT>
__device__ __forceinline__ void store_seg(uint8_t* out, uint32_t W, uint32_t y, uint32_t x0, uint32_t nin, bool vec,
                                          const float (&v)[8]) {
  const uint32_t i = y * W + x0;
  if (vec) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (nin > 4u * h) {
        if (DT == kF32)
          *reinterpret_cast<float4*>(out + 4ull * (i + 4u * h)) = make_float4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
        else
          *reinterpret_cast<uint2*>(out + 2ull * (i + 4u * h)) =
              make_uint2(f32x2_to_bf16x2(v[4 * h], v[4 * h + 1]), f32x2_to_bf16x2(v[4 * h + 2], v[4 * h + 3]));
      }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if ((uint32_t)j < nin) store_elem<DT>(out, i + j, v[j]);
  }
}

// Zero bytes of a word, as one bit (0x80) each.
__device__ __forceinline__ uint32_t zero_bytes(uint32_t w) { return ~(((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w | 0x7F7F7F7Fu); }

// A dense block by one lane, in raster order: k = pred + residual (Eq. 7-9), x = k * 2 eps; a verbatim element's k
// follows from its stored value.  Row by row, with the differences e[j] = k[j] - k[j-1] of the row above in registers;
// all that does not depend on the left neighbour -- the row's verbatim values and their k -- is worked out for the eight
// columns side by side and without branches (a column without a verbatim value reads the one that comes next), which
// leaves an addition and a selection per element as the serial chain.  `codes`: the block's 64 code bytes; oi: index of
// its first verbatim value (all of them are there, the caller has counted); o_outl, last: where the values are and the
// last one's index.  A warp restores 32 blocks in about 1,200 instructions; a lane per block row, in a wavefront over
// the columns, took 1,000 for four.
template <int DT, typename In>
__device__ __forceinline__ void restore_block(const In& in, uint32_t o_outl, uint32_t last, uint32_t oi, uint32_t (&codes)[16],
                                              float two_eps, float inv2e, uint8_t* out, uint32_t H, uint32_t W, uint32_t y0,
                                              uint32_t x0, bool vec) {
  const uint32_t nin = min(8u, W - x0), rows = min(8u, H - y0);
  int32_t e[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) e[j] = 0;
#pragma unroll 1
  for (uint32_t i = 0; i < rows; ++i) {
    const uint32_t a = codes[0], c = codes[1];
#pragma unroll
    for (int k = 0; k < 14; ++k) codes[k] = codes[k + 2];
    float v[8];
    int32_t kv[8];
    bool is[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t code = __byte_perm(a, c, 0x4440u + j) & 255u;
      e[j] += (int32_t)code - 128;
      is[j] = code == 0u && (uint32_t)j < nin;
      const uint32_t at = min(oi, last);
      v[j] = DT == kF32 ? __uint_as_float(in.ld32(o_outl + 4u * at)) : bf16_bits_to_f32(in.ld16(o_outl + 2u * at));
      oi += is[j] ? 1u : 0u;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) kv[j] = max(min(__float2int_rn(__fmul_rn(v[j], inv2e)), 1 << 24), -(1 << 24));
    int32_t left = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int32_t k = is[j] ? kv[j] : left + e[j];
      v[j] = is[j] ? v[j] : __fmul_rn((float)k, two_eps);
      e[j] = k - left;
      left = k;
    }
    store_seg<DT>(out, W, y0 + i, x0, nin, vec, v);
  }
}

// Zero bytes of a block's codes: its verbatim elements.
__device__ __forceinline__ uint32_t count_verbatim(const uint32_t (&codes)[16]) {
  uint32_t n = 0;
#pragma unroll
  for (int k = 0; k < 16; ++k) n += __popc(zero_bytes(codes[k]));
  return n;
}

// Four dense blocks by one warp: lane 8 q + j has column j of block q.  Within a row, k[j] = k[j-1] + e[j] + residual[j]
// is a scan over the block's eight lanes that starts anew at every verbatim element, so a row is four shuffles and the
// block eight such rows in series; the verbatim values and their k are worked out for all rows beforehand.  About 330
// instructions for four blocks: twice those of a lane per block (restore_block), but a quarter of its latency, which is
// what counts for planes of few blocks (14 x 14, fp32, 67 outlier-rich planes of 16,384: 22.6 -> 13.7 us a call).
//   code_at(i)  the lane's code byte of row i;  dense  the lane's block is one (the others take part with codes of 128)
//   out, y0, x0 where the block's elements go
// `locate` is told the number of verbatim elements of the lane's block (all lanes call it) and says where in the payload the
// first lies, or that the payload does not hold as many: their values are then not read.
template <int DT, typename In, typename CodeAt, typename Locate>
__device__ __forceinline__ void restore_columns(const In& in, CodeAt code_at, Locate locate, bool dense, float two_eps, float inv2e,
                                                uint8_t* out, uint32_t H, uint32_t W, uint32_t y0, uint32_t x0) {
  const uint32_t full = 0xFFFFFFFFu, lane = threadIdx.x & 31u, j = lane & 7u, q = lane >> 3;
  int32_t res[8];
  uint32_t mask[8];  // verbatim elements of row i: this lane's block's byte
  uint32_t any = 0, n = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t code = dense ? code_at(i) : 128u;
    res[i] = (int32_t)code - 128;
    const uint32_t m = __ballot_sync(full, code == 0u);
    mask[i] = (m >> (8u * q)) & 255u;
    any |= m;
    n += __popc(mask[i]);
  }
  float raw[8];
  int32_t kv[8];
  if (any) {
    uint32_t o = 0;
    const bool held = locate(n, o);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t at = o + (DT == kF32 ? 4u : 2u) * __popc(mask[i] & ((1u << j) - 1u));
      raw[i] = 0.0f;
      if (held && ((mask[i] >> j) & 1u)) raw[i] = DT == kF32 ? __uint_as_float(in.ld32(at)) : bf16_bits_to_f32(in.ld16(at));
      o += (DT == kF32 ? 4u : 2u) * __popc(mask[i]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) kv[i] = max(min(__float2int_rn(__fmul_rn(raw[i], inv2e)), 1 << 24), -(1 << 24));
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) raw[i] = 0.0f, kv[i] = 0;
  }
  int32_t e = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t upto = mask[i] & ((2u << j) - 1u);                            // verbatim elements at or before the column
    const uint32_t reach = upto ? j - (31u - (uint32_t)__clz((int)upto)) : j;   // lanes the sum may reach back
    const bool is = (mask[i] >> j) & 1u;
    int32_t k = is ? kv[i] : e + res[i];
#pragma unroll
    for (uint32_t o = 1; o < 8u; o <<= 1) {
      const int32_t t = __shfl_up_sync(full, k, o);
      if (reach >= o) k += t;
    }
    const int32_t left = __shfl_up_sync(full, k, 1);
    e = j == 0u ? k : k - left;
    if (dense && y0 + i < H && x0 + j < W) store_elem<DT>(out, (y0 + i) * W + x0 + j, is ? raw[i] : __fmul_rn((float)k, two_eps));
  }
}

// Outlier-rich plane: the inverse of salient_write.  Dense blocks a lane each, by rank (so that all lanes have one);
// where a block's verbatim values start is a scan over the zero bytes of the codes.  Sparse blocks are
// zeroed first, a lane per block row, and take their values entry by entry, eight lanes to a CSR row.  `scr` is the team's shared scratch, laid out by
// make_plan, `hd` its tables for a Huffman-coded plane (touched only when the container is of version 2); `ovf_avail` the number of readable bytes behind in.ovf; `version` the container's (2: the dense blocks'
// codes may be Huffman-coded, Section 4.4.1 "Decompression involves Huffman decoding").  Returns false in the threads
// that found the payload inconsistent.
template <int DT, typename In>
__device__ __noinline__ bool decode_salient(const Team t, const Plan& pl, const In in, uint64_t ovf_avail, float eps, uint8_t* out,
                                            uint32_t* scr, HufDecode* hd, uint32_t version) {
  const Geometry g(pl);
  const uint32_t H = g.H, W = g.W, nblk = g.nblk, nbx = g.nbx, nbm = g.nbm, e = g.esize, HW = g.HW;
  const uint32_t full = 0xFFFFFFFFu;
  const uint32_t nnz_s = in.ld32(0), n_dense = in.ld32(4), n_out_d = in.ld32(8), coded = in.ld32(12);
  if (nnz_s > HW || n_dense > nblk || n_out_d > HW) return false;
  if (coded && (version != 2u || (coded & 3u) || coded >= 64u * n_dense)) return false;
  const uint64_t size = 16ull + 4ull * nbm + 4ull * ((uint64_t)H + 1) + a4(2u * nnz_s) + a4(e * nnz_s) +
                        (coded ? (uint64_t)coded : 64ull * n_dense) + a4(e * n_out_d);
  if (size > in.npay && size - in.npay > ovf_avail) return false;
  const uint32_t o_bm = 16u, o_rp = o_bm + 4u * nbm, o_col = o_rp + 4u * (H + 1u);
  const uint32_t o_val = o_col + a4(2u * nnz_s), o_codes = o_val + a4(e * nnz_s);
  const uint32_t o_outl = o_codes + (coded ? coded : 64u * n_dense);
  const uint32_t nw = t.block ? t.nwarps : 1u, wid = t.block ? threadIdx.x >> 5 : 0u, lane = threadIdx.x & 31u;
  uint32_t* bm = scr;              // the bitmap
  uint32_t* wp = bm + nbm;         // dense blocks before each of its words
  uint32_t* wsum = wp + nbm + 1u;  // one word per warp
  uint32_t* cho = wsum + kMaxWarps;  // (Huffman) start of every chunk
  uint16_t* block_of = reinterpret_cast<uint16_t*>(cho + nblk + 1u);  // by rank
  bool ok = true;
  for (uint32_t w = t.lane; w < nbm; w += t.size) {
    uint32_t m = in.ld32(o_bm + 4u * w);
    if (w == nblk >> 5) m &= (1u << (nblk & 31u)) - 1u;
    bm[w] = m;
    wp[w] = __popc(m);
  }
  if (t.lane == 0) wp[nbm] = 0;
  uint32_t o_chunks = 0, o_cb = 0;
  if (coded) {  // Huffman-coded section: the stored lengths and the chunks' sizes
    const uint32_t smin = in.ld8(o_codes + 1u), smax = in.ld8(o_codes + 2u);
    if (smin < 1u || smax < smin) return false;
    const uint32_t nl = smax - smin + 1u;
    o_cb = o_codes + 4u + a4(nl);
    o_chunks = o_cb + a4(n_dense);
    if (o_chunks - o_codes > coded) return false;
    for (uint32_t sym = t.lane; sym < 256u; sym += t.size)
      hd->len[sym] = sym == 0u ? (uint8_t)in.ld8(o_codes) : ((sym >= smin && sym <= smax) ? (uint8_t)in.ld8(o_codes + 4u + sym - smin) : (uint8_t)0);
    for (uint32_t r = t.lane; r <= n_dense; r += t.size) cho[r] = r < n_dense ? in.ld8(o_cb + r) : 0u;
  }
  team_sync(t);
  if (wid == 0) warp_excl_scan(wp, nbm + 1u);
  if (coded) {
    if (wid == min(1u, nw - 1u)) huffman_tables(hd);
    if (wid == nw - 1u) warp_excl_scan(cho, n_dense + 1u);
  }
  team_sync(t);
  if (wp[nbm] != n_dense) return false;  // (the same for every thread, and so is the next)
  if (coded) {
    if (!hd->ok || o_chunks - o_codes + cho[n_dense] > coded) return false;
    huffman_lut(hd, t.lane, t.size);
  }
  for (uint32_t b = t.lane; b < nblk; b += t.size)
    if ((bm[b >> 5] >> (b & 31u)) & 1u) block_of[wp[b >> 5] + __popc(bm[b >> 5] & ((1u << (b & 31u)) - 1u))] = (uint16_t)b;
  const bool vec = (W & 3u) == 0u && ((uint32_t)(uintptr_t)out & (DT == kF32 ? 15u : 7u)) == 0u;
  if (n_dense < nblk) {  // sparse blocks are zero but for the CSR entries
    const StepLane sl = step_lane(g);
    const float zero[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    for (uint32_t sr = wid; sr < g.nsr; sr += nw) {
      const uint32_t by = sr * (4u >> g.qs) + sl.qrow, y = by * 8u + sl.r;
      for (uint32_t bx = sl.q & sl.qm; by < g.nby && y < H && bx < nbx; bx += sl.qm + 1u) {
        const uint32_t b = by * nbx + bx;
        if (!((bm[b >> 5] >> (b & 31u)) & 1u)) store_seg<DT>(out, W, y, bx * 8u, min(8u, W - bx * 8u), vec, zero);
      }
    }
  }
  team_sync(t);
  const float two_eps = __fmul_rn(2.0f, eps), inv2e = __fdiv_rn(1.0f, two_eps);
  uint32_t outl0 = 0;
  for (uint32_t base = 0; base < n_dense; base += t.size) {
    const uint32_t rank = base + t.lane;
    uint32_t codes[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) codes[k] = 0x80808080u;
    if (rank < n_dense) {
      if (coded) {
        ok &= huffman_decode_chunk(in, o_chunks + cho[rank], cho[rank + 1u] - cho[rank], (uint32_t)size, hd, codes);
      } else {
#pragma unroll
        for (int k = 0; k < 16; ++k) codes[k] = in.ld32(o_codes + 64u * rank + 4u * k);
      }
    }
    const uint32_t n = count_verbatim(codes);
    uint32_t incl = n;
#pragma unroll
    for (uint32_t o = 1; o < 32u; o <<= 1) {
      const uint32_t up = __shfl_up_sync(full, incl, o);
      if (lane >= o) incl += up;
    }
    uint32_t first = outl0 + incl - n, all = __shfl_sync(full, incl, 31);
    if (t.block) {
      if (lane == 31u) wsum[wid] = incl;
      __syncthreads();
      all = 0;
      for (uint32_t k = 0; k < nw; ++k) {
        first += k < wid ? wsum[k] : 0u;
        all += wsum[k];
      }
      __syncthreads();
    }
    outl0 += all;
    if (rank < n_dense) {
      const uint32_t b = block_of[rank], by = b / nbx, bx = b - by * nbx;
      if (first + n > n_out_d) {
        ok = false;
      } else {
        restore_block<DT>(in, n_out_d ? o_outl : 0u, n_out_d ? n_out_d - 1u : 0u, first, codes, two_eps, inv2e, out, H, W, by * 8u, bx * 8u, vec);
      }
    }
  }
  if (n_dense == nblk) return ok && nnz_s == 0u;
  for (uint32_t y = t.lane >> 3; y < H && nnz_s; y += t.size >> 3) {
    const uint32_t r0 = in.ld32(o_rp + 4u * y), r1 = in.ld32(o_rp + 4u * y + 4u);
    if (r0 > r1 || r1 > nnz_s) {
      ok = false;
      continue;
    }
    for (uint32_t k = r0 + (lane & 7u); k < r1; k += 8u) {
      const uint32_t col = in.ld16(o_col + 2u * k), b = (y >> 3) * nbx + (col >> 3);
      if (col >= W || ((bm[b >> 5] >> (b & 31u)) & 1u)) ok = false;
      else if (DT == kF32) reinterpret_cast<uint32_t*>(out)[y * W + col] = in.ld32(o_val + 4u * k);
      else reinterpret_cast<uint16_t*>(out)[y * W + col] = (uint16_t)in.ld16(o_val + 2u * k);
    }
  }
  return ok;
}

// Outlier-rich planes of at most four blocks (plain codes) by one warp, all their dense blocks in one step: one plane, or
// four of one block each (FOUR: the eight lanes 8 q ... of plane q pass its payload `in` -- `avail` bytes of it --, its
// destination and whether it is there).  Destinations are shared memory.
template <int DT, bool FOUR>
__device__ __noinline__ bool decode_few(const Plan& pl, const FlatIn in, uint32_t avail, bool there, float eps, uint8_t* out) {
  const Geometry g(pl);
  const uint32_t H = g.H, W = g.W, e = g.esize, full = 0xFFFFFFFFu, lane = threadIdx.x & 31u, q = lane >> 3, j = lane & 7u;
  uint32_t nnz_s = 0, n_dense = 0, n_out_d = 0, bitmap = 0;
  bool ok = true;
  if (there) {
    nnz_s = in.ld32(0);
    n_dense = in.ld32(4);
    n_out_d = in.ld32(8);
    bitmap = in.ld32(16) & ((1u << g.nblk) - 1u);
    ok = nnz_s <= g.HW && n_dense == (uint32_t)__popc(bitmap) && n_out_d <= g.HW && in.ld32(12) == 0u &&
         20u + 4u * (H + 1u) + a4(2u * nnz_s) + a4(e * nnz_s) + 64u * n_dense + a4(e * n_out_d) <= avail;
  }
  there = there && ok;
  const uint32_t o_rp = 20u, o_col = o_rp + 4u * (H + 1u), o_val = o_col + a4(2u * nnz_s), o_codes = o_val + a4(e * nnz_s);
  const uint32_t o_outl = o_codes + 64u * n_dense;
  const bool some_sparse = there && n_dense < g.nblk;
  if (some_sparse) {
    if (FOUR) {
      for (uint32_t i = j; i < g.HW; i += 8u) store_elem<DT>(out, i, 0.0f);
    } else {
      for (uint32_t i = lane; i < g.HW; i += 32u) store_elem<DT>(out, i, 0.0f);
    }
  }
  __syncwarp();
  const uint32_t rank = FOUR ? 0u : q;
  const bool dense = there && rank < n_dense;
  if (__any_sync(full, dense)) {
    uint32_t b = 0;
    if (!FOUR) {  // the rank-th dense block
      uint32_t m = bitmap;
      for (uint32_t k = 0; k < rank; ++k) m &= m - 1u;
      b = m ? (uint32_t)__ffs((int)m) - 1u : 0u;
    }
    const uint32_t by = b / g.nbx, bx = b - by * g.nbx;
    const float two_eps = __fmul_rn(2.0f, eps);
    restore_columns<DT>(
        in, [&](int i) { return in.ld8(o_codes + 64u * rank + 8u * i + j); },
        [&](uint32_t n, uint32_t& o) {
          uint32_t first = 0;
          if (!FOUR) {
            const uint32_t n0 = __shfl_sync(full, n, 0), n1 = __shfl_sync(full, n, 8), n2 = __shfl_sync(full, n, 16);
            first = (q > 0u ? n0 : 0u) + (q > 1u ? n1 : 0u) + (q > 2u ? n2 : 0u);
          }
          o = o_outl + e * first;
          const bool held = first + n <= n_out_d;
          if (dense && !held) ok = false;
          return held;
        },
        dense, two_eps, __fdiv_rn(1.0f, two_eps), out, H, W, by * 8u, bx * 8u);
  }
  __syncwarp();
  if (some_sparse && nnz_s) {  // CSR entries: eight lanes to a row, or a lane to a row of its plane
    for (uint32_t y = FOUR ? j : q; y < H; y += FOUR ? 8u : 4u) {
      const uint32_t r0 = in.ld32(o_rp + 4u * y), r1 = in.ld32(o_rp + 4u * y + 4u);
      if (r0 > r1 || r1 > nnz_s) {
        ok = false;
        continue;
      }
      for (uint32_t k = r0 + (FOUR ? 0u : j); k < r1; k += FOUR ? 1u : 8u) {
        const uint32_t col = in.ld16(o_col + 2u * k);
        if (col >= W || ((bitmap >> ((y >> 3) * g.nbx + (col >> 3))) & 1u)) ok = false;
        else if (DT == kF32) reinterpret_cast<uint32_t*>(out)[y * W + col] = in.ld32(o_val + 4u * k);
        else reinterpret_cast<uint16_t*>(out)[y * W + col] = (uint16_t)in.ld16(o_val + 2u * k);
      }
    }
  } else if (there && nnz_s) {
    ok = false;
  }
  return ok;
}

// Header of a container against what the caller expects: 0 if it does not fit, the container's version (1, 2)
// otherwise; also returns code width, eps, total size and the number of outlier-rich planes.
__device__ __forceinline__ uint32_t check_header(const Plan& pl, const uint8_t* src, unsigned long long src_bytes, uint32_t& bits,
                                                 float& eps, unsigned long long& total, uint32_t& nsal) {
  if (src_bytes < 64ull + 16ull * pl.P) return 0u;
  const uint32_t* h = reinterpret_cast<const uint32_t*>(src);
  bits = __ldg(h + 1) >> 24;
  const uint32_t version = __ldg(h + 1) & 0xFFFFu;
  bool ok = __ldg(h) == kMagic && (version == 1u || version == 2u) && ((__ldg(h + 1) >> 16) & 0xFFu) == (uint32_t)pl.dtype &&
            (bits == 2u || bits == 4u || bits == 8u) && __ldg(h + 2) == pl.N && __ldg(h + 3) == pl.C &&
            __ldg(h + 4) == (uint32_t)pl.H && __ldg(h + 5) == (uint32_t)pl.W && (__ldg(h + 6) & 0xFFFFu) == (8u | (8u << 8));
  total = (unsigned long long)__ldg(h + 14) | ((unsigned long long)__ldg(h + 15) << 32);
  eps = __uint_as_float(__ldg(h + 9));
  nsal = __ldg(h + 10);
  const unsigned long long npay = a16(4u * ((pl.HW * (bits & 15u) + 31u) / 32u));
  ok = ok && total <= src_bytes && total >= 64ull + 16ull * pl.P + pl.P * npay && eps >= 1e-30f && eps <= 1e30f;
  return ok ? version : 0u;
}

// Last step of every CTA.  The exit counter carries the CTAs that have left in its low half and, in its high half,
// how many of them had found something wrong; only such a CTA reports and fences, and the last CTA reads the
// status back only when there was one: a clean call ends with one atomic per CTA.  (The restored tensor needs no
// fence: its readers are later kernels.)
__device__ __forceinline__ void decompress_exit(const DecompressArgs& a, bool bad) {
  const bool any_bad = __syncthreads_or(bad) != 0;  // (the same for every thread)
  if (any_bad) {
    if (bad) atomicMax(&a.sc->status, (unsigned long long)kErrCorrupt);
    __threadfence();
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const unsigned long long old = atomicAdd(&a.sc->exited, 1ull | (any_bad ? 1ull << 32 : 0ull));
    if ((uint32_t)old == gridDim.x - 1u) {
      uint32_t code = kErrNone;
      if ((old >> 32) != 0ull || any_bad) {
        __threadfence();
        code = (uint32_t)ld_relaxed(&a.sc->status);
        st_relaxed(&a.sc->status, 0ull);
      }
      if (a.d_status) *a.d_status = status_word(code);
      st_relaxed(&a.sc->exited, 0ull);
    }
  }
}

// Four restored values of one group leave as one 16-byte (fp32) or 8-byte (bf16) store.
template <int DT>
__device__ __forceinline__ void store_group(uint8_t* out, uint32_t g, float v0, float v1, float v2, float v3) {
  if (DT == kF32) {
    reinterpret_cast<float4*>(out)[g] = make_float4(v0, v1, v2, v3);
  } else {
    uint2 w;
    w.x = f32x2_to_bf16x2(v0, v1);
    w.y = f32x2_to_bf16x2(v2, v3);
    reinterpret_cast<uint2*>(out)[g] = w;
  }
}

// Four codes (the low bits of `word`) as biased floats 2^23 + q; dequant2 takes the bias off again and applies scale and
// minimum, two values an instruction.  Whole bytes are put under the exponent by one byte permutation.
template <int BITS>
__device__ __forceinline__ void spread4(uint32_t word, uint32_t (&q)[4]) {
  constexpr uint32_t bias = 0x4B000000u;
  if (BITS == 8) {
#pragma unroll
    for (uint32_t j = 0; j < 4u; ++j) q[j] = __byte_perm(word, bias, 0x7440u + j);
  } else if (BITS == 4) {
    const uint32_t even = word & 0x0F0Fu, odd = (word >> 4) & 0x0F0Fu;
    q[0] = __byte_perm(even, bias, 0x7440u);
    q[1] = __byte_perm(odd, bias, 0x7440u);
    q[2] = __byte_perm(even, bias, 0x7441u);
    q[3] = __byte_perm(odd, bias, 0x7441u);
  } else {
#pragma unroll
    for (uint32_t j = 0; j < 4u; ++j) q[j] = ((word >> (2u * j)) & 3u) | bias;
  }
}
__device__ __forceinline__ void dequant2(uint32_t q0, uint32_t q1, f32x2 scale2, f32x2 lo2, float& v0, float& v1) {
  const f32x2 q = pack2(__uint_as_float(q0), __uint_as_float(q1)), back = pack2(-8388608.0f, -8388608.0f);
  unpack2(fma2(add2(q, back), scale2, lo2), v0, v1);
}

// What a warp takes of a plane at a time: up to kLines lines of 32 16-byte vectors of the OUTPUT, 4 KB (fp32) or 2 KB (bf16).
// Lane l restores vector l of every line.
template <int DT>
struct Chunk {
  static constexpr uint32_t VE = DT == kF32 ? 4u : 8u;     // elements of a vector
  static constexpr int kLines = DT == kF32 ? 8 : 4;
};
// Codes of a lane's vectors.  ALIGNED: the plane starts on a 16-byte boundary of the tensor and is whole vectors.  Codes of a
// word and more a vector are loaded by the lane that restores it, narrower ones as whole words, lane after lane, and handed on
// by shuffle (WORDS).  Otherwise vectors are counted from the one that holds the plane's first element, `shift`
// of whose elements belong to the plane before, and a vector's codes are picked out of NW + 1 words by a funnel shift.
template <int DT, int BITS, bool ALIGNED>
struct ChunkCodes {
  static constexpr int VE = (int)Chunk<DT>::VE, VB = VE * BITS, K = Chunk<DT>::kLines, NW = VB > 32 ? 2 : 1;
  static constexpr bool WORDS = ALIGNED && VB < 32;
  static constexpr int J = WORDS ? K * VB / 32 : K, N = ALIGNED ? NW : NW + 1;
  uint32_t w[J][N];

  // vectors v0 + 32 k + lane, those below v1
  __device__ __forceinline__ void load(const uint8_t* slot, uint32_t nwords, uint32_t lane, uint32_t v0, uint32_t v1, uint32_t shift) {
    const uint32_t* s32 = reinterpret_cast<const uint32_t*>(slot);
#pragma unroll
    for (int k = 0; k < J; ++k) {
      const uint32_t v = v0 + (uint32_t)k * 32u + lane;
#pragma unroll
      for (int n = 0; n < N; ++n) w[k][n] = 0;
      if (WORDS) {
        const uint32_t i = (v0 >> 5) * VB + (uint32_t)k * 32u + lane;
        if (i < (v1 * VB + 31u) >> 5) w[k][0] = __ldg(s32 + i);
      } else if (ALIGNED) {
        if (v < v1) {
          if (VB == 32) {
            w[k][0] = __ldg(s32 + v);
          } else {
            const uint2 t = __ldg(reinterpret_cast<const uint2*>(slot) + v);
            w[k][0] = t.x;
            w[k][N - 1] = t.y;
          }
        }
      } else {
        const int32_t i0 = (int32_t)(v * VE) - (int32_t)shift, w0 = (i0 * BITS) >> 5;
#pragma unroll
        for (int n = 0; n < N; ++n)
          if (v < v1 && (uint32_t)(w0 + n) < nwords) w[k][n] = __ldg(s32 + w0 + n);
      }
    }
  }

  // restores them to the plane at `out`
  __device__ __forceinline__ void restore(uint32_t lane, uint32_t v0, uint32_t v1, uint32_t HW, uint32_t shift, float scale, float lo, uint8_t* out) const {
    const f32x2 scale2 = pack2(scale, scale), lo2 = pack2(lo, lo);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t v = v0 + (uint32_t)k * 32u + lane;
      uint32_t mine = 0;
      if (WORDS) {  // the vector's bits are bits (32 k + lane) * VB ... of the chunk's
        constexpr uint32_t per = 32 / VB;  // vectors of a word
        mine = __shfl_sync(0xFFFFFFFFu, w[k * VB / 32][0], (uint32_t)(k * VB) % 32u + lane / per) >> (lane % per * VB);
      }
      if (v >= v1) continue;
      const int32_t i0 = (int32_t)(v * VE) - (int32_t)shift;
      float x[VE];
#pragma unroll
      for (int h = 0; h < VE; h += 4) {
        constexpr int per = 32 / BITS;  // codes of a word
        const int n = h / per;
        uint32_t word = WORDS ? mine : w[WORDS ? 0 : k][n], q[4];
        if (!ALIGNED) word = __funnelshift_r(word, w[WORDS ? 0 : k][n + 1 < N ? n + 1 : N - 1], (uint32_t)(i0 * BITS) & 31u);
        spread4<BITS>(word >> ((h % per) * BITS), q);
        dequant2(q[0], q[1], scale2, lo2, x[h], x[h + 1]);
        dequant2(q[2], q[3], scale2, lo2, x[h + 2], x[h + 3]);
      }
      if (ALIGNED || (i0 >= 0 && i0 + VE <= (int32_t)HW)) {
        uint4 t;
        if (DT == kF32) {
          t = make_uint4(__float_as_uint(x[0]), __float_as_uint(x[1]), __float_as_uint(x[2]), __float_as_uint(x[3]));
        } else {
          t.x = f32x2_to_bf16x2(x[0], x[1]);
          t.y = f32x2_to_bf16x2(x[2], x[3]);
          t.z = f32x2_to_bf16x2(x[VE - 4], x[VE - 3]);
          t.w = f32x2_to_bf16x2(x[VE - 2], x[VE - 1]);
        }
        *reinterpret_cast<uint4*>(out + (int64_t)i0 * (DT == kF32 ? 4 : 2)) = t;
      } else {  // the plane's first and last vectors, which it may share with its neighbours
#pragma unroll
        for (int j = 0; j < VE; ++j)
          if (i0 + j >= 0 && i0 + j < (int32_t)HW) store_elem<DT>(out, (uint32_t)(i0 + j), x[j]);
      }
    }
  }
};

// What the streaming part of decompress_kernel needs to know of the container.
struct StreamIn {
  const uint8_t* src;
  uint8_t* dst;
  unsigned long long total, slots_off, ovf_off, plane_bytes;
  uint32_t P, HW, npay, nsal;
};

// The normal and the raw planes: warp `w` takes items w, w + stride, ...; item = plane * chunks + chunk.  (Chunks of equal size
// instead of whole ones and a rest: bf16 planes of 56 x 56 31.0 -> 33.7 us.)  What bounds it is latency: the next item's codes and
// table entry are requested before the present one is worked on.
// us a call, chunk by chunk before and now: bf16, 2 bits, 128 x 96 planes of 112 x 112 84.5 -> 67.1, 128 x 144 of 56 x 56 41.9 ->
// 31.0, 128 x 192 of 28 x 28 17.1 -> 14.1; fp32, 4 bits, 64 x 128 of 28 x 28 9.3 -> 8.3.  `first`: the first item's entry,
// which was asked for along with the header.  False when the container is inconsistent.
template <int DT, int BITS, bool ALIGNED>
__device__ __forceinline__ bool stream_planes(const StreamIn& in, uint32_t w, uint32_t stride, uint4 first) {
  constexpr uint32_t VE = Chunk<DT>::VE, LINES = Chunk<DT>::kLines;
  const uint32_t lane = threadIdx.x & 31u, HW = in.HW;
  const uint32_t lines = chunk_lines(HW, VE, ALIGNED), chunks = (lines + LINES - 1u) / LINES;
  const uint32_t dp = stride / chunks, dc = stride - dp * chunks;
  const uint64_t pb = in.plane_bytes;
  uint32_t gp = w / chunks, ch = w - gp * chunks;
  bool good = true;
  if (gp >= in.P) return true;
  ChunkCodes<DT, BITS, ALIGNED> cur, nxt;
  uint4 e = first, en;
  // first vector of chunk c; `shift`: elements of the plane's first vector that belong to the plane before
  auto from = [&](uint32_t c) { return min(c * LINES, lines) * 32u; };
  auto shift_of = [&](uint32_t p) { return ALIGNED ? 0u : ((uint32_t)(p * pb) & 15u) / (DT == kF32 ? 4u : 2u); };
  auto last = [&](uint32_t p, uint32_t c) { return min(from(c + 1u), (HW + shift_of(p) + VE - 1u) / VE); };
  auto load = [&](uint32_t p, uint32_t c, ChunkCodes<DT, BITS, ALIGNED>& to) {
    // (the slot sits at a closed-form offset; what a plane of another class keeps there is read and dropped)
    to.load(in.src + in.slots_off + (uint64_t)p * in.npay, in.npay >> 2, lane, from(c), last(p, c), shift_of(p));
  };
  load(gp, ch, cur);
  for (;;) {
    uint32_t gn = gp + dp, cn = ch + dc;
    if (cn >= chunks) {
      cn -= chunks;
      ++gn;
    }
    const bool more = gn < in.P;
    if (more) {
      load(gn, cn, nxt);
      en = __ldg(reinterpret_cast<const uint4*>(in.src + 64) + gn);
    }
    const uint32_t cls = e.y & 3u;
    const unsigned long long off = (unsigned long long)e.x * 16ull;
    uint8_t* out = in.dst + gp * pb;
    if (cls == kClsNormal) {
      if (off == in.slots_off + (uint64_t)gp * in.npay)
        cur.restore(lane, from(ch), last(gp, ch), HW, shift_of(gp), __uint_as_float(e.w), __uint_as_float(e.z), out);
      else good = false;
    } else if (cls == kClsRaw) {
      // the continuation, when there is one, lies in the overflow region
      const unsigned long long ovf_avail = off ? in.total - off : 0ull;
      if ((off != 0 && (off < in.ovf_off || off > in.total)) || (pb > in.npay && pb - in.npay > ovf_avail)) {
        good = false;
      } else {
        SplitIn raw;
        raw.slot = in.src + in.slots_off + (uint64_t)gp * in.npay;
        raw.ovf = in.src + off;
        raw.npay = in.npay;
        constexpr uint32_t unit = ALIGNED ? 16u : (DT == kF32 ? 4u : 2u);
        const uint32_t n = (uint32_t)pb / unit, i1 = (uint32_t)((uint64_t)n * (ch + 1u) / chunks);
#pragma unroll 4
        for (uint32_t i = (uint32_t)((uint64_t)n * ch / chunks) + lane; i < i1; i += 32u) {
          if (ALIGNED) reinterpret_cast<uint4*>(out)[i] = __ldg(reinterpret_cast<const uint4*>(raw.at(16u * i)));
          else if (DT == kF32) reinterpret_cast<uint32_t*>(out)[i] = raw.ld32(4u * i);
          else reinterpret_cast<uint16_t*>(out)[i] = (uint16_t)raw.ld16(2u * i);
        }
      }
    } else if (cls != kClsSalient || in.nsal == 0u) {
      good = false;
    }
    if (!more) return good;
    gp = gn;
    ch = cn;
    cur = nxt;
    e = en;
  }
}

// Outlier-rich planes of the streaming kernels, from up to 256 table entries at a time: CTA c looks at those of planes c, c + hop,
// ..., gathers those that are outlier-rich and restores them, a warp each (pl.team = 32) or, when they have many blocks, the whole
// CTA one after the other.  (A macro: as a function, inlined or not, it costs the streaming loops registers, 28 x 28 planes 5 %.)
#define FH_RESTORE_OUTLIER_RICH(DT) \
  if (s_nsal) { \
    const uint32_t hop = (uint32_t)a.cta_stride, most = blockIdx.x < hop ? ((uint32_t)pl.P + hop - 1u) / hop : 0u; \
    const Team unit = pl.team == 32u ? make_warp_team(s_red) : make_team(kThreads, s_red); \
    uint32_t* scr = reinterpret_cast<uint32_t*>(smem + (pl.team == 32u ? (uint64_t)warp * pl.sal_stride : 0ull)); \
    HufDecode* hd = reinterpret_cast<HufDecode*>(reinterpret_cast<uint8_t*>(scr) + pl.sal_stride - pl.pay_bytes) - 1; \
    for (uint32_t base = 0; base < most; base += kThreads) { \
      const uint64_t gp = blockIdx.x + (uint64_t)(base + tid) * hop; \
      if (gp < pl.P && (__ldg(reinterpret_cast<const uint32_t*>(src + 64 + 16ull * gp) + 1) & 3u) == kClsSalient) \
        s_list[atomicAdd(&s_nlist, 1u)] = (uint32_t)gp; \
      __syncthreads(); \
      const uint32_t n = s_nlist; \
      for (uint32_t q = pl.team == 32u ? warp : 0u; q < n; q += pl.team == 32u ? (uint32_t)kWarps : 1u) { \
        const uint32_t gp = s_list[q]; \
        const unsigned long long off = (unsigned long long)__ldg(reinterpret_cast<const uint32_t*>(src + 64 + 16ull * gp)) * 16ull; \
        if (off != 0 && (off < ovf_off || off > total)) {  /* (the same for every thread of the unit) */ \
          bad = true; \
          continue; \
        } \
        SplitIn in; \
        in.slot = src + slots_off + (uint64_t)gp * npay; \
        in.ovf = src + off; \
        in.npay = npay; \
        /* the payload comes to shared memory first when it fits there */ \
        const unsigned long long ovf_avail = off ? total - off : 0ull; \
        const uint32_t got = (uint32_t)min((unsigned long long)pl.pay_bytes, npay + (ovf_avail & ~15ull)); \
        const uint32_t nnz_s = in.ld32(0), n_dense = in.ld32(4), n_out_d = in.ld32(8), coded = in.ld32(12), es = (uint32_t)pl.esize; \
        const uint64_t size = 16ull + 4ull * pl.nbm + 4ull * ((uint64_t)pl.H + 1) + a4(2u * nnz_s) + a4(es * nnz_s) + \
                              (coded ? (uint64_t)coded : 64ull * n_dense) + a4(es * n_out_d); \
        uint8_t* pay = reinterpret_cast<uint8_t*>(scr) + pl.sal_stride - pl.pay_bytes; \
        bool good; \
        if (nnz_s <= pl.HW && n_dense <= pl.nblk && n_out_d <= pl.HW && size <= got) { \
          for (uint32_t o = 16u * unit.lane; o < (uint32_t)size; o += 16u * unit.size) \
            *reinterpret_cast<uint4*>(pay + o) = __ldg(reinterpret_cast<const uint4*>(in.at(o))); \
          team_sync(unit); \
          FlatIn flat; \
          flat.p = pay; \
          flat.npay = got; \
          good = decode_salient<DT>(unit, s_pl, flat, 0ull, s_eps, a.dst + gp * pl.plane_bytes, scr, hd, s_hdr_ok); \
        } else { \
          good = decode_salient<DT>(unit, s_pl, in, ovf_avail, s_eps, a.dst + gp * pl.plane_bytes, scr, hd, s_hdr_ok); \
        } \
        if (!good) bad = true; \
        team_sync(unit);  /* the scratch is reused */ \
      } \
      __syncthreads(); \
      if (tid == 0) s_nlist = 0; \
      __syncthreads(); \
    } \
  }

// Planes of more than 128 groups.  Work items are (plane, chunk) pairs, a warp each (stream_planes), so that large
// planes spread over many warps; no barrier in the streaming part.  The items' stride is
// a prime (warps beyond it stay idle), so that a periodic pattern of expensive planes -- every eighth channel
// outlier-rich, say -- spreads over all warps instead of landing on the few whose index shares a factor with the period.
// ALIGNED: planes are whole 16-byte vectors (and so lie on 16-byte boundaries).
// Outlier-rich planes are left for the end (when the header says that there are any): CTA c then looks at the table
// entries of planes c, c + stride, ... -- the stride a prime again -- gathers those that are outlier-rich and restores
// them, a warp each (pl.team = 32) or, when they have many blocks, the whole CTA one after the other.
template <int DT, bool ALIGNED>
__global__ void __launch_bounds__(kThreads, 4) decompress_kernel(const Plan pl, const DecompressArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ double s_red[kMaxWarps * 4];
  __shared__ uint32_t s_hdr_ok, s_bits;
  __shared__ float s_eps;
  __shared__ unsigned long long s_total;
  __shared__ Plan s_pl;  // copy for the outlined slow path, which takes it by address
  __shared__ uint32_t s_nsal, s_list[kThreads], s_nlist;
  const uint32_t tid = threadIdx.x, warp = tid >> 5;
  if (tid == 0) {
    s_pl = pl;
    s_nlist = 0;
  }
  dep_trigger();  // the next kernel on the stream may become resident as this one drains
  dep_wait();     // the previous kernel on the stream (the one that wrote the container) has completed
  const unsigned long long off_in = a.d_off_in ? *a.d_off_in : 0ull;
  const uint8_t* src = a.src_base + off_in;
  const unsigned long long src_bytes = a.src_bytes > off_in ? a.src_bytes - off_in : 0ull;

  const uint32_t stride = (uint32_t)a.team_stride, wid = blockIdx.x * kWarps + warp;
  // the first item's table entry along with the header (every CTA checks it, it is 64 bytes)
  constexpr uint32_t VE = Chunk<DT>::VE, LINES = Chunk<DT>::kLines;
  const uint32_t gp0 = wid / ((chunk_lines(pl.HW, VE, ALIGNED) + LINES - 1u) / LINES);
  uint4 first = make_uint4(0u, 0u, 0u, 0u);
  if (gp0 < pl.P && src_bytes >= 64ull + 16ull * pl.P) first = __ldg(reinterpret_cast<const uint4*>(src + 64) + gp0);
  if (tid == 0) {
    uint32_t bits = 0;
    float eps = 0.0f;
    unsigned long long total = 0;
    uint32_t nsal = 0;
    s_hdr_ok = check_header(pl, src, src_bytes, bits, eps, total, nsal);
    s_nsal = nsal;
    s_bits = bits;
    s_eps = eps;
    s_total = total;
  }
  __syncthreads();
  const bool hdr_ok = s_hdr_ok != 0;
  bool bad = !hdr_ok;
  if (hdr_ok) {
    const uint32_t bits = s_bits;
    const unsigned long long total = s_total;
    const uint32_t npay = a16(4u * ((pl.HW * bits + 31u) / 32u));
    const unsigned long long slots_off = 64ull + 16ull * pl.P, ovf_off = slots_off + pl.P * (unsigned long long)npay;
    StreamIn in;
    in.src = src;
    in.dst = a.dst;
    in.total = total;
    in.slots_off = slots_off;
    in.ovf_off = ovf_off;
    in.plane_bytes = pl.plane_bytes;
    in.P = (uint32_t)pl.P;
    in.HW = pl.HW;
    in.npay = npay;
    in.nsal = s_nsal;
    if (wid < stride) {
      if (bits == 2u) bad = !stream_planes<DT, 2, ALIGNED>(in, wid, stride, first);
      else if (bits == 4u) bad = !stream_planes<DT, 4, ALIGNED>(in, wid, stride, first);
      else bad = !stream_planes<DT, 8, ALIGNED>(in, wid, stride, first);
    }
    FH_RESTORE_OUTLIER_RICH(DT)
  }
  decompress_exit(a, bad);
}

// Normal plane, whole-warp team, one chunk of up to 256 groups starting at group g0 (a multiple of
// 256).  The chunk's code bytes are fetched as 32-bit words, one or more coalesced loads per lane
// issued before anything else, and handed to the lanes that need them by shuffle: lane l restores
// groups g0 + l, g0 + 32 + l, ...  `w` holds the lane's words: word j*32 + l of the chunk's codes.
template <int BITS>
__device__ __forceinline__ void decode_chunk_large(const uint32_t (&w)[8], uint32_t lane, uint32_t g0, uint32_t g1,
                                               float scale, float lo, uint8_t* out) {
  constexpr uint32_t L = (1u << BITS) - 1u;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t g = g0 + (uint32_t)k * 32u + lane;
    uint32_t word;
    if (BITS == 2) {         // one code byte per group: byte k*32 + l = word k*8 + (l >> 2), byte l & 3
      const uint32_t src = __shfl_sync(0xFFFFFFFFu, w[k >> 2], (uint32_t)(k & 3) * 8u + (lane >> 2));
      word = (src >> ((lane & 3u) * 8u)) & 0xFFu;
    } else if (BITS == 4) {  // two code bytes per group: halfword k*32 + l = word k*16 + (l >> 1)
      const uint32_t src = __shfl_sync(0xFFFFFFFFu, w[k >> 1], (uint32_t)(k & 1) * 16u + (lane >> 1));
      word = (src >> ((lane & 1u) * 16u)) & 0xFFFFu;
    } else {                 // one word per group
      word = w[k];
    }
    if (g < g1)
      store_group<kF32>(out, g, dequant(word & L, scale, lo), dequant((word >> BITS) & L, scale, lo),
                      dequant((word >> (2 * BITS)) & L, scale, lo), dequant((word >> (3 * BITS)) & L, scale, lo));
  }
}

// Normal plane that does not start on a 16-byte boundary of the tensor (or whose last vector is shared with the next
// plane): lanes own aligned 16-byte vectors of the OUTPUT, and since decoding is element by element, each picks its
// elements' codes out of the bit stream with a funnel shift.  The plane's first and last vectors, which it may share
// with its neighbours, leave as element stores.  `v0`: first vector of the chunk, counted from the one that holds the
// plane's first element; `shift`: elements of that vector that belong to the plane before.
template <int BITS>
__device__ __forceinline__ void decode_chunk_large_shifted(const uint8_t* slot, uint32_t nwords, uint32_t lane, uint32_t v0, uint32_t HW,
                                                     uint32_t shift, float scale, float lo, uint8_t* out) {
  constexpr int VE = 4, K = 8;  // elements of a vector, vectors per lane
  constexpr uint32_t L = (1u << BITS) - 1u;
  constexpr int NW = VE * BITS > 32 ? 2 : 1;                      // words of codes of a vector
  const uint32_t* s32 = reinterpret_cast<const uint32_t*>(slot);
  uint32_t cw[K][NW];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int32_t i0 = (int32_t)((v0 + k * 32u + lane) * VE) - (int32_t)shift;
    const int32_t bit = i0 * BITS, w0 = bit >> 5;
    uint32_t w[NW + 1];
#pragma unroll
    for (int n = 0; n <= NW; ++n) w[n] = (i0 < (int32_t)HW && (uint32_t)(w0 + n) < nwords) ? __ldg(s32 + w0 + n) : 0u;
#pragma unroll
    for (int n = 0; n < NW; ++n) cw[k][n] = __funnelshift_r(w[n], w[n + 1], (uint32_t)bit & 31u);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int32_t i0 = (int32_t)((v0 + k * 32u + lane) * VE) - (int32_t)shift;
    float v[VE];
#pragma unroll
    for (int j = 0; j < VE; ++j) v[j] = dequant((cw[k][(j * BITS) >> 5] >> ((j * BITS) & 31)) & L, scale, lo);
    if (i0 >= 0 && i0 + VE <= (int32_t)HW) {
      *reinterpret_cast<float4*>(out + 4ll * i0) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int j = 0; j < VE; ++j)
        if (i0 + j >= 0 && i0 + j < (int32_t)HW) store_elem<kF32>(out, (uint32_t)(i0 + j), v[j]);
    }
  }
}

// fp32 tensors that are larger than the L2 cache: the same in chunks of 1,024 elements, one at a time, nothing requested ahead.
// Requests ahead pay while the restored elements stay in that cache and cost once they go to memory as they are written.  us a call,
// 4 bits, 28 x 28 / 56 x 56 / 112 x 112 planes, in this kernel and with stream_planes: 64 MiB 17.7 / 16.6 / 16.1 and 16.1 / 16.1 / 15.4, 96
// 24.2 / 22.9 / 22.9 and 23.4 / 22.9 / 22.1, 128 30.1 / 29.2 / 30.2 and 30.0 / 30.2 / 29.2, 160 36.2 / 35.2 / 37.3 and 36.1 / 36.2 / 36.4, 196
// 42.5 / 42.4 / 44.4 and 44.5 / 44.4 / 44.4, 256 53.8 / 54.8 / 55.8 and 56.7 / 56.8 / 55.8, 400 80.4 / 83.5 / 86.4 and 87.5 / 86.5 / 85.5.  (Neither
// is bound by HBM alone: DRAM is busy about half of the time, and waits for code words lead the stalls.  bf16 tensors have twice the
// elements to work on per byte and gain from requests ahead at any size.)
static __global__ void __launch_bounds__(kThreads, 4) decompress_large(const Plan pl, const DecompressArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ double s_red[kMaxWarps * 4];
  __shared__ uint32_t s_hdr_ok, s_bits;
  __shared__ float s_eps;
  __shared__ unsigned long long s_total;
  __shared__ Plan s_pl;  // copy for the outlined slow path, which takes it by address
  __shared__ uint32_t s_nsal, s_list[kThreads], s_nlist;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  if (tid == 0) {
    s_pl = pl;
    s_nlist = 0;
  }
  dep_trigger();  // the next kernel on the stream may become resident as this one drains
  dep_wait();     // the previous kernel on the stream (the one that wrote the container) has completed
  const unsigned long long off_in = a.d_off_in ? *a.d_off_in : 0ull;
  const uint8_t* src = a.src_base + off_in;
  const unsigned long long src_bytes = a.src_bytes > off_in ? a.src_bytes - off_in : 0ull;

  // header check (every CTA, it is 64 bytes)
  if (tid == 0) {
    uint32_t bits = 0;
    float eps = 0.0f;
    unsigned long long total = 0;
    uint32_t nsal = 0;
    s_hdr_ok = check_header(pl, src, src_bytes, bits, eps, total, nsal);
    s_nsal = nsal;
    s_bits = bits;
    s_eps = eps;
    s_total = total;
  }
  __syncthreads();
  const bool hdr_ok = s_hdr_ok != 0;
  bool bad = !hdr_ok;
  if (hdr_ok) {
    const uint32_t bits = s_bits;
    const unsigned long long total = s_total;
    const uint32_t npay = a16(4u * ((pl.HW * bits + 31u) / 32u));
    const unsigned long long slots_off = 64ull + 16ull * pl.P, ovf_off = slots_off + pl.P * (unsigned long long)npay;
    constexpr uint32_t VE = 4u;
    const bool aligned = (pl.plane_bytes & 15u) == 0u;  // (dst is 16-byte aligned)
    const uint32_t chunks = (pl.HW + (aligned ? 0u : VE - 1u) + 1023u) >> 10;
    const uint32_t items = (uint32_t)pl.P * chunks, stride = (uint32_t)a.team_stride;
    const uint32_t first = blockIdx.x * kWarps + warp;
    for (uint32_t item = first < stride ? first : items; item < items; item += stride) {
      const uint32_t gp = item / chunks, ch = item - gp * chunks;
      const uint32_t g0 = ch * 256u, g1 = min(pl.groups, g0 + 256u);
      const uint8_t* slot = src + slots_off + (uint64_t)gp * npay;
      // the chunk's code words are requested before the table entry is known (the slot sits at a closed-form offset;
      // what a salient plane keeps there is read and dropped)
      uint32_t cw[8];
      if (aligned) {
        const uint32_t* s32 = reinterpret_cast<const uint32_t*>(slot);
        const uint32_t nwords = npay >> 2, w0 = (g0 * bits) >> 3, per = bits;  // words per lane: 2, 4 or 8
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t i = w0 + (uint32_t)j * 32u + lane;
          cw[j] = ((uint32_t)j < per && i < nwords) ? __ldg(s32 + i) : 0u;
        }
      }
      const uint4 e = __ldg(reinterpret_cast<const uint4*>(src + 64) + gp);
      const unsigned long long off = (unsigned long long)e.x * 16ull;
      const uint32_t cls = e.y & 3u;
      uint8_t* out = a.dst + gp * pl.plane_bytes;
      if (cls == kClsNormal) {
        if (off != slots_off + (uint64_t)gp * npay) {
          bad = true;
          continue;
        }
        const float lo = __uint_as_float(e.z), scale = __uint_as_float(e.w);
        if (!aligned) {
          const uint32_t shift = ((uint32_t)(gp * pl.plane_bytes) & 15u) / 4u, v0 = ch * (1024u / VE);
          if (bits == 2u) decode_chunk_large_shifted<2>(slot, npay >> 2, lane, v0, pl.HW, shift, scale, lo, out);
          else if (bits == 4u) decode_chunk_large_shifted<4>(slot, npay >> 2, lane, v0, pl.HW, shift, scale, lo, out);
          else decode_chunk_large_shifted<8>(slot, npay >> 2, lane, v0, pl.HW, shift, scale, lo, out);
        } else {
          if (bits == 2u) decode_chunk_large<2>(cw, lane, g0, g1, scale, lo, out);
          else if (bits == 4u) decode_chunk_large<4>(cw, lane, g0, g1, scale, lo, out);
          else decode_chunk_large<8>(cw, lane, g0, g1, scale, lo, out);
        }
      } else if (cls == kClsRaw) {
        // the continuation, when there is one, lies in the overflow region
        const unsigned long long ovf_avail = off ? total - off : 0ull;
        if ((off != 0 && (off < ovf_off || off > total)) || (pl.plane_bytes > npay && pl.plane_bytes - npay > ovf_avail)) {
          bad = true;
          continue;
        }
        SplitIn in;
        in.slot = slot;
        in.ovf = src + off;
        in.npay = npay;
        const uint32_t i1 = min(pl.HW, (ch + 1u) * 1024u);
        for (uint32_t i = ch * 1024u + lane; i < i1; i += 32u) reinterpret_cast<uint32_t*>(out)[i] = in.ld32(4u * i);
      } else if (cls != kClsSalient || s_nsal == 0u) {
        bad = true;
      }
    }
    FH_RESTORE_OUTLIER_RICH(kF32)
  }
  decompress_exit(a, bad);
}

// -------------------------------------------------------------------------------------------------
// Small planes (at most 128 groups: 7x7, 14x14, 16x16, ...).  Such planes rarely start on 16-byte boundaries,
// and a team of a few lanes that stores its plane element by element scatters 4-byte stores over many
// sectors.  Here a CTA restores a tile of consecutive planes into shared memory -- a team of lanes per
// normal plane, the whole warp for an outlier-rich one -- and the tile leaves as one bulk (TMA) store.
// Tiles (256 / team planes) start on 16-byte boundaries; two buffers alternate.
// -------------------------------------------------------------------------------------------------

constexpr uint32_t kSmallGroups = 8;  // a lane restores at most so many groups

// Code words of groups lane, lane + tt, ... of a plane.
template <int BITS>
__device__ __forceinline__ void load_codes(const uint8_t* slot, uint32_t lane, uint32_t tt, uint32_t groups, uint32_t (&code)[kSmallGroups]) {
#pragma unroll
  for (uint32_t k = 0; k < kSmallGroups; ++k) {
    const uint32_t g = lane + k * tt;
    code[k] = 0;
    if (g < groups)
      code[k] = BITS == 2 ? (uint32_t)__ldg(slot + g)
                          : (BITS == 4 ? (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(slot) + g) : __ldg(reinterpret_cast<const uint32_t*>(slot) + g));
  }
}

template <int DT>
__global__ void __launch_bounds__(kThreads, 4) decompress_small(const Plan pl, const DecompressArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint32_t s_hdr_ok, s_bits;
  __shared__ float s_eps;
  __shared__ unsigned long long s_total;
  __shared__ Plan s_pl;  // copy for the outlined slow path, which takes it by address
  const uint32_t tid = threadIdx.x, wlane = tid & 31u;
  if (tid == 0) s_pl = pl;
  dep_trigger();  // the next kernel on the stream may become resident as this one drains
  dep_wait();     // the previous kernel on the stream (the one that wrote the container) has completed
  const unsigned long long off_in = a.d_off_in ? *a.d_off_in : 0ull;
  const uint8_t* src = a.src_base + off_in;
  const unsigned long long src_bytes = a.src_bytes > off_in ? a.src_bytes - off_in : 0ull;
  // table entry of the team's plane: the first is fetched along with the header, a tile's at the end of the one before
  const uint32_t tt = pl.team, lane = tid & (tt - 1u), lp = tid / tt;
  auto entry_of = [&](uint32_t tile) {
    const uint64_t gp = (uint64_t)tile * pl.ppt + lp;
    return tile < pl.ntiles && lp < pl.ppt && gp < pl.P ? __ldg(reinterpret_cast<const uint4*>(src + 64) + gp) : make_uint4(0u, 0u, 0u, 0u);
  };
  uint4 en = src_bytes >= 64ull + 16ull * pl.P ? entry_of(blockIdx.x) : make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    uint32_t bits = 0;
    float eps = 0.0f;
    unsigned long long total = 0;
    uint32_t nsal = 0;
    s_hdr_ok = check_header(pl, src, src_bytes, bits, eps, total, nsal);
    s_bits = bits;
    s_eps = eps;
    s_total = total;
  }
  __syncthreads();
  bool bad = s_hdr_ok == 0;
  if (!bad) {
    const uint32_t bits = s_bits, L = (1u << bits) - 1u;
    const float eps = s_eps;
    const unsigned long long total = s_total;
    const uint32_t npay = a16(4u * ((pl.HW * bits + 31u) / 32u));
    const unsigned long long slots_off = 64ull + 16ull * pl.P, ovf_off = slots_off + pl.P * (unsigned long long)npay;
    const Team warp_team = make_warp_team(nullptr);
    const bool vec = (pl.plane_bytes & (DT == kF32 ? 15u : 7u)) == 0u;  // planes start on vector boundaries in the tile buffer
    // (the warps' tables for Huffman-coded planes lie where the second tile buffer is: a container that may hold such planes
    // is restored with one buffer)
    const uint32_t other = s_hdr_ok == 1u ? pl.stage_bytes : 0u;
    uint32_t at = 0;
    for (uint32_t tile = blockIdx.x; tile < pl.ntiles; tile += gridDim.x, at = other - at) {
      uint8_t* tbuf = smem + at;
      const uint64_t p0 = (uint64_t)tile * pl.ppt;
      const uint32_t np = (uint32_t)min((uint64_t)pl.ppt, pl.P - p0);
      // the codes are requested before the entry is looked at (what another plane keeps in its slot is read and dropped)
      uint32_t code[kSmallGroups], ln = lane, st = tt;
      asm volatile("" : "+r"(ln), "+r"(st));  // (a lane's group numbers are worked out anew for each tile, not kept in registers)
      {
        const uint8_t* slot = src + slots_off + (p0 + lp) * npay;
        const uint32_t n = lp < np ? pl.groups : 0u;
        if (bits == 2u) load_codes<2>(slot, ln, st, n, code);
        else if (bits == 4u) load_codes<4>(slot, ln, st, n, code);
        else load_codes<8>(slot, ln, st, n, code);
      }
      if (tid == 0) {  // the store that left this buffer last has read it
        if (other) bulk_wait_read<1>();
        else bulk_wait_read<0>();
      }
      __syncthreads();
      bool salient = false, raw = false;
      uint32_t my_off16 = 0;
      if (lp < np) {
        const uint64_t gp = p0 + lp;
        my_off16 = en.x;
        const unsigned long long off = (unsigned long long)en.x * 16ull;
        const uint32_t cls = en.y & 3u;
        uint8_t* out = tbuf + (uint64_t)lp * pl.plane_bytes;
        if (cls == kClsNormal) {
          if (off != slots_off + gp * npay) {
            bad = true;
          } else {
            const float lo = __uint_as_float(en.z), scale = __uint_as_float(en.w);
#pragma unroll
            for (uint32_t k0 = 0; k0 < kSmallGroups; ++k0) {
              const uint32_t g = ln + k0 * st, word = code[k0];
              if (g >= pl.groups) break;
              const uint32_t i = 4u * g;
              if (vec && i + 3u < pl.HW) {  // whole group of a plane on a vector boundary: one store
                store_group<DT>(out, g, dequant(word & L, scale, lo), dequant((word >> bits) & L, scale, lo),
                                dequant((word >> (2u * bits)) & L, scale, lo), dequant((word >> (3u * bits)) & L, scale, lo));
              } else {
#pragma unroll
                for (uint32_t k = 0; k < 4u; ++k)
                  if (i + k < pl.HW) store_elem<DT>(out, i + k, dequant((word >> (k * bits)) & L, scale, lo));
              }
            }
          }
        } else if (cls == kClsRaw) {
          const unsigned long long ovf_avail = off ? total - off : 0ull;
          raw = !((off != 0 && (off < ovf_off || off > total)) || (pl.plane_bytes > npay && pl.plane_bytes - npay > ovf_avail));
          if (!raw) bad = true;
        } else if (cls == kClsSalient) {
          salient = true;
        } else {
          bad = true;
        }
      }
      // raw planes of the warp's slice, a word per lane and turn: each by its own team, or, when there are fewer of them than a
      // team would take rounds of eight loads, one after the other by the whole warp (always by the warp, 4,581,888 planes of
      // 1 x 2 took 518 us, 91,500 of 7 x 7 in bf16 31)
      if (uint32_t m = __ballot_sync(0xFFFFFFFFu, raw && lane == 0)) {
        const uint32_t pb = (uint32_t)pl.plane_bytes;
        auto copy = [&](uint32_t rlp, uint32_t off16, uint32_t j, uint32_t lanes) {
          SplitIn in;
          in.slot = src + slots_off + (p0 + rlp) * npay;
          in.ovf = src + (unsigned long long)off16 * 16ull;
          in.npay = npay;
          uint8_t* out = tbuf + (uint64_t)rlp * pb;
#pragma unroll 4
          for (uint32_t o = 4u * j; o < pb; o += 4u * lanes) {
            if (DT == kF32) {
              *reinterpret_cast<uint32_t*>(out + o) = in.ld32(o);
            } else if (o + 2u < pb) {
              const uint32_t w = in.ld32(o);
              *reinterpret_cast<uint16_t*>(out + o) = (uint16_t)w;
              *reinterpret_cast<uint16_t*>(out + o + 2u) = (uint16_t)(w >> 16);
            } else {
              *reinterpret_cast<uint16_t*>(out + o) = (uint16_t)in.ld16(o);
            }
          }
        };
        if (32u * tt * __popc(m) > pb) {
          if (raw) copy(lp, my_off16, lane, tt);
        } else {
          for (; m; m &= m - 1u) {
            const uint32_t first = (uint32_t)__ffs((int)m) - 1u;
            copy((tid & ~31u) / tt + first / tt, __shfl_sync(0xFFFFFFFFu, my_off16, (int)first), wlane, 32u);
          }
        }
      }
      // outlier-rich planes of the warp's slice, by the whole warp: four at a time when a plane is one block, one after
      // the other otherwise.  A payload (shorter than its plane, or it would have been stored raw) is copied to the
      // warp's scratch in one go, before its header is known, and decoded from there.
      uint32_t* scr = reinterpret_cast<uint32_t*>(smem + pl.sm_sal + (uint64_t)(tid >> 5) * pl.sal_stride);
      const bool four = pl.nblk == 1u;
      const uint32_t pay_max = a16((uint32_t)pl.plane_bytes), per = four ? 8u : 32u;
      uint8_t* pay = reinterpret_cast<uint8_t*>(scr) + pl.sal_stride - pl.pay_bytes + (four ? (wlane >> 3) * (pay_max + 16u) : 0u);
      for (uint32_t m = __ballot_sync(0xFFFFFFFFu, salient && lane == 0); m;) {
        uint32_t mm = m;  // the lane's plane: the (lane / 8)-th or the first of those that are left
        for (uint32_t k = 0; k < (four ? wlane >> 3 : 0u); ++k) mm &= mm - 1u;
        for (uint32_t k = 0; k < (four ? 4u : 1u); ++k) m &= m - 1u;
        const bool there = mm != 0u;
        const uint32_t first = there ? (uint32_t)__ffs((int)mm) - 1u : 0u, slp = (tid & ~31u) / tt + first / tt;
        const uint64_t gp = p0 + slp;
        const unsigned long long off = (unsigned long long)__shfl_sync(0xFFFFFFFFu, my_off16, (int)first) * 16ull;
        const bool use = there && !(off != 0 && (off < ovf_off || off > total));
        if (there && !use) bad = true;
        SplitIn in;
        in.slot = src + slots_off + gp * npay;
        in.ovf = src + off;
        in.npay = npay;
        const unsigned long long ovf_avail = off ? total - off : 0ull;
        const uint32_t avail = use ? (uint32_t)min((unsigned long long)pay_max, npay + (ovf_avail & ~15ull)) : 0u;
        for (uint32_t o = 16u * (wlane & (per - 1u)); o < avail; o += 16u * per)
          *reinterpret_cast<uint4*>(pay + o) = __ldg(reinterpret_cast<const uint4*>(in.at(o)));
        __syncwarp();
        FlatIn flat;
        flat.p = pay;
        flat.npay = avail;  // (what was copied: a payload longer than that is no salient plane's)
        uint8_t* out = tbuf + (uint64_t)slp * pl.plane_bytes;
        const bool coded = use && flat.ld32(12) != 0u;
        if (pl.nblk <= 4u && !__any_sync(0xFFFFFFFFu, coded)) {
          if (!(four ? decode_few<DT, true>(s_pl, flat, avail, use, eps, out) : decode_few<DT, false>(s_pl, flat, avail, use, eps, out)))
            bad = true;
        } else {  // planes of more blocks, and Huffman-coded ones (one after the other)
          for (uint32_t k = 0; k < 32u; k += per) {
            if (!__shfl_sync(0xFFFFFFFFu, use, (int)k)) continue;
            uint8_t* to = (uint8_t*)__shfl_sync(0xFFFFFFFFu, (unsigned long long)out, (int)k);
            FlatIn one;
            one.p = (const uint8_t*)__shfl_sync(0xFFFFFFFFu, (unsigned long long)flat.p, (int)k);
            one.npay = __shfl_sync(0xFFFFFFFFu, avail, (int)k);
            HufDecode* hd = reinterpret_cast<HufDecode*>(smem + pl.stage_bytes) + (tid >> 5);
            if (!decode_salient<DT>(warp_team, s_pl, one, 0ull, eps, to, scr, hd, s_hdr_ok)) bad = true;
            __syncwarp();
          }
        }
        __syncwarp();
      }
      en = entry_of(tile + gridDim.x);
      __syncthreads();
      // the tile leaves: one bulk store when it is whole 16-byte chunks, plain stores otherwise
      const uint32_t bytes = np * (uint32_t)pl.plane_bytes;
      uint8_t* dst = a.dst + p0 * pl.plane_bytes;
      if ((bytes & 15u) == 0u) {
        if (tid == 0) {
          fence_proxy_async();
          bulk_s2g(dst, tbuf, bytes);
          bulk_commit();
        }
      } else {
        for (uint32_t i = tid; i < (bytes >> 1); i += kThreads)
          reinterpret_cast<uint16_t*>(dst)[i] = reinterpret_cast<const uint16_t*>(tbuf)[i];
      }
    }
    if (tid == 0) bulk_wait<0>();  // every store of this CTA is complete
  }
  decompress_exit(a, bad);
}

}  // namespace fh

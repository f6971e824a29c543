// Compress kernels.
//
// Container recap: every plane owns a slot of npay bytes at a closed-form offset; a normal plane's
// codes fill its slot; the payload of an outlier-rich (salient) or raw plane runs through its slot and
// continues in the overflow region, in plane order.
//
// A call is ONE kernel, one pass over the dense tensor.  Tiles (runs of consecutive planes) are handed
// out in order by a ticket.  Per plane: statistics, three-sigma class, and
//   normal plane:   codes and table entry, written at once (the slot's offset is closed-form);
//   other planes:   measured (block classes, CSR and code sizes, salient versus raw) while they lie in shared memory or,
//                   larger ones of the warp-team kernel, when the CTA has run out of tiles; the tile publishes the overflow
//                   size of its planes, obtains the sum over all earlier tiles from the placement scan (fh_device.cuh) and
//                   the payloads are written.
// Variants by plane size:
//   compress_warp<DT, SIGMA, TT, K, EDGE>   planes of at most 256 groups: bulk-copy (TMA) pipeline, a sub-warp
//       team per plane, groups kept in registers; a warp handles an outlier-rich plane;
//   compress_cta_regs<DT, SIGMA, K, EDGE, PARTS, WORDS>   planes of up to 8,960 groups: one plane per CTA and tile, in registers;
//   compress_cta<SIGMA>                    still larger bf16 planes of whole 16-byte chunks: swept in shared memory;
//   compress_generic<DT, BITS, ROUND>      everything else (still larger ragged or fp32 planes, random rounding outside
//       the plane-wise three-sigma mode).
// The kernel's last CTA writes the header and the result words and returns the scratch to its idle state.
#pragma once

#include "fh_blocks.cuh"

namespace fh {

// Class and outlier count of plane gp when mu and sigma are taken per channel over the batch (the class is
// the channel's) or over the whole tensor (the class follows from the plane's own count).
__device__ __forceinline__ uint32_t channel_class(const Plan& pl, const CompressArgs& a, uint64_t gp, uint32_t& n_out) {
  n_out = a.plane_nout[gp];
  if (pl.mode == kModeTensor)
    return (uint64_t)n_out * pl.rho_den > (uint64_t)pl.rho_num * pl.HW ? kClsSalient : kClsNormal;
  const unsigned long long total = a.chan_stats[(gp % pl.C) * 4ull + 3ull];  // (see ChanStat)
  return total * pl.rho_den > (unsigned long long)pl.rho_num * pl.N * pl.HW ? kClsSalient : kClsNormal;
}

// What a CTA adds to the call's sums: the overflow units and numbers of its outlier-rich planes, and whether it has
// reported an error.  They stay with the CTA until it leaves (cta_exit).
struct CtaTotals {
  uint32_t units, nsal, nraw, err;
};
__device__ __forceinline__ CtaTotals* cta_totals() {
  __shared__ CtaTotals t;
  return &t;
}
__device__ __forceinline__ void report_error(const CompressArgs& a, uint32_t code) {
  *(volatile uint32_t*)&cta_totals()->err = 1u;
  atomicMax(&a.sc->status, (unsigned long long)code);
}

// Raw plane: verbatim copy through the slot into the overflow part, zero padded.
static __device__ __noinline__ void raw_write(const Team t, const Plan& pl, const uint8_t* plane, const SplitOut out) {
  const uint32_t n = (uint32_t)pl.plane_bytes, end = max(out.npay, a16(n));
  for (uint32_t o = 2u * t.lane; o < end; o += 2u * t.size)
    out.st16(o, o < n ? (uint32_t)*reinterpret_cast<const uint16_t*>(plane + o) : 0u);
}

// -------------------------------------------------------------------------------------------------
// Small planes (at most four blocks: 7x7, 8x8, 14x14, 16x16, ...) are encoded by one warp in one step, a lane per block
// row as in salient_measure: the blocks of one plane, or (FOUR) the single blocks of four planes, plane q = lane & 3.
// The elements are in registers, so the payload -- shorter than the plane, or the plane would be stored raw -- is put
// together in shared memory over the plane itself; what is left to do once its place is known is a copy.
// With a lane per two elements and a second encoding when the place was known, a plane took 1.6 us and 1.8 us of a warp's
// latency; the four of a step now take about the first together, and 0.5 us for the copy.
// -------------------------------------------------------------------------------------------------
constexpr uint32_t kSmallBlocks = 4;
__device__ __forceinline__ bool is_small_plane(const Plan& pl) { return pl.nblk <= kSmallBlocks && !pl.entropy; }
// Where a small plane's payload begins: its first word boundary (a bf16 plane may start between two).
__device__ __forceinline__ uint8_t* small_payload(uint8_t* plane) { return plane + (smem_u32(plane) & 2u); }

// `there`: the lane's plane is one to encode.  size: bytes of its payload; raw: it is left as it is and stored verbatim.
template <int DT, bool FOUR>
__device__ __noinline__ void encode_few(const Plan& pl, uint8_t* plane, bool there, uint32_t& size, bool& raw) {
  const uint32_t lane = threadIdx.x & 31u, r = lane >> 2, q = lane & 3u, full = 0xFFFFFFFFu;
  const uint32_t H = (uint32_t)pl.H, W = (uint32_t)pl.W, e = (uint32_t)pl.esize;
  const uint32_t qs = FOUR ? 0u : pl.qs, qm = (1u << qs) - 1u;
  const uint32_t by = FOUR ? 0u : q >> qs, bx = q & qm, y = by * 8u + r, x0 = bx * 8u;
  const bool valid = there && by < pl.nby && bx < pl.nbx;
  const uint32_t nin = valid && y < H ? min(8u, W - x0) : 0u;
  float v[8];
  load_seg<DT>(plane, W, y, x0, nin, seg_vec<DT>(plane, W), v);
  uint32_t nz = nonzero_mask(v), cnt = __popc(nz);
  const bool dense = block_sum(cnt) * pl.tau_den >= pl.tau_num * 64u && valid;
  const uint32_t dm = __ballot_sync(full, dense) & 15u;  // (row 0 of every block)
  uint32_t ca = 0, cb = 0, vm = 0;
  if (dm) {
    seg_codes(v, nin, __fdiv_rn(1.0f, __fmul_rn(2.0f, pl.eps)), ca, cb, vm);
    if (!dense) vm = 0;
  }
  if (dense) nz = cnt = 0;
  // CSR: entries of the plane's row and of the rows before it; entries of the row in the blocks to the left
  uint32_t left = cnt;
  if (qs > 0) {
    const uint32_t up = __shfl_up_sync(full, left, 1);
    if (bx >= 1u) left += up;
  }
  if (qs > 1) {
    const uint32_t up = __shfl_up_sync(full, left, 2);
    if (bx >= 2u) left += up;
  }
  const uint32_t row = __shfl_sync(full, left, (int)(lane | qm));
  const uint32_t rincl = block_prefix(row);
  const uint32_t r0 = __shfl_sync(full, rincl, 28), r1 = __shfl_sync(full, rincl, 29), r2 = __shfl_sync(full, rincl, 30),
                 r3 = __shfl_sync(full, rincl, 31);
  uint32_t rbefore = 0, nnz = 0;
  if (FOUR) {
    nnz = q < 2u ? (q ? r1 : r0) : (q == 2u ? r2 : r3);
  } else if (qs == 0u) {
    rbefore = (q > 0u ? r0 : 0u) + (q > 1u ? r1 : 0u) + (q > 2u ? r2 : 0u);
    nnz = r0 + r1 + r2 + r3;
  } else {
    rbefore = qs == 1u && q >= 2u ? r0 : 0u;
    nnz = qs == 1u ? r0 + r2 : r0;
  }
  const uint32_t rowp = rbefore + rincl - row;
  uint32_t pos = rowp + left - cnt;
  // verbatim elements, in raster order within a block
  const uint32_t c = __popc(vm), vincl = block_prefix(c);
  uint32_t vbefore = 0, n_out = 0;
  if (FOUR) n_out = __shfl_sync(full, vincl, (int)(28u + q));
  else across_blocks(vincl, q, vbefore, n_out);
  const uint32_t n_dense = FOUR ? (dense ? 1u : 0u) : __popc(dm), rank = FOUR ? 0u : __popc(dm & ((1u << q) - 1u));
  const uint32_t o_rp = 20u, o_col = o_rp + 4u * (H + 1u), o_val = o_col + a4(2u * nnz), o_codes = o_val + a4(e * nnz);
  const uint32_t o_outl = o_codes + 64u * n_dense;
  size = o_outl + a4(e * n_out);
  raw = a16(size) >= a16((uint32_t)pl.plane_bytes);
  __syncwarp();  // every element has been read
  if (!there || raw) return;
  uint8_t* const pay = small_payload(plane);
  auto st32 = [&](uint32_t o, uint32_t w) { *reinterpret_cast<uint32_t*>(pay + o) = w; };
  auto st16 = [&](uint32_t o, uint32_t w) { *reinterpret_cast<uint16_t*>(pay + o) = (uint16_t)w; };
  auto value = [&](uint32_t o, float f) {
    if (DT == kF32) st32(o, __float_as_uint(f));
    else st16(o, __float_as_uint(f) >> 16);
  };
  if (r == 0u && (FOUR || q == 0u)) {
    st32(0, nnz);
    st32(4, n_dense);
    st32(8, n_out);
    st32(12, 0);
    st32(16, FOUR ? n_dense : dm);
    st32(o_rp + 4u * H, nnz);
    // pads the section writers leave: col (2 bytes), val / verbatim values (bf16: 2 bytes)
    if (nnz & 1u) st16(o_col + 2u * nnz, 0);
    if (DT == kBF16 && (nnz & 1u)) st16(o_val + 2u * nnz, 0);
    if (DT == kBF16 && (n_out & 1u)) st16(o_outl + 2u * n_out, 0);
  }
  if (valid && bx == 0u && y < H) st32(o_rp + 4u * y, rowp);
#pragma unroll
  for (uint32_t j = 0; j < 8u; ++j)
    if ((nz >> j) & 1u) {
      st16(o_col + 2u * pos, x0 + j);
      value(o_val + e * pos, v[j]);
      ++pos;
    }
  if (dense) {
    st32(o_codes + 64u * rank + 8u * r, ca);
    st32(o_codes + 64u * rank + 8u * r + 4u, cb);
    uint32_t o = o_outl + e * (vbefore + vincl - c);
#pragma unroll
    for (uint32_t j = 0; j < 8u; ++j)
      if ((vm >> j) & 1u) {
        value(o, v[j]);
        o += e;
      }
  }
}

// `lanes` lanes (this is number j of them) store `n` bytes of a payload or a raw plane from shared memory through slot and
// overflow part, zero padded.  A bf16 plane may start between two words.
__device__ __forceinline__ void payload_copy(const uint8_t* from, uint32_t n, const SplitOut& out, uint32_t j, uint32_t lanes) {
  const uint32_t end = max(out.npay, a16(n));
  const bool half = (smem_u32(from) & 2u) != 0u;
  for (uint32_t o = 16u * j; o < end; o += 16u * lanes) {
    uint32_t w[4];
#pragma unroll
    for (uint32_t k = 0; k < 4u; ++k) {
      const uint32_t i = o + 4u * k;
      w[k] = 0;
      if (i + 4u <= n && !half) w[k] = *reinterpret_cast<const uint32_t*>(from + i);
      else if (i + 2u <= n) {
        w[k] = *reinterpret_cast<const uint16_t*>(from + i);
        if (i + 4u <= n) w[k] |= (uint32_t)*reinterpret_cast<const uint16_t*>(from + i + 2u) << 16;
      }
    }
    *reinterpret_cast<uint4*>(out.at(o)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// What every thread of a CTA knows about the destination.
struct Dest {
  uint8_t* dst;
  unsigned long long capacity, off_in;
  bool fits;  // header, table and slots fit the capacity
};
__device__ __forceinline__ Dest make_dest(const Plan& pl, const CompressArgs& a) {
  Dest d;
  d.off_in = a.d_off_in ? *a.d_off_in : 0ull;
  d.dst = a.dst_base + d.off_in;
  d.capacity = a.capacity > d.off_in ? a.capacity - d.off_in : 0ull;
  d.fits = d.capacity >= pl.ovf_off;
  return d;
}

// Overflow size, in 16-byte units, of a payload of `size` bytes.
__device__ __forceinline__ uint32_t ovf_units(const Plan& pl, uint32_t size) {
  return a16(size) > pl.npay ? (a16(size) - pl.npay) >> 4 : 0u;
}
// A measured plane is stored salient, or raw when that would not be smaller; returns its overflow units.
__device__ __forceinline__ uint32_t plane_units(const Plan& pl, const SalientInfo& info, bool& raw) {
  raw = a16(info.size) >= a16((uint32_t)pl.plane_bytes);
  return ovf_units(pl, raw ? (uint32_t)pl.plane_bytes : info.size);
}

// A tile's outlier-rich planes are added to the CTA's totals (one thread).
__device__ __forceinline__ void count_blockwise(uint32_t units, uint32_t nsal, uint32_t nraw) {
  CtaTotals* t = cta_totals();
  if (units) atomicAdd(&t->units, units);
  if (nsal) atomicAdd(&t->nsal, nsal);
  if (nraw) atomicAdd(&t->nraw, nraw);
}

// Writes the payload of the measured plane gp (`plane` in shared memory, `info` and `sal` from
// salient_measure) with its overflow part `at` units into the overflow region, and its table entry.
template <int DT, bool PARTS>
__device__ __forceinline__ void write_blockwise(const Team& t, const Plan& pl, const Dest& d, uint64_t gp,
                                                const uint8_t* plane, const SalientInfo& info, uint32_t* sal,
                                                uint32_t n_out, uint32_t at) {
  bool raw;
  const uint32_t my_units = plane_units(pl, info, raw);
  const unsigned long long off16 = (pl.ovf_off >> 4) + at;
  if (!d.fits || (off16 + my_units) * 16ull > d.capacity) return;  // never write past the capacity
  SplitOut out;
  out.slot = d.dst + pl.slots_off + gp * pl.npay;
  out.ovf = d.dst + off16 * 16ull;
  out.npay = pl.npay;
  if (raw) raw_write(t, pl, plane, out);
  else salient_write<DT, PARTS>(t, pl, plane, info, sal, out);
  if (t.lane == 0)
    reinterpret_cast<uint4*>(d.dst + 64)[gp] =
        make_uint4(my_units ? (uint32_t)off16 : 0u, (raw ? kClsRaw : kClsSalient) | (n_out << 2), 0u, 0u);
}

// One thread, after everything else of the call is done: header and result words.
__device__ __forceinline__ void finalize(const Plan& pl, const CompressArgs& a, const Dest& d, unsigned long long ovf16, uint32_t nsal,
                                         uint32_t nraw, uint32_t code) {
  const unsigned long long total = pl.ovf_off + ovf16 * 16ull;
  if (total > d.capacity && code < kErrCapacity) code = kErrCapacity;
  if (d.capacity >= 64) {
    uint4* hd = reinterpret_cast<uint4*>(d.dst);
    // a failed container must not pass for a valid one: no magic
    // (version 2: payloads may carry Huffman-coded sections)
    hd[0] = make_uint4(code == kErrNone ? kMagic : 0u, (pl.entropy ? 2u : 1u) | ((uint32_t)pl.dtype << 16) | ((uint32_t)pl.bits << 24),
                       pl.N, pl.C);
    hd[1] = make_uint4((uint32_t)pl.H, (uint32_t)pl.W, 8u | (8u << 8) | ((uint32_t)pl.rounding << 16) | ((uint32_t)pl.mode << 24),
                       pl.rho_num | (pl.rho_den << 16));
    hd[2] = make_uint4(pl.tau_num | (pl.tau_den << 16), __float_as_uint(pl.eps), nsal, nraw);
    hd[3] = make_uint4((uint32_t)pl.tensor_id, (uint32_t)(pl.tensor_id >> 32), (uint32_t)total, (uint32_t)(total >> 32));
  }
  if (a.out2) {
    a.out2[0] = total;
    a.out2[1] = status_word(code);
  }
  if (a.d_off_out) *a.d_off_out = code == kErrNone ? d.off_in + ((total + 255ull) & ~255ull) : (~0ull >> 1);
}

// Last step of every CTA: the last CTA to leave returns the group sums of the previous call's placement scan, the
// hand-out counters and the statistics of the channel- and tensor-wide modes to zero and finishes the container.
// The exit word carries the CTAs that have left, how many of them had something to add, and the overflow units of all:
//   CTAs | CTAs with something << 13 | units << 26
// The numbers of planes go the same way, each next to a count of the CTAs that added to it, by which the last CTA knows
// that a sum is complete: nothing has to be ordered, so that only a CTA with an error to report fences (the number of these
// is the topmost part of one of the sums).  (With counters
// changed while the CTA worked, a fence ahead of the exit word and another ahead of reading them back, a call with
// outlier-rich planes took 2.0 us from its last CTA's last store to its end, one without 0.5.)  The container itself
// needs no fence either: its readers are later kernels.
constexpr uint32_t kExitBits = 13, kExitMask = (1u << kExitBits) - 1u;  // (a grid has at most 32 CTAs per SM)
__device__ __forceinline__ bool has_totals(const CtaTotals& t) { return (t.units | t.nsal | t.nraw | t.err) != 0u; }
__device__ __forceinline__ void cta_exit(const Plan& pl, const CompressArgs& a, const Dest& d, uint32_t* s_last) {
  __syncthreads();  // every thread's notes are in
  const CtaTotals t = *cta_totals();
  unsigned long long now = 0;
  if (threadIdx.x == 0) {
    const bool some = has_totals(t);
    if (t.err) __threadfence();  // the error code before the CTA is counted out
    if (some) {
      atomicAdd(&a.sc->nsal, 1ull | (unsigned long long)t.nsal << kExitBits);
      atomicAdd(&a.sc->nraw, 1ull | (unsigned long long)t.nraw << kExitBits | (t.err ? 1ull << (64 - kExitBits) : 0ull));
    }
    const unsigned long long mine = 1ull | (some ? 1ull << kExitBits : 0ull) | (unsigned long long)t.units << (2 * kExitBits);
    now = atomicAdd(&a.sc->exited, mine) + mine;
    *s_last = ((uint32_t)now & kExitMask) == gridDim.x ? 1u : 0u;
  }
  __syncthreads();
  if (!*s_last) return;
  if (pl.mode != kModeOff)
    for (uint32_t k = threadIdx.x; k < a.scan.clear_groups; k += blockDim.x) a.scan.grp_clear[k] = 0ull;
  for (uint32_t k = threadIdx.x; k < a.chan_words; k += blockDim.x) a.chan_stats[k] = 0ull;  // (every CTA has read what it needed)
  if (threadIdx.x != 0) return;
  // (what follows is read by later kernels only, which start work after this one has completed: no fence)
  st_relaxed(&a.sc->ticket[a.parity], 0ull);
  st_relaxed(&a.sc->exited, 0ull);
  const uint32_t adders = (uint32_t)(now >> kExitBits) & kExitMask;
  unsigned long long vs = 0, vr = 0;
  uint32_t code = kErrNone;
  if (adders) {
    bool complete = false;
    for (uint32_t k = 0; k < a.scan.polls && !complete; ++k) {
      vs = ld_relaxed(&a.sc->nsal);
      vr = ld_relaxed(&a.sc->nraw);
      complete = ((uint32_t)vs & kExitMask) == adders && ((uint32_t)vr & kExitMask) == adders;
    }
    if (!complete) code = kErrTimeout;
    if (vr >> (64 - kExitBits)) {  // somebody has reported an error
      __threadfence();
      code = max(code, (uint32_t)ld_relaxed(&a.sc->status));
      st_relaxed(&a.sc->status, 0ull);
    }
    st_relaxed(&a.sc->nsal, 0ull);
    st_relaxed(&a.sc->nraw, 0ull);
    st_relaxed(&a.sc->done, 0ull);
    st_relaxed(&a.sc->queue, 0ull);
  }
  finalize(pl, a, d, now >> (2 * kExitBits), (uint32_t)(vs >> kExitBits), (uint32_t)(vr >> kExitBits), code);
  // after an error, entries may be left of tiles that were put off: they are zero between calls
  if (code && pl.mode != kModeOff)
    for (uint32_t k = 0; k < pl.ntiles; ++k) a.defer_next[k] = 0u;
}

__device__ __forceinline__ void store_table_entry(const Dest& d, uint64_t plane, uint32_t off16, uint32_t meta, float lo,
                                                  float scale) {
  reinterpret_cast<uint4*>(d.dst + 64)[plane] = make_uint4(off16, meta, __float_as_uint(lo), __float_as_uint(scale));
}

// Table entry of a plane that takes the block-wise path, until its payload is written: class salient, the
// three-sigma count; phase 1 leaves the plane's overflow size (16-byte units) where the offset will go, and of a small
// plane the bytes to store and whether it is raw.
__device__ __forceinline__ void store_marker(const Dest& d, uint64_t plane, uint32_t meta, uint32_t units, uint32_t bytes = 0, bool raw = false) {
  reinterpret_cast<uint4*>(d.dst + 64)[plane] = make_uint4(units, (meta & ~3u) | kClsSalient, bytes, raw ? 1u : 0u);
}
__device__ __forceinline__ uint2 load_marker(const Dest& d, uint64_t plane) {
  const volatile uint32_t* e = reinterpret_cast<const volatile uint32_t*>(d.dst + 64 + 16ull * plane);
  return make_uint2(e[0], e[1]);
}

// The block-wise path runs in two phases so that nothing in the streaming phase ever waits for another CTA.
// Phase 1, while a tile lies in shared memory: its outlier-rich planes are measured, or listed and measured when the CTA has run
// out of tiles (see warp_measure_put_off); the tile publishes the
// overflow size of its planes to the scan and is put off.  Phase 2, then: tiles put off are
// taken again (they come from the L2 cache when the tensor is small), obtain their place from the scan -- every tile
// before one has been published, or is about to be, by a CTA in phase 1 -- and the payloads are written.  Tiles put off
// wait in `defer_next`: linked from the CTA's own list (entry [tile]: the tile listed before it), or, in the CTA-team
// kernels, in a queue that all CTAs share (entry [n]: the n-th tile queued, plus one); an entry is returned to zero by
// who takes it.  This block sits in shared memory: what the outlined functions of both phases need.
constexpr uint32_t kNoTile = 0xFFFFFFFFu;
struct BlockCtl {
  Plan pl;
  CompressArgs a;
  Dest d;
  uint32_t U[kMaxStages], C[kMaxStages], arr[kMaxStages];  // warp-team kernel, per stage: units, counts (see kRawShift), warps done
  uint32_t base, ok;
  uint32_t head;                                           // warp-team and generic kernel: the tile this CTA listed last
  uint32_t held[kMaxStages];                               // the tile each stage buffer holds
  uint32_t next, ahead;                                    // CTA-team kernels, phase 2: the plane in hand, the one after it
  uint32_t own, own_stage, own_held;                       // ... the plane the measuring scratch is about (kNoTile: none), its stage, whether it still lies there ...
  SalientInfo own_info;                                    // ... and its sizes
};

// Warp-team kernel: what the tiles in the stages have gathered so far, and the tiles put off, as far as there is room (the
// others are linked like those of the CTA-team kernels).  A slice is what one warp sweeps of a tile.
constexpr uint32_t kListed = 32, kListedPlanes = 128;  // (static shared memory stays below what kSmemLimit leaves)
// Planes of more than four blocks are put off before they are measured (see warp_measure_put_off), as many of a CTA as are listed.  A
// tile with such a plane has to be listed too: the first warp that finds one asks for the entry.
constexpr uint32_t kNoEntry = 0xFFFFFFFFu, kEntryAsked = 0xFFFFFFFEu, kEntryFull = 0xFFFFFFFDu;
// A stage's counts: salient planes, raw ones, those put off (a tile has at most 256 planes).
constexpr uint32_t kRawShift = 10, kOffShift = 20, kCountMask = (1u << kRawShift) - 1u;
struct WarpList {
  uint32_t sum[kMaxStages][kWarps];  // overflow units of a slice (when the slice has outlier-rich planes)
  uint32_t mask[kMaxStages];         // slices that have some
  uint32_t count;                    // tiles put off
  uint32_t entry[kMaxStages];        // larger planes: the list entry of the tile in a stage
  uint32_t handed[2];                // phase 2: items handed out, in each of two passes
  uint32_t tile[kListed];
  uint32_t units[kListed], base[kListed];  // the tile's overflow units and, in phase 2, its place (kNoTile: not to be had)
  uint32_t before[kListed][kWarps];  // units of the tile's slices before this one
  uint8_t stage[kListed], slices[kListed];  // slices: those with such planes; larger planes: 0 for a tile that has been published
  uint32_t n[kListed];               // outlier-rich planes of the tile (as far as they are measured)
  // planes of more than four blocks: those put off, then, in phase 2, those of the listed tiles
  uint32_t planes;
  uint32_t place[kListedPlanes], meta[kListedPlanes];
  uint16_t lp[kListedPlanes];
  uint8_t of[kListedPlanes];         // whose entry (kListed: nobody's)
};

// One thread: tile `tile` has `units` of overflow in `nsal` salient and `nraw` raw planes.
__device__ __forceinline__ void publish_tile(BlockCtl* c, uint32_t tile, uint32_t units, uint32_t nsal, uint32_t nraw) {
  scan_publish(c->a.scan, tile, units);
  count_blockwise(units, nsal, nraw);
  if ((nsal | nraw) && c->d.fits) c->a.defer_next[tile] = atomicExch(&c->head, tile);
}

// Copies planes [p0, p0 + np) into `buf` (whole 16-byte chunks from the aligned start, the ragged end of the
// tensor byte-wise; all threads of the CTA) and returns the offset of plane p0 in it.
__device__ __forceinline__ uint32_t stage_planes(const Plan& pl, const uint8_t* src, uint64_t p0, uint32_t np, uint8_t* buf) {
  const uint64_t start = p0 * pl.plane_bytes, end = start + (uint64_t)np * pl.plane_bytes;
  const uint64_t a0 = start & ~15ull;
  const uint64_t a1 = min((end + 15ull) & ~15ull, pl.dense_bytes & ~15ull);
  const uint4* s16 = reinterpret_cast<const uint4*>(src + a0);
  uint4* t16 = reinterpret_cast<uint4*>(buf);
  const uint32_t n16 = (uint32_t)((a1 - a0) >> 4);
  for (uint32_t i = threadIdx.x; i < n16; i += blockDim.x) t16[i] = __ldg(s16 + i);
  for (uint64_t i = a1 + threadIdx.x; i < end; i += blockDim.x) buf[i - a0] = src[i];
  return (uint32_t)(start - a0);
}

// Distances d = x - lo of group g of a plane; positions past HW read as 0.
template <int DT>
__device__ __forceinline__ void load_dist(const uint8_t* plane, uint32_t g, uint32_t HW, bool vec, float lo, float d[4]) {
  float v[4];
  load_group<DT>(plane, g, HW, vec, v);
#pragma unroll
  for (int k = 0; k < 4; ++k) d[k] = (g * 4u + k < HW) ? __fsub_rn(v[k], lo) : 0.0f;
}

// Per-plane record kept in shared memory while a tile of the generic kernel is processed.
struct Rec {
  float lo, scale;
  uint32_t meta;   // class | n_out << 2
  uint32_t units;  // overflow units of a salient / raw plane
};

// =================================================================================================
// Generic streaming kernel
// =================================================================================================
// Tiles of consecutive planes are staged in shared memory with plain loads (planes need not start
// on a 16-byte boundary); a team per plane computes statistics and class; the codes of normal planes
// are staged in shared memory and leave with 16-byte stores.  Outlier-rich planes of the tile are then
// measured one after the other by the whole CTA, and written the same way in phase 2 (this kernel serves the
// odd shapes and is not tuned).  ROUND: random rounding, which serves planes of any size in the modes without plane-wise
// statistics and wants four CTAs to an SM (64 registers; with the 119 that the compiler takes, 64 x 64 fp32 planes of 56 x 56
// in mode OFF took 68.5 us, now 48.0); otherwise planes are so large that one or two CTAs fit.
template <int DT, int BITS, bool ROUND>
__global__ void __launch_bounds__(kThreads, ROUND ? 4 : 1) compress_generic(const Plan pl, const CompressArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ double s_red[kMaxWarps * 4];
  __shared__ uint32_t s_tile, s_last;
  __shared__ BlockCtl s_ctl;

  const uint32_t tid = threadIdx.x;
  if (tid == 0) *cta_totals() = CtaTotals{0u, 0u, 0u, 0u};
  if (tid == 0 && a.early_ticket) s_tile = (uint32_t)atomicAdd(&a.sc->ticket[a.parity], 1ull);
  if (tid == 0 && pl.mode != kModeOff) {  // (before the wait for the previous kernel, whose tail hides it)
    s_ctl.pl = pl;
    s_ctl.a = a;
    s_ctl.head = kNoTile;
  }
  dep_wait();     // the previous kernel on the stream has completed
  dep_trigger();  // the next kernel on the stream may become resident as this one drains
  uint8_t* tile_buf = smem + pl.sm_tile;
  uint8_t* out_buf = smem + pl.sm_out;
  Rec* rec = reinterpret_cast<Rec*>(smem + pl.sm_rec);
  uint32_t* sal = reinterpret_cast<uint32_t*>(smem + pl.sm_sal);
  const Dest d = make_dest(pl, a);
  if (tid == 0 && pl.mode != kModeOff) s_ctl.d = d;
  const Team team = make_team(pl.team, s_red);
  const Team cta = make_team(kThreads, s_red);
  const uint32_t nteams = team.block ? 1u : kThreads / team.size;
  const uint32_t my_team = team.block ? 0u : tid / team.size;
  constexpr uint32_t L = (1u << BITS) - 1u;
  const bool need_sigma = pl.mode == kModeAuto;
  uint32_t rp = 0;  // reduction counter (see red_half)
  if (!d.fits && tid == 0 && blockIdx.x == 0) report_error(a, kErrCapacity);

  for (bool first = true;; first = false) {
    if (tid == 0 && !(first && a.early_ticket)) s_tile = (uint32_t)atomicAdd(&a.sc->ticket[a.parity], 1ull);
    __syncthreads();
    const uint32_t tile = s_tile;
    if (tile >= pl.ntiles) break;
    const uint64_t p0 = (uint64_t)tile * pl.ppt;
    const uint32_t np = (uint32_t)min((uint64_t)pl.ppt, pl.P - p0);

    // ---- stage the tile
    const uint32_t head = stage_planes(pl, a.src, p0, np, tile_buf);
    __syncthreads();

    // ---- phase A: per-plane statistics, class, codes
    for (uint32_t lp = my_team; lp < np; lp += nteams) {
      const uint8_t* plane = tile_buf + head + (uint64_t)lp * pl.plane_bytes;
      const bool vec = (smem_u32(plane) & (DT == kF32 ? 15u : 7u)) == 0u;
      const uint32_t HW = pl.HW, nfull = HW >> 2, groups = pl.groups;
      float lo = __int_as_float(0x7F800000), hi = __int_as_float(0xFF800000);
      for (uint32_t g = team.lane; g < nfull; g += team.size) {
        float v[4];
        load_group<DT>(plane, g, HW, vec, v);
        lo = min3_nan(lo, min_nan(v[0], v[1]), min_nan(v[2], v[3]));
        hi = max3_nan(hi, max_nan(v[0], v[1]), max_nan(v[2], v[3]));
      }
      if ((HW & 3u) && team.lane == 0) {  // ragged last group
        for (uint32_t i = nfull * 4u; i < HW; ++i) {
          const float x = load_elem<DT>(plane, i);
          lo = min_nan(lo, x);
          hi = max_nan(hi, x);
        }
      }
      team_minmax(team, lo, hi, rp);
      const float range = __fsub_rn(hi, lo);
      if (!(fabsf(range) <= 3.402823466e38f) && team.lane == 0)
        report_error(a, kErrNonfinite);

      uint32_t cls = kClsNormal, n_out = 0;
      if (need_sigma) {
        const SigmaScale sc = sigma_scale(range);
        if (sc.applies) {  // (the same for every thread of the team)
          uint32_t as = 0, aq = 0, ng = 0;
          for (uint32_t g = team.lane; g < groups; g += team.size) {
            float dd[4];
            load_dist<DT>(plane, g, HW, vec, lo, dd);
            sigma_addends(dd, sc, as, aq);
            ++ng;
          }
          long long Is, Iq;
          if (team.block)
            team_sum2_wide(team, (long long)(int32_t)(as - ng * kMagicBits), (long long)(int32_t)(aq - ng * kMagicBits),
                           Is, Iq, rp);
          else
            team_sum2(team, (int32_t)(as - ng * kMagicBits), (int32_t)(aq - ng * kMagicBits), Is, Iq, rp);
          float dlo, dhi;
          sigma_thresholds(Is, Iq, sc, pl.inv_hw, dlo, dhi);
          uint32_t cnt = 0;
          for (uint32_t g = team.lane; g < groups; g += team.size) {
            float dd[4];
            load_dist<DT>(plane, g, HW, vec, lo, dd);
#pragma unroll
            for (int k = 0; k < 4; ++k) cnt += (g * 4u + k < HW) && ((dd[k] > dhi) || (dd[k] < dlo));
          }
          n_out = team_sum_u32(team, cnt, rp);
          if ((uint64_t)n_out * pl.rho_den > (uint64_t)pl.rho_num * HW) cls = kClsSalient;
        }
      } else if (pl.mode == kModeAll) {
        cls = kClsSalient;
      } else if (pl.mode >= kModeChannel) {
        cls = channel_class(pl, a, p0 + lp, n_out);
      }

      Rec r;
      r.lo = 0.0f;
      r.scale = 0.0f;
      r.units = 0;
      if (cls == kClsNormal) {
        float inv, scale;
        quant_params(range, L, inv, scale);
        r.lo = lo;
        r.scale = scale;
        uint8_t* o = out_buf + (uint64_t)lp * pl.npay;
        const uint32_t ogroups = pl.npay * 2u / BITS;
        for (uint32_t g = team.lane; g < ogroups; g += team.size) {
          uint32_t word = 0;
          if (g < groups) {
            float dd[4];
            load_dist<DT>(plane, g, HW, vec, lo, dd);
            if (ROUND) {  // one generator call per group: counter = (group, plane, tensor id), key = seed
              uint32_t rnd[4];
              philox4x32_10(g, (uint32_t)(p0 + lp), (uint32_t)pl.tensor_id, (uint32_t)(pl.tensor_id >> 32),
                            (uint32_t)pl.seed, (uint32_t)(pl.seed >> 32), rnd);
              word = quant4_random<BITS>(dd, inv, rnd);
              if (HW - g * 4u < 4u) word &= (1u << ((HW - g * 4u) * BITS)) - 1u;
            } else {
#pragma unroll
              for (int k = 0; k < 4; ++k) word |= (g * 4u + k < HW ? quant_code(dd[k], inv, L) : 0u) << (k * BITS);
            }
          }
          if (BITS == 2) o[g] = (uint8_t)word;
          else if (BITS == 4) reinterpret_cast<uint16_t*>(o)[g] = (uint16_t)word;
          else reinterpret_cast<uint32_t*>(o)[g] = word;
        }
      }
      r.meta = cls | (n_out << 2);
      if (team.lane == 0) rec[lp] = r;
    }
    __syncthreads();

    // ---- phase B: table entries and slots of the normal planes
    if (d.fits) {
      const uint32_t chunks = pl.npay >> 4;
      uint4* slots = reinterpret_cast<uint4*>(d.dst + pl.slots_off + p0 * pl.npay);
      for (uint32_t i = tid; i < np * chunks; i += kThreads) {
        const uint32_t lp = i / chunks;
        if ((rec[lp].meta & 3u) == kClsNormal) slots[i] = reinterpret_cast<const uint4*>(out_buf)[i];
      }
      for (uint32_t i = tid; i < np; i += kThreads)
        if ((rec[i].meta & 3u) == kClsNormal)
          store_table_entry(d, p0 + i, (uint32_t)((pl.slots_off + (p0 + i) * pl.npay) >> 4), rec[i].meta, rec[i].lo,
                            rec[i].scale);
    }

    // ---- phase C: the other planes are measured, one after the other by the whole CTA; the tile publishes
    // their overflow size and is put off until the CTA has run out of tiles
    if (pl.mode != kModeOff) {
      uint32_t U = 0, nsal = 0, nraw = 0;  // (every thread keeps the same figures)
      for (uint32_t lp = 0; lp < np; ++lp) {
        if ((rec[lp].meta & 3u) == kClsNormal) continue;
        const SalientInfo info = salient_measure_outlined<DT, true>(cta, s_ctl.pl, tile_buf + head + (uint64_t)lp * pl.plane_bytes, sal);
        bool raw;
        const uint32_t u = plane_units(pl, info, raw);
        if (tid == 0 && d.fits) store_marker(d, p0 + lp, rec[lp].meta, u);
        U += u;
        nsal += raw ? 0u : 1u;
        nraw += raw ? 1u : 0u;
        __syncthreads();  // the measuring scratch is reused
      }
      if (tid == 0) publish_tile(&s_ctl, tile, U, nsal, nraw);
    }
    __syncthreads();
  }

  // ---- phase 2: the tiles put off, newest first
  __syncthreads();
  for (uint32_t tile = pl.mode != kModeOff ? s_ctl.head : kNoTile; tile != kNoTile;) {
    const uint32_t next = a.defer_next[tile];
    const uint64_t p0 = (uint64_t)tile * pl.ppt;
    const uint32_t np = (uint32_t)min((uint64_t)pl.ppt, pl.P - p0);
    const uint32_t head = stage_planes(pl, a.src, p0, np, tile_buf);
    uint32_t U = 0;
    for (uint32_t i = tid; i < np; i += kThreads) {
      const uint2 m = load_marker(d, p0 + i);
      rec[i].meta = m.y;
      rec[i].units = (m.y & 3u) != kClsNormal ? m.x : 0u;
      U += rec[i].units;
    }
    U = __syncthreads_or(U);  // (only whether the tile has any overflow matters here)
    if (tid < 32u) {
      bool ok = true;
      uint32_t base = 0;
      if (U) ok = scan_prefix(a.scan, tile, base);
      if (tid == 0) {
        if (!ok) report_error(a, kErrTimeout);
        s_ctl.base = base;
        s_ctl.ok = ok;
      }
    }
    __syncthreads();
    if (s_ctl.ok) {
      uint32_t at = s_ctl.base;
      for (uint32_t lp = 0; lp < np; ++lp) {
        if ((rec[lp].meta & 3u) == kClsNormal) continue;
        const uint8_t* plane = tile_buf + head + (uint64_t)lp * pl.plane_bytes;
        const SalientInfo info = salient_measure_outlined<DT, true>(cta, s_ctl.pl, plane, sal);
        write_blockwise<DT, true>(cta, s_ctl.pl, d, p0 + lp, plane, info, sal, rec[lp].meta >> 2, at);
        at += rec[lp].units;
        __syncthreads();
      }
    }
    __syncthreads();
    if (tid == 0) a.defer_next[tile] = 0u;
    tile = next;
  }
  cta_exit(pl, a, d, &s_last);
}

// =================================================================================================
// Fast kernels
// =================================================================================================
// A team of TT lanes takes a run of groups, lane l groups l, l + TT, ... (K slots per lane), and keeps them in registers
// as fp32 for all that follows: minimum and maximum, distances from the minimum, integer moments, outlier count, codes.
// A run is a whole plane (warp-team kernel) or a warp's share of one (CTA-team kernel).
//
// K is chosen so that all slots but the last EDGE of them lie wholly inside the run for every lane; only those EDGE slots
// are masked.  (Checking every element against the plane's end made the 7 x 7 planes cost 75 instructions per element;
// a slot count known at run time only made the compiler spill: 56 x 56 18 -> 40 us.)  A masked position reads as another
// element of the run for minimum and maximum and is then held as distance 0, which adds exactly nothing to the moments
// and carries code 0; a lower threshold above 0 counts it, and it is subtracted again.
//
// Loads group `v` of the run at `p` (shared memory).  `grain`: the run starts on a 16-byte (2) or 8-byte (1) boundary, or
// on an element (0).  May read up to 16 bytes past the group.  fp32: the four values; bf16: two words of two.
template <int DT>
__device__ __forceinline__ void group_load(const uint8_t* p, uint32_t v, uint32_t grain, uint32_t (&w)[4]) {
  if (DT == kF32) {
    if (grain == 2u) {
      const uint4 t = reinterpret_cast<const uint4*>(p)[v];
      w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
    } else if (grain == 1u) {
      const uint2 t = reinterpret_cast<const uint2*>(p)[2u * v], u = reinterpret_cast<const uint2*>(p)[2u * v + 1u];
      w[0] = t.x; w[1] = t.y; w[2] = u.x; w[3] = u.y;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) w[e] = reinterpret_cast<const uint32_t*>(p)[4u * v + e];
    }
  } else {
    if (grain >= 1u) {
      const uint2 t = reinterpret_cast<const uint2*>(p)[v];
      w[0] = t.x; w[1] = t.y;
    } else {  // three aligned words hold the four elements at either parity
      const uint32_t odd = smem_u32(p) & 2u;
      const uint32_t* q = reinterpret_cast<const uint32_t*>(p - odd) + 2u * v;
      const uint32_t q0 = q[0], q1 = q[1], q2 = q[2];
      w[0] = __funnelshift_r(q0, q1, odd * 8u);
      w[1] = __funnelshift_r(q1, q2, odd * 8u);
    }
    w[2] = w[3] = 0;
  }
}
// Two bf16 minima / maxima per instruction; a NaN anywhere surfaces, -0 sorts below +0, as with the fp32 ones.
__device__ __forceinline__ uint32_t min2_nan_bf16(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("min.NaN.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t max2_nan_bf16(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// Runs of exactly K * TT groups (EDGE 0) start on 16-byte boundaries; in bf16 a lane then takes groups in neighbouring
// pairs, so that loads are 16 bytes wide and codes leave twice as wide (1 GiB of 32 x 32 planes: 373 -> 342 us).
// Loads a bf16 run of `n` elements as it lies there, two words a group, and takes the lane's minimum and maximum.
template <int K, int TT, int EDGE, int GRAIN>
__device__ __forceinline__ void run_load_words(const uint8_t* p, uint32_t lane, int32_t n, uint32_t (&x)[K][2], float& lo, float& hi) {
  static_assert(EDGE > 0 || K % 2 == 0, "pairs");
  const uint32_t last = (uint32_t)(n - 1) >> 2;
  uint32_t l0 = 0, h0 = 0, l1 = 0, h1 = 0, safe = 0;
  uint4 pair = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t v = lane + (uint32_t)(k * TT);
    uint32_t w[4];
    if (EDGE == 0) {
      if (k & 1) {
        w[0] = pair.z; w[1] = pair.w;
      } else {
        pair = (reinterpret_cast<const uint4*>(p) + lane)[(k >> 1) * TT];
        w[0] = pair.x; w[1] = pair.y;
      }
    } else {
      group_load<kBF16>(p, k >= K - EDGE ? min(v, last) : v, GRAIN, w);
    }
    if (k == 0) safe = __byte_perm(w[0], 0u, 0x1010);
    if (k >= K - EDGE) {
      const int32_t in = n - 4 * (int32_t)v;
      w[0] = in >= 2 ? w[0] : (in == 1 ? __byte_perm(w[0], safe, 0x5410) : safe);
      w[1] = in >= 4 ? w[1] : (in == 3 ? __byte_perm(w[1], safe, 0x5410) : safe);
    }
    if (k == 0) l0 = h0 = w[0], l1 = h1 = w[1];
    else {
      l0 = min2_nan_bf16(l0, w[0]); l1 = min2_nan_bf16(l1, w[1]);
      h0 = max2_nan_bf16(h0, w[0]); h1 = max2_nan_bf16(h1, w[1]);
    }
    x[k][0] = w[0];
    x[k][1] = w[1];
  }
  l0 = min2_nan_bf16(l0, l1);
  h0 = max2_nan_bf16(h0, h1);
  lo = min_nan(__uint_as_float(l0 << 16), __uint_as_float(l0 & 0xFFFF0000u));
  hi = max_nan(__uint_as_float(h0 << 16), __uint_as_float(h0 & 0xFFFF0000u));
}
// Loads the run of `n` elements and takes the lane's minimum and maximum.
template <int DT, int K, int TT, int EDGE, int GRAIN>
__device__ __forceinline__ void run_load_as(const uint8_t* p, uint32_t lane, int32_t n, float (&x)[K][4], float& lo, float& hi) {
  const uint32_t last = (uint32_t)(n - 1) >> 2;
  if (DT == kF32) {
    float lo1, hi1;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t v = lane + (uint32_t)(k * TT);
      uint32_t w[4];
      group_load<DT>(p, k >= K - EDGE ? min(v, last) : v, GRAIN, w);
#pragma unroll
      for (int e = 0; e < 4; ++e) x[k][e] = __uint_as_float(w[e]);
      if (k >= K - EDGE) {
        const int32_t in = n - 4 * (int32_t)v;
#pragma unroll
        for (int e = 0; e < 4; ++e) x[k][e] = e < in ? x[k][e] : (k == 0 ? __uint_as_float(w[0]) : x[0][0]);
      }
    }
    // per-group partial results keep the dependency chains short
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const float gl = min_nan(min3_nan(x[k][0], x[k][1], x[k][2]), x[k][3]);
      const float gh = max_nan(max3_nan(x[k][0], x[k][1], x[k][2]), x[k][3]);
      if (k == 0) lo = gl, hi = gh;
      else if (k == 1) lo1 = gl, hi1 = gh;
      else if (k & 1) lo1 = min_nan(lo1, gl), hi1 = max_nan(hi1, gh);
      else lo = min_nan(lo, gl), hi = max_nan(hi, gh);
    }
    lo = min_nan(lo, lo1);
    hi = max_nan(hi, hi1);
  } else {
    uint32_t w[K][2];
    run_load_words<K, TT, EDGE, GRAIN>(p, lane, n, w, lo, hi);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      x[k][0] = __uint_as_float(w[k][0] << 16); x[k][1] = __uint_as_float(w[k][0] & 0xFFFF0000u);
      x[k][2] = __uint_as_float(w[k][1] << 16); x[k][3] = __uint_as_float(w[k][1] & 0xFFFF0000u);
    }
  }
}
template <int DT, int K, int TT, int EDGE>
__device__ __forceinline__ void run_load(const uint8_t* p, uint32_t lane, int32_t n, uint32_t grain, float (&x)[K][4], float& lo, float& hi) {
  if (EDGE == 0 || grain == 2u) run_load_as<DT, K, TT, EDGE, 2>(p, lane, n, x, lo, hi);
  else if (DT == kF32 && grain == 1u) run_load_as<DT, K, TT, EDGE, 1>(p, lane, n, x, lo, hi);
  else run_load_as<DT, K, TT, EDGE, 0>(p, lane, n, x, lo, hi);
}
template <int DT, int K, int TT, int EDGE>
__device__ __forceinline__ void run_load(const uint8_t* p, uint32_t lane, int32_t n, uint32_t grain, uint32_t (&x)[K][2], float& lo, float& hi) {
  if (EDGE == 0 || grain >= 1u) run_load_words<K, TT, EDGE, 2>(p, lane, n, x, lo, hi);
  else run_load_words<K, TT, EDGE, 0>(p, lane, n, x, lo, hi);
}
// The grain of planes that follow one another from a 16-byte boundary on (for bf16 an 8-byte boundary is as good).
__device__ __forceinline__ uint32_t plane_grain(const Plan& pl) {
  return (pl.plane_bytes & 15u) == 0u ? 2u : ((pl.plane_bytes & 7u) == 0u ? (pl.esize == 2 ? 2u : 1u) : 0u);
}

// Distances from the minimum, in place (x - lo is x + (-lo): the same rounding); masked positions become distance 0.
// With SIGMA also the raw mantissa images of the groups' fixed-point addends (see sigma_addends2), summed with
// wrap-around: K magics beyond the addends themselves.
template <int DT, int K, int TT, int EDGE, bool SIGMA>
__device__ __forceinline__ void run_distances(uint32_t lane, int32_t n, float lo, const SigmaScale& sc, float (&x)[K][4], uint32_t& as,
                                              uint32_t& aq) {
  const float nlo = -lo;
  const f32x2 nlo2 = pack2(nlo, nlo);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    unpack2(add2(pack2(x[k][0], x[k][1]), nlo2), x[k][0], x[k][1]);
    unpack2(add2(pack2(x[k][2], x[k][3]), nlo2), x[k][2], x[k][3]);
    if (k >= K - EDGE) {
      const int32_t in = n - 4 * (int32_t)(lane + (uint32_t)(k * TT));
#pragma unroll
      for (int e = 0; e < 4; ++e) x[k][e] = e < in ? x[k][e] : 0.0f;
    }
    if (SIGMA) sigma_addends4(x[k][0], x[k][1], x[k][2], x[k][3], sc, as, aq);
  }
}

// Outliers among the lane's distances.  (Called only when some element can lie outside.)
template <int DT, int K, int TT, int EDGE>
__device__ __forceinline__ uint32_t run_count(uint32_t lane, int32_t n, float dlo, float dhi, const float (&x)[K][4]) {
  uint32_t c[4] = {0, 0, 0, 0};  // four counters: short dependency chains
  if (!__any_sync(0xFFFFFFFFu, 0.0f < dlo)) {  // nothing below: one compare per element
#pragma unroll
    for (int k = 0; k < K; ++k) {
#pragma unroll
      for (int e = 0; e < 4; ++e) c[e] += x[k][e] > dhi;
    }
    return (c[0] + c[1]) + (c[2] + c[3]);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
#pragma unroll
    for (int e = 0; e < 4; ++e) c[e] += (x[k][e] > dhi) || (x[k][e] < dlo);
  }
  uint32_t all = (c[0] + c[1]) + (c[2] + c[3]);
#pragma unroll
  for (int k = K - EDGE; k < K && EDGE > 0; ++k)  // masked positions (distance 0) are no elements
    if (0.0f < dlo) all -= (uint32_t)(4 - min(max(n - 4 * (int32_t)(lane + (uint32_t)(k * TT)), 0), 4));
  return all;
}

// Codes of the lane's groups, packed and stored to `slot` (where the run's first group goes).  Four codes of a group are
// the sum of (magic + q_e) << (e * BITS) minus the magic's contribution.
template <int DT, int K, int TT, int EDGE, int BITS>
__device__ __forceinline__ void run_codes(uint32_t lane, int32_t n, float inv, uint8_t* slot, const float (&x)[K][4]) {
  constexpr uint32_t bias = kMagicBits * (1u + (1u << BITS) + (1u << (2 * BITS)) + (1u << (3 * BITS)));
  constexpr bool PAIR = DT == kBF16 && EDGE == 0;
  const f32x2 inv2 = pack2(inv, inv), mag2 = pack2(kMagicF, kMagicF);
  uint8_t* out = slot + lane * (PAIR ? BITS : BITS / 2);
  uint32_t before = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    uint32_t w0, w1, w2, w3;
    unpack2u(fma2(pack2(x[k][0], x[k][1]), inv2, mag2), w0, w1);
    unpack2u(fma2(pack2(x[k][2], x[k][3]), inv2, mag2), w2, w3);
    const uint32_t word = w0 + (w1 << BITS) + (w2 << (2 * BITS)) + (w3 << (3 * BITS)) - bias;
    if (PAIR) {
      const int o = (k >> 1) * TT * BITS;
      if (!(k & 1)) before = word;
      else if (BITS == 2) *reinterpret_cast<uint16_t*>(out + o) = (uint16_t)(before | (word << 8));
      else if (BITS == 4) *reinterpret_cast<uint32_t*>(out + o) = before | (word << 16);
      else *reinterpret_cast<uint2*>(out + o) = make_uint2(before, word);
    } else if (k < K - EDGE || n > 4 * (int32_t)(lane + (uint32_t)(k * TT))) {
      if (BITS == 2) out[k * TT] = (uint8_t)word;
      else if (BITS == 4) *reinterpret_cast<uint16_t*>(out + 2 * k * TT) = (uint16_t)word;
      else *reinterpret_cast<uint32_t*>(out + 4 * k * TT) = word;
    }
  }
}
// Codes under random rounding: one generator call per group, counter = (group, plane, tensor id), key = seed; positions
// past the plane's end carry code 0 whatever the draw.  The run is read from its stage at `p` once more, in a loop: with
// the distances held in registers the generator's rounds, unrolled over the slots, spilled and overran the instruction
// cache (112 x 112: 150 us a call).  `g0`: the run's first group, whose codes go to `slot`.
// GRAIN: the run's, when the kernel fixes it (runs of whole groups), so that the loop holds one form of load; -1: `grain`.
// With width and grain looked at in the loop, 512 x 64 planes of 32 x 32 took 71.6 us, now 63.6.
template <int DT, int BITS, int GRAIN>
__device__ __forceinline__ void run_codes_random(const Plan& pl, const uint8_t* p, uint32_t grain, uint32_t lane, uint32_t step, int32_t n,
                                                 float lo, float inv, uint32_t g0, uint64_t gp, uint8_t* slot) {
  const uint32_t groups = (uint32_t)(n + 3) >> 2;
#pragma unroll 4
  for (uint32_t v = lane; v < groups; v += step) {
    uint32_t w[4], rnd[4];
    group_load<DT>(p, v, GRAIN < 0 ? grain : (uint32_t)GRAIN, w);
    philox4x32_10(g0 + v, (uint32_t)gp, (uint32_t)pl.tensor_id, (uint32_t)(pl.tensor_id >> 32), (uint32_t)pl.seed,
                  (uint32_t)(pl.seed >> 32), rnd);
    float x[4];
    if (DT == kF32) {
#pragma unroll
      for (int e = 0; e < 4; ++e) x[e] = __uint_as_float(w[e]);
    } else {
      x[0] = __uint_as_float(w[0] << 16); x[1] = __uint_as_float(w[0] & 0xFFFF0000u);
      x[2] = __uint_as_float(w[1] << 16); x[3] = __uint_as_float(w[1] & 0xFFFF0000u);
    }
    const float nlo = -lo;
    unpack2(add2(pack2(x[0], x[1]), pack2(nlo, nlo)), x[0], x[1]);
    unpack2(add2(pack2(x[2], x[3]), pack2(nlo, nlo)), x[2], x[3]);
    uint32_t word = quant4_random<BITS>(x, inv, rnd);
    const int32_t in = n - 4 * (int32_t)v;
    if (GRAIN < 0 && in < 4) word &= (1u << ((uint32_t)in * BITS)) - 1u;
    if (BITS == 2) slot[v] = (uint8_t)word;
    else if (BITS == 4) reinterpret_cast<uint16_t*>(slot)[v] = (uint16_t)word;
    else reinterpret_cast<uint32_t*>(slot)[v] = word;
  }
}
// Codes of a run, however they are rounded; `slot`: the plane's.
template <int DT, int SIGMA, int K, int TT, int EDGE>
__device__ __forceinline__ void run_codes_any(const Plan& pl, const uint8_t* p, uint32_t grain, uint32_t lane, int32_t n, float lo,
                                              float inv, uint32_t g0, uint64_t gp, uint8_t* slot, const float (&x)[K][4]) {
  uint8_t* at = slot + g0 * (uint32_t)pl.bits / 2u;
  constexpr int GRAIN = EDGE == 0 ? 2 : -1;
  if (SIGMA == 2) {
    if (pl.bits == 2) run_codes_random<DT, 2, GRAIN>(pl, p, grain, lane, TT, n, lo, inv, g0, gp, at);
    else if (pl.bits == 4) run_codes_random<DT, 4, GRAIN>(pl, p, grain, lane, TT, n, lo, inv, g0, gp, at);
    else run_codes_random<DT, 8, GRAIN>(pl, p, grain, lane, TT, n, lo, inv, g0, gp, at);
  } else if (pl.bits == 2) run_codes<DT, K, TT, EDGE, 2>(lane, n, inv, at, x);
  else if (pl.bits == 4) run_codes<DT, K, TT, EDGE, 4>(lane, n, inv, at, x);
  else run_codes<DT, K, TT, EDGE, 8>(lane, n, inv, at, x);
}

// ---- The same for bf16 runs that stay in registers as they lie in memory, two words a group: half the registers, so that more
// warps are resident, for six more instructions a group where distances are needed once more.
// Distances of a group's elements from the minimum.
__device__ __forceinline__ void word_distances(uint32_t w0, uint32_t w1, f32x2 nlo2, f32x2& p, f32x2& q) {
  p = add2(pack2(__uint_as_float(w0 << 16), __uint_as_float(w0 & 0xFFFF0000u)), nlo2);
  q = add2(pack2(__uint_as_float(w1 << 16), __uint_as_float(w1 & 0xFFFF0000u)), nlo2);
}
// Masked positions are set to the minimum, which is distance 0; then the moments.
template <int DT, int K, int TT, int EDGE, bool SIGMA>
__device__ __forceinline__ void run_distances(uint32_t lane, int32_t n, float lo, const SigmaScale& sc, uint32_t (&x)[K][2], uint32_t& as,
                                              uint32_t& aq) {
  const uint32_t lo2 = __byte_perm(__float_as_uint(lo), 0u, 0x3232);  // (the minimum is one of the elements)
  const f32x2 nlo2 = pack2(-lo, -lo);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (k >= K - EDGE) {
      const int32_t in = n - 4 * (int32_t)(lane + (uint32_t)(k * TT));
      x[k][0] = in >= 2 ? x[k][0] : (in == 1 ? __byte_perm(x[k][0], lo2, 0x5410) : lo2);
      x[k][1] = in >= 4 ? x[k][1] : (in == 3 ? __byte_perm(x[k][1], lo2, 0x5410) : lo2);
    }
    if (SIGMA) {
      f32x2 p, q;
      word_distances(x[k][0], x[k][1], nlo2, p, q);
      sigma_addends2(p, q, sc, as, aq);
      // (or the compiler keeps the distances for what follows, in local memory)
      asm volatile("" : "+r"(x[k][0]), "+r"(x[k][1]));
    }
  }
}
// The element that comes right above or below in the order of bf16 values.
__device__ __forceinline__ uint32_t bf16_above(uint32_t c) { return c & 0x8000u ? (c == 0x8000u ? 1u : c - 1u) : c + 1u; }
__device__ __forceinline__ uint32_t bf16_below(uint32_t c) { return c & 0x8000u ? c + 1u : (c == 0u ? 0x8001u : c - 1u); }
// A threshold on distances as one on elements: the largest element whose distance from `lo` does not exceed `t` (EQUAL: is less
// than `t`), twice in a word.  Distances, rounded as they are, grow with the element, so the neighbours of lo + t are looked at; false when
// none of three is it (the sum cancels), which leaves the comparison of distances.
// (Comparing distances always, 128 x 96 planes of 112 x 112: 109.1 -> 127.5 us.  Runs held as fp32 do better to compare their distances
// than to read the words again for this: 56 x 56 50.2 -> 57.0.)
template <bool EQUAL>
__device__ __forceinline__ bool element_cut(float lo, float t, uint32_t& cut) {
  const uint32_t b = __float_as_uint(__fadd_rn(lo, t));
  uint32_t c = (b >> 16) + ((b >> 31) && (b & 0xFFFFu) ? 1u : 0u);
  auto beyond = [&](uint32_t e) {
    const float d = __fsub_rn(__uint_as_float(e << 16), lo);
    return EQUAL ? !(d < t) : d > t;
  };
  if (beyond(c)) c = bf16_below(c);
  else if (!beyond(bf16_above(c))) c = bf16_above(c);
  cut = c | c << 16;
  return !beyond(c) && beyond(bf16_above(c));
}
struct Cuts {  // outliers are the elements above `above` and, when `low`, those up to `below`; !exact: compare distances
  uint32_t above, below, low, exact;
};
__device__ __forceinline__ Cuts element_cuts(float lo, float dlo, float dhi) {
  Cuts c;
  c.low = 0.0f < dlo;
  c.below = 0;
  bool exact = element_cut<false>(lo, dhi, c.above);
  if (c.low) exact &= element_cut<true>(lo, dlo, c.below);
  c.exact = exact;
  return c;
}
template <int DT, int K, int TT, int EDGE>
__device__ __forceinline__ uint32_t run_count(uint32_t lane, int32_t n, float lo, float dlo, float dhi, const Cuts& c, const uint32_t (&x)[K][2]) {
  uint32_t all = 0;
  if (c.exact) {  // one comparison and one addition for two elements; counts of at most 4 K are exact in bf16
    static_assert(2 * K <= 256, "counts in bf16");
    auto pair = [](uint32_t w) { return *reinterpret_cast<const __nv_bfloat162*>(&w); };
    const __nv_bfloat162 above = pair(c.above), below = pair(c.below);
    __nv_bfloat162 c0 = pair(0u), c1 = pair(0u);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      c0 = __hadd2(c0, __hgt2(pair(x[k][0]), above));
      c1 = __hadd2(c1, __hgt2(pair(x[k][1]), above));
    }
    if (c.low) {
#pragma unroll
      for (int k = 0; k < K; ++k) {
        c0 = __hadd2(c0, __hle2(pair(x[k][0]), below));
        c1 = __hadd2(c1, __hle2(pair(x[k][1]), below));
      }
    }
    c0 = __hadd2(c0, c1);
    all = (uint32_t)(__low2float(c0) + __high2float(c0));
  } else {
    const f32x2 nlo2 = pack2(-lo, -lo);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      f32x2 p, q;
      uint32_t w0 = x[k][0], w1 = x[k][1];
      asm volatile("" : "+r"(w0), "+r"(w1));
      word_distances(w0, w1, nlo2, p, q);
      float d[4];
      unpack2(p, d[0], d[1]);
      unpack2(q, d[2], d[3]);
#pragma unroll
      for (int e = 0; e < 4; ++e) all += (d[e] > dhi) || (d[e] < dlo);
    }
  }
#pragma unroll
  for (int k = K - EDGE; k < K && EDGE > 0; ++k)  // masked positions (distance 0) are no elements
    if (0.0f < dlo) all -= (uint32_t)(4 - min(max(n - 4 * (int32_t)(lane + (uint32_t)(k * TT)), 0), 4));
  return all;
}
template <int DT, int K, int TT, int EDGE, int BITS>
__device__ __forceinline__ void run_codes(uint32_t lane, int32_t n, float lo, float inv, uint8_t* slot, const uint32_t (&x)[K][2]) {
  constexpr uint32_t bias = kMagicBits * (1u + (1u << BITS) + (1u << (2 * BITS)) + (1u << (3 * BITS)));
  constexpr bool PAIR = EDGE == 0;
  const f32x2 inv2 = pack2(inv, inv), mag2 = pack2(kMagicF, kMagicF), nlo2 = pack2(-lo, -lo);
  uint8_t* out = slot + lane * (PAIR ? BITS : BITS / 2);
  uint32_t before = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    f32x2 p, q;
    uint32_t a = x[k][0], b = x[k][1], w0, w1, w2, w3;
    // (or the compiler works out all groups' distances ahead of the branch on the width, and has no registers for them)
    asm volatile("// %2" : "+r"(a), "+r"(b) : "n"(BITS));
    word_distances(a, b, nlo2, p, q);
    unpack2u(fma2(p, inv2, mag2), w0, w1);
    unpack2u(fma2(q, inv2, mag2), w2, w3);
    const uint32_t word = w0 + (w1 << BITS) + (w2 << (2 * BITS)) + (w3 << (3 * BITS)) - bias;
    if (PAIR) {
      const int o = (k >> 1) * TT * BITS;
      if (!(k & 1)) before = word;
      else if (BITS == 2) *reinterpret_cast<uint16_t*>(out + o) = (uint16_t)(before | (word << 8));
      else if (BITS == 4) *reinterpret_cast<uint32_t*>(out + o) = before | (word << 16);
      else *reinterpret_cast<uint2*>(out + o) = make_uint2(before, word);
    } else if (k < K - EDGE || n > 4 * (int32_t)(lane + (uint32_t)(k * TT))) {
      if (BITS == 2) out[k * TT] = (uint8_t)word;
      else if (BITS == 4) *reinterpret_cast<uint16_t*>(out + 2 * k * TT) = (uint16_t)word;
      else *reinterpret_cast<uint32_t*>(out + 4 * k * TT) = word;
    }
  }
}
template <int DT, int SIGMA, int K, int TT, int EDGE>
__device__ __forceinline__ void run_codes_any(const Plan& pl, const uint8_t* p, uint32_t grain, uint32_t lane, int32_t n, float lo,
                                              float inv, uint32_t g0, uint64_t gp, uint8_t* slot, const uint32_t (&x)[K][2]) {
  uint8_t* at = slot + g0 * (uint32_t)pl.bits / 2u;
  constexpr int GRAIN = EDGE == 0 ? 2 : -1;
  if (SIGMA == 2) {
    if (pl.bits == 2) run_codes_random<DT, 2, GRAIN>(pl, p, grain, lane, TT, n, lo, inv, g0, gp, at);
    else if (pl.bits == 4) run_codes_random<DT, 4, GRAIN>(pl, p, grain, lane, TT, n, lo, inv, g0, gp, at);
    else run_codes_random<DT, 8, GRAIN>(pl, p, grain, lane, TT, n, lo, inv, g0, gp, at);
  } else if (pl.bits == 2) run_codes<DT, K, TT, EDGE, 2>(lane, n, lo, inv, at, x);
  else if (pl.bits == 4) run_codes<DT, K, TT, EDGE, 4>(lane, n, lo, inv, at, x);
  else run_codes<DT, K, TT, EDGE, 8>(lane, n, lo, inv, at, x);
}
// Zero padding of a slot behind the codes, by `n` threads of which this is number `i`.
__device__ __forceinline__ void pad_slot(const Plan& pl, uint8_t* slot, uint32_t i, uint32_t n) {
  const uint32_t end = pl.groups * (uint32_t)pl.bits / 2u;
  if (end >= pl.npay) return;
  for (uint32_t o = end + i; o < a4(end); o += n) slot[o] = 0;
  for (uint32_t o = a4(end) + 4u * i; o < pl.npay; o += 4u * n) *reinterpret_cast<uint32_t*>(slot + o) = 0u;
}

// One sweep over a plane by a team of TT lanes: min/max -> distances from the minimum -> (integer moments -> thresholds
// -> count -> class) -> codes, stored straight to the plane's slot together with its table entry.  Returns class |
// n_out << 2; a normal plane is complete when the function returns.  All lanes of the warp run through it together
// (`active` is false in teams without a plane of their own: they look at somebody's and store nothing); what differs
// between teams is selected, not branched on, but for whole warps.
// SIGMA: 0 no three-sigma statistics, 1 the plane's own, 2 the same with random rounding of the codes.
template <int DT, int SIGMA, int K, int TT, int EDGE>
__device__ __forceinline__ uint32_t plane_sweep(const Team& team, const Plan& pl, const Dest& d, const CompressArgs& a,
                                                const uint8_t* plane, uint64_t gp, uint32_t grain, bool active, uint32_t& rp) {
  const uint32_t lane = team.lane, full = 0xFFFFFFFFu;
  const int32_t n = (int32_t)pl.HW;
  float x[K][4], lo, hi;
  run_load<DT, K, TT, EDGE>(plane, lane, n, grain, x, lo, hi);
  team_minmax(team, lo, hi, rp);
  const float range = __fsub_rn(hi, lo);
  if (!(fabsf(range) <= 3.402823466e38f) && lane == 0 && active) report_error(a, kErrNonfinite);
  uint32_t cls = kClsNormal, n_out = 0, as = 0, aq = 0;
  const SigmaScale sc = sigma_scale(range);
  run_distances<DT, K, TT, EDGE, (SIGMA != 0)>(lane, n, lo, sc, x, as, aq);
  if (SIGMA) {
    long long Is, Iq;
    team_sum2(team, (int32_t)(as - (uint32_t)K * kMagicBits), (int32_t)(aq - (uint32_t)K * kMagicBits), Is, Iq, rp);
    float dlo, dhi;
    sigma_thresholds((int32_t)Is, (int32_t)Iq, sc, pl.inv_hw, dlo, dhi);
    // outside [dlo, dhi] of a plane that the rule does not apply to, or whose extremes lie inside, there is nothing
    const bool look = sc.applies && (range > dhi || 0.0f < dlo);
    if (__any_sync(full, look)) {
      const uint32_t cnt = team_sum_u32(team, run_count<DT, K, TT, EDGE>(lane, n, dlo, dhi, x), rp);
      n_out = look ? cnt : 0u;
    }
    if ((uint64_t)n_out * pl.rho_den > (uint64_t)pl.rho_num * pl.HW) cls = kClsSalient;
  } else if (pl.mode == kModeAll) {
    cls = kClsSalient;
  } else if (pl.mode >= kModeChannel) {
    cls = channel_class(pl, a, gp, n_out);
  }
  const uint32_t meta = cls | (n_out << 2);
  if (cls != kClsNormal || !d.fits || !active) return meta;  // (the caller sees to a plane that is not normal)
  float inv, scale;
  quant_params(range, (1u << pl.bits) - 1u, inv, scale);
  uint8_t* slot = d.dst + pl.slots_off + gp * pl.npay;
  run_codes_any<DT, SIGMA, K, TT, EDGE>(pl, plane, grain, lane, n, lo, inv, 0u, gp, slot, x);
  pad_slot(pl, slot, lane, TT);
  if (lane == 0) store_table_entry(d, gp, (uint32_t)((pl.slots_off + gp * pl.npay) >> 4), meta, lo, scale);
  return meta;
}

// -------------------------------------------------------------------------------------------------
// Warp-team streaming kernel: planes of at most 256 groups.  Eight consumer warps and one producer
// warp per CTA.  The producer requests tiles and streams them into a ring of shared-memory stages
// with bulk copies.  A consumer warp sweeps its own planes of a tile (statistics, class, codes, stores)
// and never waits for another warp.  Outlier-rich planes are rare: a warp that has some in its slice encodes them (planes of at
// most four blocks) and adds their overflow size to the tile's sum in shared memory, or lists them (larger ones); the last of the
// tile's eight warps to get there publishes the tile or, when planes of it are only listed, puts it on the CTA's list for later.
//
// Registers are what this kernel is short of: 72 a thread at three CTAs to an SM.  What the compiler cannot keep goes to local
// memory, for which the stages leave some 28 KB of L1, so little is held across the calls of the outlined functions: a version of the
// sweep with 36 bytes a thread spilled instead of 24 took 3 % longer on 32 x 32 fp32 planes, 6 % on 24 x 24.  Stored bytes as the
// compiler reports them now, three-sigma rule, fp32: 8 to 20 in teams of a warp (32 x 32: 8), 8 to 32 in smaller ones (14 x 14: 28, 7 x 7:
// 32), up to 72 in those of one lane; bf16 8 to 24 and up to 64; without the rule 28 to 84, with random rounding 20 to 92.
// -------------------------------------------------------------------------------------------------
constexpr int kWarpKernelThreads = kThreads + 32;

// What was measured of a plane of more than four blocks waits for phase 2 in the plane's own slot, when that holds it:
// sizes, the measuring scratch and, with the Huffman stage, the code.  (Measuring a second time was half of phase 2.)
template <bool PARTS>
__device__ __forceinline__ uint32_t scratch_words(const Plan& pl) {
  return (uint32_t)pl.H * (PARTS ? pl.seg : 1u) + 1u + 2u * (pl.nsr + 1u) + pl.nbm + (pl.entropy ? pl.nsr + 1u : 0u);
}
template <bool PARTS>
__device__ __forceinline__ bool scratch_saved(const Plan& pl) {
  return 32u + 4u * scratch_words<PARTS>(pl) + (pl.entropy ? 4u * 256u : 0u) <= pl.npay;
}
template <bool PARTS>
__device__ __forceinline__ void scratch_save(const Team& t, const Plan& pl, const Dest& d, uint64_t gp, const SalientInfo& info, uint32_t* sal) {
  uint4* slot = reinterpret_cast<uint4*>(d.dst + pl.slots_off + gp * pl.npay);
  const HufEncode* h = sal_scratch(Geometry(pl), sal, Split<PARTS>(pl).seg).huf;
  if (t.lane == 0) {
    slot[0] = make_uint4(info.nnz_s, info.n_dense, info.n_out_d, info.size);
    slot[1] = pl.entropy ? make_uint4(info.coded, h->nlens, h->smin, h->smax) : make_uint4(0u, 0u, 0u, 0u);
  }
  uint32_t* w = reinterpret_cast<uint32_t*>(slot + 2);
  const uint32_t n = scratch_words<PARTS>(pl);
  for (uint32_t i = t.lane; i < n; i += t.size) w[i] = sal[i];
  if (info.coded)
    for (uint32_t i = t.lane; i < 256u; i += t.size) w[n + i] = h->code[i];
}
template <bool PARTS>
__device__ __forceinline__ SalientInfo scratch_load(const Team& t, const Plan& pl, const Dest& d, uint64_t gp, uint32_t* sal) {
  const uint4* slot = reinterpret_cast<const uint4*>(d.dst + pl.slots_off + gp * pl.npay);
  HufEncode* h = sal_scratch(Geometry(pl), sal, Split<PARTS>(pl).seg).huf;
  const uint4 v = __ldcg(slot), x = __ldcg(slot + 1);
  const uint32_t* w = reinterpret_cast<const uint32_t*>(slot + 2);
  const uint32_t n = scratch_words<PARTS>(pl);
  for (uint32_t i = t.lane; i < n; i += t.size) sal[i] = __ldcg(w + i);
  if (x.x) {
    for (uint32_t i = t.lane; i < 256u; i += t.size) h->code[i] = __ldcg(w + n + i);
    if (t.lane == 0) {
      h->nlens = x.y;
      h->smin = x.z;
      h->smax = x.w;
    }
  }
  SalientInfo info;
  info.nnz_s = v.x;
  info.n_dense = v.y;
  info.n_out_d = v.z;
  info.size = v.w;
  info.coded = x.x;
  return info;
}

// The lane that holds the k-th set bit of m (m has more than k).
__device__ __forceinline__ uint32_t nth_bit(uint32_t m, uint32_t k) {
  for (; k; --k) m &= m - 1u;
  return (uint32_t)__ffs((int)m) - 1u;
}

// Encodes small planes of a warp's slice where they lie, `plane_of(k)` the k-th of them, and passes their sizes on:
// done(k, size, raw) runs in one lane per plane.
template <int DT, typename PlaneOf, typename Done>
__device__ __forceinline__ void encode_small(const Plan& pl, uint32_t n, PlaneOf plane_of, Done done) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t size;
  bool raw;
  if (pl.nblk == 1u) {
    for (uint32_t k0 = 0; k0 < n; k0 += 4u) {
      const uint32_t k = k0 + (lane & 3u);
      encode_few<DT, true>(pl, plane_of(min(k, n - 1u)), k < n, size, raw);
      if (lane < 4u && k < n) done(k, size, raw);
    }
  } else {
    for (uint32_t k = 0; k < n; ++k) {
      encode_few<DT, false>(pl, plane_of(k), true, size, raw);
      if (lane == 0u) done(k, size, raw);
    }
  }
}

// The slice of a tile that the warp sweeps: it changes from tile to tile, so that a periodic pattern of outlier-rich planes does
// not land on the same warp every time.
__device__ __forceinline__ uint32_t warp_slice(uint32_t tile) { return ((threadIdx.x >> 5) + tile) & ((uint32_t)kWarps - 1u); }

// Phase 1, a warp with small outlier-rich planes in its slice (`leaders`: the first lanes of their teams; lp0: first
// plane of the slice): they are encoded where they lie, their sizes go into the sums of the tile in stage s and into their table
// markers.
template <int DT, int TT>
__device__ __noinline__ void warp_tile_encode(BlockCtl* c, WarpList* l, uint8_t* tbuf, uint32_t s, uint32_t leaders, uint32_t meta) {
  const Plan& pl = c->pl;
  const uint32_t tile = c->held[s], slice = warp_slice(tile);
  const uint64_t p0 = (uint64_t)tile * pl.ppt;
  const uint32_t lane = threadIdx.x & 31u, lp0 = slice * (32u / TT), n = __popc(leaders), full = 0xFFFFFFFFu;
  const uint32_t fits = c->d.fits;
  uint32_t total = 0, nraw = 0;
  encode_small<DT>(
      pl, n, [&](uint32_t k) { return tbuf + (uint64_t)(lp0 + nth_bit(leaders, k) / TT) * pl.plane_bytes; },
      [&](uint32_t k, uint32_t size, bool raw) {
        const uint32_t bytes = raw ? (uint32_t)pl.plane_bytes : size, u = ovf_units(pl, bytes);
        total += u;
        nraw += raw ? 1u : 0u;
        // (the leader's lane adds class and count afterwards)
        if (fits) store_marker(c->d, p0 + lp0 + nth_bit(leaders, k) / TT, 0u, u, bytes, raw);
      });
  __syncwarp();
  if (fits && ((leaders >> lane) & 1u))
    reinterpret_cast<uint32_t*>(c->d.dst + 64)[4ull * (p0 + lp0 + lane / TT) + 1ull] = (meta & ~3u) | kClsSalient;
  total += __shfl_xor_sync(full, total, 1);
  total += __shfl_xor_sync(full, total, 2);
  nraw += __shfl_xor_sync(full, nraw, 1);
  nraw += __shfl_xor_sync(full, nraw, 2);
  if (lane == 0) {
    l->sum[s][slice] = total;
    atomicOr(&l->mask[s], 1u << slice);
    if (total) atomicAdd(&c->U[s], total);
    atomicAdd(&c->C[s], (n - nraw) | (nraw << kRawShift));
  }
}

// The same for larger planes, which are listed, and measured when the CTA has run out of tiles (see warp_measure_put_off), as
// long as the list has room, and measured at once otherwise.
template <int DT, int TT>
__device__ __noinline__ void warp_tile_measure(BlockCtl* c, uint8_t* tbuf, uint64_t p0, uint32_t s, uint32_t slice, uint32_t leaders,
                                               uint32_t meta, uint32_t* sal) {
  const Plan& pl = c->pl;
  const uint32_t lane = threadIdx.x & 31u, lp0 = slice * (32u / TT), n = __popc(leaders), full = 0xFFFFFFFFu;
  uint32_t total = 0, nraw = 0;
  const Team team = make_warp_team(nullptr);
  for (uint32_t m = leaders; m; m &= m - 1u) {
    const uint32_t src = (uint32_t)__ffs((int)m) - 1u, lp = lp0 + src / TT;
    const SalientInfo info = salient_measure<DT, false>(team, pl, tbuf + (uint64_t)lp * pl.plane_bytes, sal);
    bool raw;
    const uint32_t u = plane_units(pl, info, raw);
    total += u;
    nraw += raw ? 1u : 0u;
    const uint32_t mt = __shfl_sync(full, meta, (int)src);
    if (lane == 0 && c->d.fits) store_marker(c->d, p0 + lp, mt, u);
    if (c->d.fits && scratch_saved<false>(pl)) scratch_save<false>(team, pl, c->d, p0 + lp, info, sal);
    __syncwarp();
  }
  if (lane == 0) {
    if (total) atomicAdd(&c->U[s], total);
    atomicAdd(&c->C[s], (n - nraw) | (nraw << kRawShift));
  }
}
template <int DT, int TT>
__device__ __noinline__ void warp_tile_put_off(BlockCtl* c, WarpList* l, uint8_t* tbuf, uint32_t s, uint32_t leaders, uint32_t meta,
                                               uint8_t* sal_base) {
  const uint32_t tile = c->held[s], slice = warp_slice(tile), lane = threadIdx.x & 31u, n = __popc(leaders);
  // (Not when every plane is outlier-rich and a CTA has several tiles: every warp has as many of them then, and measures its own while
  // the next tile is on its way.  us a call, put off / at once: fp32, 512 x 64 planes of 20 x 20 212 / 188, 2,358 x 16 of 172 x 2
  // 322 / 295; with one tile to a CTA the plane measured last need not be measured again: bf16, 4 x 513 of 23 x 23 26 / 33.)
  const bool even = c->pl.mode == kModeAll && !c->pl.entropy && c->pl.ntiles > gridDim.x;
  uint32_t at = kListedPlanes, e = kEntryFull;
  if (lane == 0 && !even) {
    at = atomicAdd(&l->planes, n);
    if (at + n <= kListedPlanes) {
      e = atomicCAS(&l->entry[s], kNoEntry, kEntryAsked);
      if (e == kNoEntry) {
        e = atomicAdd(&l->count, 1u);
        if (e < kListed) {
          l->tile[e] = tile;
          l->stage[e] = (uint8_t)s;
          l->slices[e] = 0xFFu;
        } else {
          e = kEntryFull;
        }
        atomicExch(&l->entry[s], e);
      }
      // (another warp is about to store it; without it the planes are measured here)
      for (uint32_t k = 0; e == kEntryAsked && k < (1u << 16); ++k) e = *(volatile uint32_t*)&l->entry[s];
    }
  }
  at = __shfl_sync(0xFFFFFFFFu, at, 0);
  e = __shfl_sync(0xFFFFFFFFu, e, 0);
  if (e < kListed) {
    if ((leaders >> lane) & 1u) {
      const uint32_t k = at + __popc(leaders & ((1u << lane) - 1u));
      l->of[k] = (uint8_t)e;
      l->lp[k] = (uint16_t)(slice * (32u / TT) + lane / TT);
      l->meta[k] = meta;
    }
    if (lane == 0) atomicAdd(&c->C[s], n << kOffShift);
    return;
  }
  if (lane < n && at + lane < kListedPlanes) l->of[at + lane] = (uint8_t)kListed;  // (nobody's)
  warp_tile_measure<DT, TT>(c, tbuf, (uint64_t)tile * c->pl.ppt, s, slice, leaders, meta,
                            reinterpret_cast<uint32_t*>(sal_base + (threadIdx.x >> 5) * c->pl.sal_stride));
}

// Phase 1, one thread: a tile with outlier-rich planes is published, or, when some of them are put off unmeasured, listed until
// they are.
static __device__ __noinline__ void warp_tile_publish(BlockCtl* c, WarpList* l, uint32_t s, uint32_t tile) {
  const uint32_t U = c->U[s], C = c->C[s];
  if (C < (1u << kOffShift)) scan_publish(c->a.scan, tile, U);
  const uint32_t nsal = C & kCountMask, nraw = (C >> kRawShift) & kCountMask, off = C >> kOffShift;
  count_blockwise(U, nsal, nraw);
  const uint32_t mask = l->mask[s];
  const uint32_t entry = l->entry[s];
  c->U[s] = 0;
  c->C[s] = 0;
  l->mask[s] = 0;
  l->entry[s] = kNoEntry;
  if (off) {
    l->units[entry] = U;
    l->n[entry] = nsal + nraw;
    return;
  }
  if (!c->d.fits) return;
  const uint32_t i = atomicAdd(&l->count, 1u);
  if (i >= kListed) {
    c->a.defer_next[tile] = atomicExch(&c->head, tile);
    return;
  }
  l->tile[i] = tile;
  l->units[i] = U;
  l->n[i] = nsal + nraw;
  l->stage[i] = (uint8_t)s;
  l->slices[i] = (uint8_t)mask;  // (larger planes' warps set none)
  uint32_t run = 0;
#pragma unroll
  for (uint32_t k = 0; k < (uint32_t)kWarps; ++k) {
    l->before[i][k] = run;
    run += ((mask >> k) & 1u) ? l->sum[s][k] : 0u;
  }
}

// `lanes` lanes (this is number j of them) fetch plane gp with the 16-byte chunks around it; returns where it starts.
__device__ __forceinline__ uint8_t* fetch_plane(const Plan& pl, const uint8_t* src, uint64_t gp, uint8_t* to, uint32_t j, uint32_t lanes,
                                                bool mine) {
  const uint64_t start = gp * pl.plane_bytes, end = start + pl.plane_bytes, a0 = start & ~15ull, whole = pl.dense_bytes & ~15ull;
  if (mine)
    for (uint64_t o = a0 + 16u * j; o < end; o += 16u * lanes) {
      if (o < whole) {
        *reinterpret_cast<uint4*>(to + (o - a0)) = __ldg(reinterpret_cast<const uint4*>(src + o));
      } else {
        for (uint64_t i = o; i < pl.dense_bytes; i += 2) *reinterpret_cast<uint16_t*>(to + (i - a0)) = *reinterpret_cast<const uint16_t*>(src + i);
      }
    }
  return to + (start - a0);
}

// Exclusive prefix sum over the warp, `run` going on to what follows.
__device__ __forceinline__ uint32_t warp_excl(uint32_t v, uint32_t& run) {
  const uint32_t lane = threadIdx.x & 31u, full = 0xFFFFFFFFu;
  uint32_t incl = v;
#pragma unroll
  for (uint32_t o = 1; o < 32u; o <<= 1) {
    const uint32_t up = __shfl_up_sync(full, incl, o);
    if (lane >= o) incl += up;
  }
  const uint32_t r = run + incl - v;
  run += __shfl_sync(full, incl, 31);
  return r;
}

// Phase 2, a warp: the small outlier-rich planes of one slice of a tile, whose overflow parts start `at` units into the region.
// `mk`: the table marker of the slice's plane `lane`; `staged`: where the tile still lies (null: nowhere, the planes are fetched
// again into `buf`).  Returns the slice's units.
template <int DT, int TT>
__device__ __forceinline__ uint4 slice_marker(BlockCtl* c, uint32_t tile, uint32_t slice) {
  const Plan& pl = c->pl;
  const uint32_t lane = threadIdx.x & 31u, lp = slice * (32u / TT) + lane;
  const uint64_t gp = (uint64_t)tile * pl.ppt + lp;
  return lane < 32u / TT && lp < pl.ppt && gp < pl.P ? __ldcg(reinterpret_cast<const uint4*>(c->d.dst + 64) + gp) : make_uint4(0u, 0u, 0u, 0u);
}
template <int DT, int TT>
__device__ __noinline__ uint32_t warp_slice_write(BlockCtl* c, uint32_t tile, uint32_t slice, const uint4 mk, uint32_t at, uint8_t* staged,
                                                  uint8_t* buf) {
  const Plan& pl = c->pl;
  const Dest& d = c->d;
  const uint32_t lane = threadIdx.x & 31u, full = 0xFFFFFFFFu, lp0 = slice * (32u / TT);
  const uint64_t p0 = (uint64_t)tile * pl.ppt;
  const uint32_t pb = (uint32_t)pl.plane_bytes;
  const uint32_t planes = __ballot_sync(full, (mk.y & 3u) != kClsNormal), n = __popc(planes);
  if (n == 0u) return 0u;
  uint32_t end = at;
  const uint32_t place = warp_excl((mk.y & 3u) != kClsNormal ? mk.x : 0u, end);  // (of the lane's plane)
  // as many planes at a time as have room in the buffer (at least four: a quarter of a stage), eight lanes or all to one
  const uint32_t lanes = pl.nblk == 1u ? 8u : 32u, step = pl.nblk == 1u ? 4u : 1u, room = a16(pb + 16u);
  for (uint32_t k0 = 0; k0 < n; k0 += step) {
    const uint32_t here = min(step, n - k0), k = k0 + lane / lanes, j = lane & (lanes - 1u);
    const bool mine = lane / lanes < here;
    const uint32_t b = nth_bit(planes, mine ? k : k0);
    const uint64_t gp = p0 + lp0 + b;
    uint32_t w = __shfl_sync(full, mk.w, (int)b);
    const uint32_t bytes = __shfl_sync(full, mk.z, (int)b), meta = __shfl_sync(full, mk.y, (int)b),
                   units = __shfl_sync(full, mk.x, (int)b), off = __shfl_sync(full, place, (int)b);
    uint8_t* plane;
    if (staged) {
      plane = staged + (uint64_t)(lp0 + b) * pb;
    } else {
      auto at_buf = [&](uint32_t i) { return buf + i * room + ((uint32_t)((p0 + lp0 + nth_bit(planes, k0 + i)) * pb) & 15u); };
      plane = fetch_plane(pl, c->a.src, gp, buf + (lane / lanes) * room, j, lanes, mine);
      __syncwarp();
      encode_small<DT>(pl, here, at_buf, [](uint32_t, uint32_t, bool) {});
      __syncwarp();
    }
    const unsigned long long off16 = (pl.ovf_off >> 4) + off;
    if (mine && (off16 + units) * 16ull <= d.capacity) {  // (never write past the capacity)
      SplitOut out;
      out.slot = d.dst + pl.slots_off + gp * pl.npay;
      out.ovf = d.dst + off16 * 16ull;
      out.npay = pl.npay;
      payload_copy(w ? plane : small_payload(plane), bytes, out, j, lanes);
      if (j == 0u)
        reinterpret_cast<uint4*>(d.dst + 64)[gp] = make_uint4(units ? (uint32_t)off16 : 0u, (w ? kClsRaw : kClsSalient) | (meta & ~3u), 0u, 0u);
    }
    __syncwarp();
  }
  return end - at;
}

// Phase 2, a warp: an outlier-rich plane of more than four blocks, whose overflow part starts `place` units into the region.
// `plane`: where it still lies, or null.
template <int DT>
__device__ __noinline__ void warp_plane_write(BlockCtl* c, uint64_t gp, const uint8_t* plane, uint32_t meta, uint32_t place, uint8_t* buf,
                                              uint32_t* sal) {
  const Plan& pl = c->pl;
  const Team team = make_warp_team(nullptr);
  if (!plane) plane = fetch_plane(pl, c->a.src, gp, buf, team.lane, 32u, true);
  __syncwarp();
  const SalientInfo info = scratch_saved<false>(pl) ? scratch_load<false>(team, pl, c->d, gp, sal) : salient_measure<DT, false>(team, pl, plane, sal);
  __syncwarp();
  write_blockwise<DT, false>(team, pl, c->d, gp, plane, info, sal, meta >> 2, place);
  __syncwarp();
}

// Phase 2, a warp: takes one of the tiles that were not listed, and its place; kNoTile when there are none left.
static __device__ __noinline__ uint32_t warp_take_linked(BlockCtl* c, uint32_t& place) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t tile = kNoTile;
  if (lane == 0)
    for (tile = *(volatile uint32_t*)&c->head; tile != kNoTile;) {
      const uint32_t seen = atomicCAS(&c->head, tile, c->a.defer_next[tile]);
      if (seen == tile) {
        c->a.defer_next[tile] = 0u;
        break;
      }
      tile = seen;
    }
  tile = __shfl_sync(0xFFFFFFFFu, tile, 0);
  place = 0;
  if (tile == kNoTile || scan_prefix(c->a.scan, tile, place)) return tile;
  if (lane == 0) report_error(c->a, kErrTimeout);
  return kNoTile;
}

// Phase 2, one warp: the places of the n listed tiles that have overflow (kNoTile: not to be had; units are below 2^32 - 1).
static __device__ __noinline__ void warp_list_places(BlockCtl* c, WarpList* l, uint32_t n) {
  const uint32_t lane = threadIdx.x & 31u;
  const bool asks = lane < n && l->units[min(lane, kListed - 1u)] != 0u;
  const uint32_t m = __ballot_sync(0xFFFFFFFFu, asks), want = __popc(m);
  if (lane < n && !asks) l->base[lane] = 0u;
  if (want == 0u) return;
  const uint32_t from = lane < want ? nth_bit(m, lane) : nth_bit(m, 0u);
  uint32_t base = 0;
  const bool ok = want == 1u ? scan_prefix(c->a.scan, l->tile[from], base) : scan_places(c->a.scan, l->tile[from], want, base);
  if (!ok && lane == 0) report_error(c->a, kErrTimeout);
  if (lane < want) l->base[from] = ok ? base : kNoTile;
}

// Phase 2 of the warp-team kernel, small planes.  The places of the listed tiles are looked up first: by one warp for all of them or,
// when a CTA has at most two tiles, a warp to a tile.  (us a call, by one / a warp to a tile / as they are.  By one the last place
// comes later: fp32, 170 x 513 planes of 22 x 2 45 / 41 / 40, 200 x 512 of 7 x 7 40 / 35 / 34, 64 x 256 of 14 x 14 18.1 / 17.1 / 17.0.  When there
// are many, more warps that poll hold up the publications they wait for: bf16, every eighth channel outlier-rich, 128 x 960 of 7 x 7 39 /
// 44 / 38, 128 x 384 of 14 x 14 45 / 53 / 47.  Every warp for itself: 7 x 7 planes, fp32: 25 -> 45.)
// Then every warp copies the payloads of the slices it has encoded, of tiles that still lie in a
// stage: the last ones the CTA streamed, all of them when the tensor is small.  The other tiles, if there are any, are handed out
// slice by slice; their planes are fetched and encoded again, in the stages, a part to a warp.
template <int DT, int TT>
__device__ __noinline__ void warp_phase2_small(BlockCtl* c, WarpList* l, uint8_t* stages) {
  const Plan& pl = c->pl;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, full = 0xFFFFFFFFu, n = min(l->count, kListed);
  uint8_t* buf = stages + min(warp, (uint32_t)kWarps - 1u) * ((pl.sm_sal / (uint32_t)kWarps) & ~15u);
  // (the warp's slice of a tile, as in phase 1; the first one's markers are on their way while the places are looked up)
  uint4 ahead = make_uint4(0u, 0u, 0u, 0u);
  if (warp < (uint32_t)kWarps) ahead = slice_marker<DT, TT>(c, l->tile[0], warp_slice(l->tile[0]));
  if (pl.ntiles > 2u * gridDim.x) {
    if (warp == (uint32_t)kWarps) warp_list_places(c, l, n);
  } else {
    for (uint32_t i = (uint32_t)kWarps - warp; i < n; i += (uint32_t)kWarps + 1u) {
      uint32_t base = 0;
      const bool ok = l->units[i] == 0u || scan_prefix(c->a.scan, l->tile[i], base);
      if (!ok && lane == 0) report_error(c->a, kErrTimeout);
      if (lane == 0) l->base[i] = ok ? base : kNoTile;  // (units are below 2^32 - 1)
    }
  }
  const bool away = threadIdx.x < n && c->held[l->stage[min(threadIdx.x, kListed - 1u)]] != l->tile[min(threadIdx.x, kListed - 1u)];
  const bool others = __syncthreads_or(away || c->head != kNoTile) != 0;  // (the places are known)
  if (warp < (uint32_t)kWarps)
    for (uint32_t i = 0; i < n; ++i) {
      const uint32_t tile = l->tile[i], slice = warp_slice(tile), st = l->stage[i];
      if (c->held[st] != tile || !((l->slices[i] >> slice) & 1u) || l->base[i] == kNoTile) continue;
      const uint4 mk = i ? slice_marker<DT, TT>(c, tile, slice) : ahead;
      warp_slice_write<DT, TT>(c, tile, slice, mk, l->base[i] + l->before[i][slice], stages + (uint64_t)st * pl.stage_bytes, buf);
    }
  if (!others) return;
  __syncthreads();  // the stages are free
  if (warp == (uint32_t)kWarps) return;
  for (;;) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(&l->handed[0], 1u);
    item = __shfl_sync(full, item, 0);
    if (item >= n * (uint32_t)kWarps) break;
    const uint32_t i = item / (uint32_t)kWarps, slice = item % (uint32_t)kWarps, tile = l->tile[i];
    if (c->held[l->stage[i]] == tile || !((l->slices[i] >> slice) & 1u) || l->base[i] == kNoTile) continue;
    warp_slice_write<DT, TT>(c, tile, slice, slice_marker<DT, TT>(c, tile, slice), l->base[i] + l->before[i][slice], nullptr, buf);
  }
  uint32_t at;
  for (uint32_t tile; (tile = warp_take_linked(c, at)) != kNoTile;)
    for (uint32_t slice = 0; slice < (uint32_t)kWarps; ++slice)
      at += warp_slice_write<DT, TT>(c, tile, slice, slice_marker<DT, TT>(c, tile, slice), at, nullptr, buf);
}

// Measuring a plane of more than four blocks is a chain of 10,000 to 30,000 cycles in one warp.  A warp that does it where the
// plane is found holds up its tile's stage, and with it the ring: so the planes that a CTA finds are listed, and measured by all
// its warps side by side when it has run out of tiles; only then are their tiles published.  (A CTA that waits for a tile's
// publication waits for one that is doing this or is still streaming; neither waits for anybody.)  Each warp keeps what it
// measured last, and phase 2 has it write that plane without measuring it again.  Planes that still lie in their stages are taken
// there when all do; otherwise all are fetched, into the stages, a part to a warp.  us a call, measured where they are found / so: bf16,
// 2 bits, 128 x 192 planes of 28 x 28, every eighth channel outlier-rich 91 / 71, 66,666 x 3 of 54 x 1, 13 % outlier-rich, 136 / 102; Huffman
// stage, fp32, 8 x 512 of 7 x 7, 14 % outlier-rich, 95 / 26, 8 x 128 of 28 x 28 55 / 36.
struct WarpOwn {
  uint32_t tile, lp;  // tile: kNoTile if there is none
  const uint8_t* plane;
  SalientInfo info;
};
template <int DT>
__device__ __noinline__ void warp_measure_put_off(BlockCtl* c, WarpList* l, uint8_t* stages, uint8_t* buf, uint32_t* sal, WarpOwn& own) {
  const Plan& pl = c->pl;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, full = 0xFFFFFFFFu;
  const uint32_t n = min(l->planes, kListedPlanes), tiles = min(l->count, kListed), mine = min(threadIdx.x, tiles - 1u);
  const Team team = make_warp_team(nullptr);
  if (n == 0u) return;
  const bool held = __syncthreads_and(c->held[l->stage[mine]] == l->tile[mine]) != 0;
  while (warp < (uint32_t)kWarps) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(&l->handed[0], 1u);
    item = __shfl_sync(full, item, 0);
    if (item >= n) break;
    const uint32_t i = l->of[item];
    if (i == kListed) continue;
    const uint32_t tile = l->tile[i], lp = l->lp[item];
    const uint64_t gp = (uint64_t)tile * pl.ppt + lp;
    const uint8_t* plane = held ? stages + (uint64_t)l->stage[i] * pl.stage_bytes + (uint64_t)lp * pl.plane_bytes
                                : fetch_plane(pl, c->a.src, gp, buf, lane, 32u, true);
    __syncwarp();
    const SalientInfo info = salient_measure<DT, false>(team, pl, plane, sal);
    bool raw;
    const uint32_t u = plane_units(pl, info, raw);
    if (lane == 0) {
      if (c->d.fits) store_marker(c->d, gp, l->meta[item], u);
      atomicAdd(&l->units[i], u);
      atomicAdd(&l->n[i], 1u);
      count_blockwise(u, raw ? 0u : 1u, raw ? 1u : 0u);
    }
    if (c->d.fits && scratch_saved<false>(pl)) scratch_save<false>(team, pl, c->d, gp, info, sal);
    own.tile = tile;
    own.lp = lp;
    own.plane = plane;
    own.info = info;
    __syncwarp();
  }
  __syncthreads();
  if (threadIdx.x < tiles && l->slices[threadIdx.x]) scan_publish(c->a.scan, l->tile[threadIdx.x], l->units[threadIdx.x]);
  if (threadIdx.x < (uint32_t)kMaxStages && !held) c->held[threadIdx.x] = kNoTile;
  if (threadIdx.x == 0) l->planes = l->handed[0] = 0;
  __syncthreads();
}

// Phase 2 of the warp-team kernel, planes of more than four blocks.  The places of the listed tiles first, by one warp; then their
// planes go to the warps one by one, each warp's own first; then the tiles that were not listed, a warp each.
template <int DT>
__device__ __noinline__ void warp_phase2_large(BlockCtl* c, WarpList* l, uint8_t* stages, uint8_t* sal_base) {
  const Plan& pl = c->pl;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, full = 0xFFFFFFFFu;
  uint32_t* sal = reinterpret_cast<uint32_t*>(sal_base + min(warp, (uint32_t)kWarps - 1u) * pl.sal_stride);
  uint8_t* buf = stages + min(warp, (uint32_t)kWarps - 1u) * ((pl.sm_sal / (uint32_t)kWarps) & ~15u);
  WarpOwn own;
  own.tile = kNoTile;
  warp_measure_put_off<DT>(c, l, stages, buf, sal, own);
  if (!c->d.fits) return;
  const uint32_t n = min(l->count, kListed);
  if (warp == (uint32_t)kWarps) warp_list_places(c, l, n);
  __syncthreads();
  for (uint32_t i = warp; i < n; i += (uint32_t)kWarps + 1u) {
    const uint32_t tile = l->tile[i], base = l->base[i];
    if (base == kNoTile) continue;
    // the tile's planes join the list; without room there, the tile joins the others
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(&l->planes, l->n[i]);
    at = __shfl_sync(full, at, 0);
    if (at + l->n[i] > kListedPlanes) {
      for (uint32_t k = at + lane; k < kListedPlanes; k += 32u) l->of[k] = (uint8_t)kListed;
      if (lane == 0) c->a.defer_next[tile] = atomicExch(&c->head, tile);
      continue;
    }
    const uint64_t p0 = (uint64_t)tile * pl.ppt;
    const uint32_t np = (uint32_t)min((uint64_t)pl.ppt, pl.P - p0);
    for (uint32_t lp0 = 0, run = base; lp0 < np; lp0 += 32u) {
      const uint2 mk = lp0 + lane < np ? load_marker(c->d, p0 + lp0 + lane) : make_uint2(0u, 0u);
      const bool mine = (mk.y & 3u) != kClsNormal;
      const uint32_t m = __ballot_sync(full, mine), place = warp_excl(mine ? mk.x : 0u, run);
      if (mine) {
        const uint32_t k = at + __popc(m & ((1u << lane) - 1u));
        l->place[k] = place;
        l->meta[k] = mk.y;
        l->lp[k] = (uint16_t)(lp0 + lane);
        l->of[k] = (uint8_t)i;
      }
      at += __popc(m);
    }
  }
  __syncthreads();  // the list is complete
  const uint32_t planes = min(l->planes, kListedPlanes);
  uint32_t own_place = kNoTile, own_meta = 0;
  for (uint32_t k0 = 0; own.tile != kNoTile && own_place == kNoTile && k0 < planes; k0 += 32u) {  // the warp's own plane leaves it
    const uint32_t k = min(k0 + lane, planes - 1u), i = l->of[k];
    const uint32_t m = __ballot_sync(full, i < kListed && l->tile[min(i, kListed - 1u)] == own.tile && l->lp[k] == own.lp);
    if (m == 0u) continue;
    const uint32_t at = k0 + (uint32_t)__ffs((int)m) - 1u;
    own_place = l->place[at];
    own_meta = l->meta[at];
    __syncwarp();
    if (lane == 0) l->of[at] = (uint8_t)kListed;
  }
  const bool away = threadIdx.x < n && c->held[l->stage[min(threadIdx.x, kListed - 1u)]] != l->tile[min(threadIdx.x, kListed - 1u)];
  const bool others = __syncthreads_or(away || c->head != kNoTile) != 0;
  if (own_place != kNoTile) {
    write_blockwise<DT, false>(make_warp_team(nullptr), pl, c->d, (uint64_t)own.tile * pl.ppt + own.lp, own.plane, own.info, sal, own_meta >> 2,
                               own_place);
    __syncwarp();
  }
  // planes that lie in stages, then those that are fetched into them (where planes have been put off, one or the other: see above)
  for (uint32_t pass = 0; pass < (others ? 2u : 1u); ++pass) {
    if (pass) __syncthreads();  // the stages are free
    while (warp < (uint32_t)kWarps) {
      uint32_t item = 0;
      if (lane == 0) item = atomicAdd(&l->handed[pass], 1u);
      item = __shfl_sync(full, item, 0);
      if (item >= planes) break;
      const uint32_t i = l->of[item];
      if (i == kListed) continue;
      const uint32_t tile = l->tile[i], st = l->stage[i], lp = l->lp[item];
      const bool held = c->held[st] == tile;
      if (held != (pass == 0u)) continue;
      warp_plane_write<DT>(c, (uint64_t)tile * pl.ppt + lp, held ? stages + (uint64_t)st * pl.stage_bytes + (uint64_t)lp * pl.plane_bytes : nullptr,
                           l->meta[item], l->place[item], buf, sal);
    }
  }
  if (!others || warp == (uint32_t)kWarps) return;
  uint32_t at;
  for (uint32_t tile; (tile = warp_take_linked(c, at)) != kNoTile;) {
    const uint64_t p0 = (uint64_t)tile * pl.ppt;
    const uint32_t np = (uint32_t)min((uint64_t)pl.ppt, pl.P - p0);
    for (uint32_t lp0 = 0; lp0 < np; lp0 += 32u) {
      const uint2 mk = lp0 + lane < np ? load_marker(c->d, p0 + lp0 + lane) : make_uint2(0u, 0u);
      const uint32_t place = warp_excl((mk.y & 3u) != kClsNormal ? mk.x : 0u, at);
      for (uint32_t m = __ballot_sync(full, (mk.y & 3u) != kClsNormal); m; m &= m - 1u) {
        const uint32_t b = (uint32_t)__ffs((int)m) - 1u;
        warp_plane_write<DT>(c, p0 + lp0 + b, nullptr, __shfl_sync(full, mk.y, (int)b), __shfl_sync(full, place, (int)b), buf, sal);
      }
    }
  }
}

template <int DT, int SIGMA, int TT, int K, int EDGE>
__global__ void __launch_bounds__(kWarpKernelThreads, 3) compress_warp(const Plan pl, const CompressArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) uint64_t s_full[kMaxStages], s_empty[kMaxStages];
  __shared__ uint32_t s_tiles[kMaxStages];
  __shared__ volatile uint32_t s_abort;
  __shared__ uint32_t s_last;
  __shared__ BlockCtl s_ctl;
  __shared__ WarpList s_list;

  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t nstage = pl.nstage;
  const bool scan_on = pl.mode != kModeOff;
  uint32_t first_ticket = 0;
  // Everything that needs no global memory comes before the wait for the previous kernel, whose tail hides it.
  if (tid == 0) {
    for (uint32_t s = 0; s < nstage; ++s) {
      mbar_init(&s_full[s], 1);
      mbar_init(&s_empty[s], kWarps);
    }
    fence_mbar_init();
    s_abort = 0;
    *cta_totals() = CtaTotals{0u, 0u, 0u, 0u};
    if (scan_on) {
      s_ctl.pl = pl;
      s_ctl.a = a;
      s_ctl.head = kNoTile;
      for (uint32_t s = 0; s < nstage; ++s) {
        s_ctl.U[s] = s_ctl.C[s] = s_ctl.arr[s] = 0;
        s_ctl.held[s] = kNoTile;
        s_list.mask[s] = 0;
        s_list.entry[s] = kNoEntry;
      }
      s_list.count = s_list.planes = s_list.handed[0] = s_list.handed[1] = 0;
    }
  }
  // (the ticket counter of this call was returned to zero by the call before the previous one, which had
  // completed before the previous kernel let this one start)
  if (tid == (uint32_t)kThreads && a.early_ticket)
    first_ticket = (uint32_t)atomicAdd(&a.sc->ticket[a.parity], (unsigned long long)pl.first_req);
  __syncthreads();
  if (warp < (uint32_t)kWarps || !a.early_load) {  // (the producer only reads the input and takes tickets: see dep_wait)
    dep_wait();     // the previous kernel on the stream has completed; global memory may be touched from here on
    dep_trigger();  // the next kernel on the stream may become resident as this one drains
  }
  // (the sweeps only need the first and the last of these: the others wait in shared memory, not in registers)
  Dest d = {};
  if (warp < (uint32_t)kWarps) {  // (the producer goes straight to its first loads)
    const Dest all = make_dest(pl, a);
    d.dst = all.dst;
    d.fits = all.fits;
    if (tid == 0) {
      if (!d.fits && blockIdx.x == 0) report_error(a, kErrCapacity);
      s_ctl.d = all;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");  // the consumer warps: s_ctl.d is in place
  }

  if (warp == (uint32_t)kWarps) {
    // ======================= producer (all 32 lanes walk the loop, lane 0 issues) =======================
    uint32_t s = 0, empty_phase = 0;
    bool aborted = false;
    if (!a.early_ticket && lane == 0)
      first_ticket = (uint32_t)atomicAdd(&a.sc->ticket[a.parity], (unsigned long long)pl.first_req);
    first_ticket = __shfl_sync(0xFFFFFFFFu, first_ticket, 0);
    // Waits until every consumer warp is done with the tile in stage q.
    auto drain = [&](uint32_t q) -> bool {
      bool ok = mbar_wait_abortable(&s_empty[q], (empty_phase >> q) & 1u, 1u << 20, &s_abort);
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (ok) empty_phase ^= 1u << q;
      return ok;
    };
    // Tensors of no more tiles than the grid has stages: every CTA takes as many as its first request is for, those of the lowest
    // numbers -- one to an SM -- one more, and nobody asks whether there is another: the answer took a microsecond that the
    // CTA's last sweep did not hide (fp32, us a call among others, with the question / without: 32 x 16 planes of 32 x 32 5.6 / 5.2,
    // 128 of 28 x 28 5.0 / 4.4, 16 x 64 of 14 x 14 5.5 / 5.0; nothing where the host takes longer to call).
    // (Tickets are still handed out in order: the tiles before a CTA's are with CTAs that run.)
    const uint32_t rest = pl.ntiles - min(pl.ntiles, pl.first_req * gridDim.x);
    const uint32_t most = pl.ntiles <= nstage * gridDim.x ? pl.first_req + (blockIdx.x < rest ? 1u : 0u) : 0xFFFFFFFFu;
    for (uint32_t n = 0;; ++n) {
      if (n >= nstage && !drain(s)) {
        aborted = true;
        break;
      }
      // tiles come in ticket order: the first of them in one request, then one at a time.  The tiles that are left of a small
      // tensor when every CTA has its first go to the CTAs of the lowest numbers -- one to an SM -- as soon as their first
      // load has arrived, so that the second is on its way while the first is swept (14 x 14, fp32, 512 tiles: 11.2 ->
      // 9.9 us; whoever came first took them at first, three to an SM, which cost as much as it gave when the sweep is long).
      uint32_t t = n < most ? first_ticket + n : kNoTile;
      if (n >= pl.first_req && n < most) {
        if (n < nstage) {
          const uint64_t given = (uint64_t)n * gridDim.x;
          const bool soon = given < pl.ntiles && blockIdx.x < pl.ntiles - given;
          bool here = soon ? mbar_wait_abortable(&s_full[s - 1u], 0u, 1u << 20, &s_abort)
                           : mbar_wait_abortable(&s_empty[s - 1u], 0u, 1u << 20, &s_abort);
          here = __all_sync(0xFFFFFFFFu, here);
          if (!here) {
            aborted = true;
            break;
          }
        }
        if (lane == 0) t = (uint32_t)atomicAdd(&a.sc->ticket[a.parity], 1ull);
        t = __shfl_sync(0xFFFFFFFFu, t, 0);
      }
      if (t >= pl.ntiles) {
        // no more tiles: wake the consumers at this stage, then wait for the tiles still in the ring
        const uint32_t first = n >= nstage ? n - nstage + 1u : 0u;
        uint32_t q = first % nstage;
        __syncwarp();
        if (lane == 0) {
          s_tiles[s] = kNoTile;
          mbar_arrive(&s_full[s]);
        }
        for (uint32_t m = first; m < n; ++m) {
          if (!drain(q)) {
            aborted = true;
            break;
          }
          q = q + 1 == nstage ? 0 : q + 1;
        }
        break;
      }
      if (lane == 0) {
        s_tiles[s] = t;
        if (scan_on) s_ctl.held[s] = t;
        const uint32_t p0 = t * pl.ppt;
        const uint32_t np = (uint32_t)min((uint64_t)pl.ppt, pl.P - p0);
        const uint32_t bytes = np * (uint32_t)pl.plane_bytes;
        uint8_t* stage = smem + pl.sm_tile + (uint64_t)s * pl.stage_bytes;
        // whole 16-byte chunks by bulk copy; what is left of the tensor's last tile by this thread, ahead of its arrival
        const uint32_t whole = bytes & ~15u;
        const uint8_t* from = a.src + (uint64_t)p0 * pl.plane_bytes;
        for (uint32_t i = whole; i < bytes; i += 2u) *reinterpret_cast<uint16_t*>(stage + i) = *reinterpret_cast<const uint16_t*>(from + i);
        if (whole) {
          fence_proxy_async();
          mbar_expect_tx(&s_full[s], whole);
          bulk_g2s(stage, from, whole, &s_full[s]);
        } else {
          mbar_arrive(&s_full[s]);
        }
      }
      __syncwarp();
      s = s + 1 == nstage ? 0 : s + 1;
    }
    if (aborted) {  // wait (bounded) for copies still in flight before the CTA may exit
      s_abort = 1;
      if (lane == 0) {
        report_error(a, kErrTimeout);
        for (uint32_t k = 0; k < nstage; ++k) {
          mbar_wait(&s_full[k], 0u, 1u << 10);
          mbar_wait(&s_full[k], 1u, 1u << 10);
        }
      }
    }
  } else {
    // ======================= consumers =======================
    const uint32_t grain = plane_grain(pl);
    uint32_t rp = 0, s = 0, phase = 0;
    for (;;) {
      const uint32_t par = (phase >> s) & 1u;
      bool ok = mbar_wait_abortable(&s_full[s], par, 1u << 20, &s_abort);
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (!ok) {
        s_abort = 1;
        break;
      }
      phase ^= 1u << s;
      const uint32_t tile = s_tiles[s];
      if (tile >= pl.ntiles) break;
      const uint32_t p0 = tile * pl.ppt;
      const uint32_t np = (uint32_t)min((uint64_t)pl.ppt, pl.P - p0);
      // (what follows from the lane's number is worked out anew for each tile: kept in registers, it takes those of the sweep)
      uint32_t me = lane;
      asm volatile("" : "+r"(me));
      Team team;
      team.size = TT;
      team.lane = me & (TT - 1u);
      team.mask = TT == 32 ? 0xFFFFFFFFu : ((1u << (TT & 31)) - 1u) << (me & ~(TT - 1u));
      team.block = false;
      team.nwarps = 0;
      team.red = nullptr;
      const uint32_t slice = warp_slice(tile);
      const uint32_t lp = slice * (32u / TT) + me / TT, at = min(lp, np - 1u);
      const bool active = lp < np;
      uint8_t* stage = smem + pl.sm_tile + (uint64_t)s * pl.stage_bytes;
      const uint32_t meta = plane_sweep<DT, SIGMA, K, TT, EDGE>(team, pl, d, a, stage + (uint64_t)at * pl.plane_bytes,
                                                                (uint64_t)p0 + at, grain, active, rp);
      if (scan_on) {  // phase 1 of the block-wise path
        const uint32_t leaders = __ballot_sync(0xFFFFFFFFu, active && (meta & 3u) != kClsNormal && team.lane == 0);
        // (planes of teams of sixteen lanes and more have more than four blocks)
        if (leaders) {
          if (TT <= 8 && is_small_plane(pl)) warp_tile_encode<DT, (TT <= 8 ? TT : 8)>(&s_ctl, &s_list, stage, s, leaders, meta);
          else
            warp_tile_put_off<DT, TT>(&s_ctl, &s_list, stage, s, leaders, meta, smem + pl.sm_sal);
        }
        if (lane == 0) {
          if (leaders) __threadfence_block();  // the warp's sums before its arrival
          if ((atomicAdd(&s_ctl.arr[s], 1u) & 7u) == 7u) {  // the last of the tile's eight warps: its sums are complete
            __threadfence_block();                          // (the other warps' after their arrivals)
            if (*(volatile uint32_t*)&s_ctl.C[s] == 0u) scan_publish(a.scan, tile, 0u);
            else warp_tile_publish(&s_ctl, &s_list, s, tile);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&s_empty[s]);
      if (s_abort) break;
      s = s + 1 == nstage ? 0 : s + 1;
    }
  }
  if (scan_on) {
    __syncthreads();
    if (s_list.count != 0u && !s_abort) {
      if (TT <= 8 && is_small_plane(pl)) warp_phase2_small<DT, (TT <= 8 ? TT : 8)>(&s_ctl, &s_list, smem + pl.sm_tile);
      else warp_phase2_large<DT>(&s_ctl, &s_list, smem + pl.sm_tile, smem + pl.sm_sal);
    }
  }
  cta_exit(pl, a, s_ctl.d, &s_last);
}

// -------------------------------------------------------------------------------------------------
// CTA-team kernel: bf16 planes beyond the register variant's reach, of whole 16-byte chunks (of such a plane in fp32 two
// stages do not fit).  One plane per tile, all threads of the CTA work on it.  The plane stays in its shared-memory stage
// and is swept two or three times (min/max; integer moments; count + codes), so that few registers are needed.
// A warp has at most 892 groups, whose integer sums fit 32 bits.  Thread 0 keeps the next ticket in flight while the CTA works.
// An outlier-rich plane is measured by the whole CTA while it lies in its stage and written in phase 2.
// -------------------------------------------------------------------------------------------------
// Phase 1: the plane in `plane` is measured, tile (= plane) `tile` published.  Ends with a barrier.
template <int DT, bool PARTS>
__device__ __noinline__ void cta_tile_measure(BlockCtl* c, double* red, const uint8_t* plane, uint32_t* sal, uint32_t tile,
                                              uint32_t meta) {
  const Team team = make_cta_team(blockDim.x, red);
  const SalientInfo info = salient_measure<DT, PARTS>(team, c->pl, plane, sal);
  if (threadIdx.x == 0) {
    bool raw;
    const uint32_t units = plane_units(c->pl, info, raw);
    scan_publish(c->a.scan, tile, units);
    count_blockwise(units, raw ? 0u : 1u, raw ? 1u : 0u);
    if (c->d.fits) store_marker(c->d, tile, meta, units);
  }
  if (c->d.fits && scratch_saved<PARTS>(c->pl)) scratch_save<PARTS>(team, c->pl, c->d, tile, info, sal);
  if (threadIdx.x == 0) c->own_info = info;
  __syncthreads();
}

// The queue of planes put off (CTA-team kernels).  Which CTA has measured how many outlier-rich planes is a matter of
// chance -- none to twice the mean --, so phase 2 deals them out anew: with every CTA writing its own, the bf16 112 x 112
// tensor with every eighth channel outlier-rich spent 168 to 335 us of 338 in phase 2, depending on the CTA.
// A CTA that has claimed an entry that is not there yet waits for it until no CTA can queue another plane.  Those that can
// are CTAs that have started, as the ticket word counts them along with its tickets: whoever starts once the tickets are
// used up gets no tile.  It must not wait for CTAs that have not started, which may find no room while it stays (kernels on
// other streams hold the rest of the GPU).  Leaving at once when the queue is empty, instead of waiting, left the last planes
// to the CTAs that had measured them: 128 x 144 bf16 planes of 56 x 56, 125 -> 141 us.
//
// One thread, behind a barrier that follows the measuring: plane `tile`, of `stage`, is put off.  `held`: no other plane
// will be loaded there.
constexpr unsigned long long kStarted = 1ull << 32;  // added to the ticket word with a CTA's first request
static __device__ __noinline__ void queue_push(BlockCtl* c, uint32_t tile, uint32_t stage, bool held) {
  if (!c->d.fits) return;
  // the CTA keeps its last plane, whose scratch lies ready; the one before joins the queue
  const uint32_t before = c->own;
  c->own = tile;
  c->own_stage = stage;
  c->own_held = held;
  if (before == kNoTile) return;
  const uint32_t n = (uint32_t)(atomicAdd(&c->a.sc->queue, 1ull << 32) >> 32);
  __threadfence();  // marker and saved scratch, of all threads, before the entry
  st_relaxed32(&c->a.defer_next[n], before + 1u);
}
constexpr uint32_t kPending = 0xFFFFFFFEu;
// One thread: the plane of queue entry n, which is this CTA's; kNoTile when there will be none -- every CTA that has started
// has finished phase 1 and the queue is shorter --, kPending (unless `wait`) when it is not known yet.  A CTA in phase 1 waits
// for nobody, so the wait ends; it is bounded all the same.
static __device__ __noinline__ uint32_t queue_entry(BlockCtl* c, uint32_t n, bool wait) {
  const CompressArgs& a = c->a;
  if (n >= c->pl.ntiles) return kNoTile;
  for (uint32_t k = 0; k < a.scan.polls; ++k) {
    uint32_t e = ld_relaxed32(&a.defer_next[n]);
    if (!e && wait) {
      const unsigned long long left = ld_relaxed(&a.sc->exited), in2 = ld_relaxed(&a.sc->done);
      __threadfence();  // (those that have finished before those that have started: the latter can only be more)
      const uint32_t quiet = ((uint32_t)left & kExitMask) - ((uint32_t)(left >> kExitBits) & kExitMask);  // left with nothing
      const uint32_t started = (uint32_t)(ld_relaxed(&a.sc->ticket[a.parity]) / kStarted);
      if (quiet + (uint32_t)in2 == started && n >= (uint32_t)(ld_relaxed(&a.sc->queue) >> 32)) return kNoTile;
      e = ld_relaxed32(&a.defer_next[n]);
    }
    if (e) {
      st_relaxed32(&a.defer_next[n], 0u);
      __threadfence();
      return e - 1u;
    }
    if (!wait) return kPending;
    __nanosleep(200);
  }
  report_error(a, kErrTimeout);
  return kNoTile;
}

// All threads of the CTA start to copy plane gp with the 16-byte chunks around it; fetch_wait and a barrier end it.
__device__ __forceinline__ void fetch_start(const Plan& pl, const uint8_t* src, uint64_t gp, uint8_t* to) {
  const uint64_t start = gp * pl.plane_bytes, end = start + pl.plane_bytes, a0 = start & ~15ull;
  const uint64_t whole = min((end + 15ull) & ~15ull, pl.dense_bytes & ~15ull);
  for (uint64_t o = a0 + 16u * threadIdx.x; o < whole; o += 16u * blockDim.x)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(to + (o - a0))), "l"(src + o) : "memory");
  if (threadIdx.x == 0)
    for (uint64_t i = whole; i < end; i += 2) *reinterpret_cast<uint16_t*>(to + (i - a0)) = *reinterpret_cast<const uint16_t*>(src + i);
}
__device__ __forceinline__ void fetch_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Bulk load of plane `gp` with the 16-byte chunks around it (one thread); plane_head says where the plane starts in the
// stage.  The last bytes of a tensor that does not end on a 16-byte boundary are copied by the thread itself, ahead of
// its arrival at the barrier.
__device__ __forceinline__ uint32_t plane_head(const Plan& pl, uint64_t gp) { return (uint32_t)(gp * pl.plane_bytes) & 15u; }
__device__ __forceinline__ void plane_load(const Plan& pl, const uint8_t* src, uint64_t gp, uint8_t* stage, uint64_t* bar) {
  const uint64_t start = gp * pl.plane_bytes, a0 = start & ~15ull;
  const uint64_t whole = min((start + pl.plane_bytes + 15ull) & ~15ull, pl.dense_bytes & ~15ull);
  for (uint64_t i = whole; i < start + pl.plane_bytes; i += 2)
    *reinterpret_cast<uint16_t*>(stage + (i - a0)) = *reinterpret_cast<const uint16_t*>(src + i);
  fence_proxy_async();
  mbar_expect_tx(bar, (uint32_t)(whole - a0));
  bulk_g2s(stage, src + a0, (uint32_t)(whole - a0), bar);
}

// Phase 2 of the CTA-team kernels: the CTA's own plane, then planes from the queue until it is empty.  While one is written,
// the next is claimed and fetched into the other stage.
template <int DT, bool PARTS>
__device__ __noinline__ void cta_phase2(BlockCtl* c, double* red, uint8_t* stages, uint32_t* sal) {
  const Plan& pl = c->pl;
  const Team team = make_cta_team(blockDim.x, red);
  const uint32_t tid = threadIdx.x;
  const bool claims = tid == blockDim.x - 32u;  // (not in the warp that looks up places, where there are two)
  uint32_t mine = 0, cur = 0;
  auto claim = [&]() { mine = (uint32_t)atomicAdd(&c->a.sc->queue, 1ull); };
  if (claims) {
    __threadfence();  // the CTA's entries before the note that it has finished phase 1
    atomicAdd(&c->a.sc->done, 1ull);
    c->next = c->own;
  }
  bool kept = true;  // the plane in hand is the CTA's own: its scratch lies ready
  cur = c->own_stage;
  for (bool fetched = c->own_held != 0u;;) {
    __syncthreads();
    const uint32_t tile = c->next;
    if (tile >= pl.ntiles) break;  // (the same for every thread)
    uint8_t* stage = stages + (uint64_t)cur * pl.stage_bytes;
    if (!fetched) fetch_start(pl, c->a.src, tile, stage);
    if (claims) claim();
    const uint2 mk = load_marker(c->d, tile);  // units, class and count
    if (tid < 32u) {
      bool ok = true;
      uint32_t base = 0;
      if (mk.x) ok = scan_prefix(c->a.scan, tile, base);
      if (tid == 0) {
        if (!ok) report_error(c->a, kErrTimeout);
        c->base = base;
        c->ok = ok;
      }
    }
    SalientInfo info;
    const bool saved = scratch_saved<PARTS>(pl);
    if (kept) info = c->own_info;
    else if (saved) info = scratch_load<PARTS>(team, pl, c->d, tile, sal);
    if (claims) c->ahead = queue_entry(c, mine, false);
    fetch_wait();
    __syncthreads();
    const uint32_t ahead = c->ahead;
    const uint8_t* plane = stage + plane_head(pl, tile);
    fetched = ahead < pl.ntiles;
    if (fetched) fetch_start(pl, c->a.src, ahead, stages + (uint64_t)(cur ^ 1u) * pl.stage_bytes);
    if (!saved && !kept) info = salient_measure<DT, PARTS>(team, pl, plane, sal);
    kept = false;
    if (c->ok) write_blockwise<DT, PARTS>(team, pl, c->d, (uint64_t)tile, plane, info, sal, mk.y >> 2, c->base);
    if (claims) c->next = ahead == kPending ? queue_entry(c, mine, true) : ahead;
    fetch_wait();
    if (fetched) cur ^= 1u;
  }
}
// Behind phase 1 of a CTA-team kernel.
template <int DT, bool PARTS>
__device__ __forceinline__ void cta_finish(BlockCtl* c, double* red, uint8_t* stages, uint32_t* sal, bool aborted) {
  __syncthreads();
  if (c->own != kNoTile && !aborted) cta_phase2<DT, PARTS>(c, red, stages, sal);
  else if (threadIdx.x == 0 && has_totals(*cta_totals())) atomicAdd(&c->a.sc->done, 1ull);  // (see queue_entry)
}

__device__ __forceinline__ void lds_group(const uint8_t* plane, uint32_t g, float (&v)[4]) {
  const uint2 t2 = reinterpret_cast<const uint2*>(plane)[g];
  v[0] = __uint_as_float(t2.x << 16); v[1] = __uint_as_float(t2.x & 0xFFFF0000u);
  v[2] = __uint_as_float(t2.y << 16); v[3] = __uint_as_float(t2.y & 0xFFFF0000u);
}
// The group's distances from lo (x - lo is x + (-lo): the same rounding).
__device__ __forceinline__ void lds_dist(const uint8_t* plane, uint32_t g, float nlo, float (&v)[4]) {
  lds_group(plane, g, v);
  const f32x2 nlo2 = pack2(nlo, nlo);
  unpack2(add2(pack2(v[0], v[1]), nlo2), v[0], v[1]);
  unpack2(add2(pack2(v[2], v[3]), nlo2), v[2], v[3]);
}

#define FH_CTA_STORE_CODES(BITS)                                                                              \
  {                                                                                                           \
    constexpr uint32_t bias = kMagicBits * (1u + (1u << (BITS)) + (1u << (2 * (BITS))) + (1u << (3 * (BITS)))); \
    const f32x2 inv2 = pack2(inv, inv), mag2 = pack2(kMagicF, kMagicF);                                         \
    _Pragma("unroll 2") for (uint32_t g = tid; g < groups; g += NT) {                                         \
      float v[4];                                                                                             \
      lds_dist(plane, g, nlo, v);                                                                         \
      uint32_t w0, w1, w2, w3;                                                                                \
      unpack2u(fma2(pack2(v[0], v[1]), inv2, mag2), w0, w1);                                                  \
      unpack2u(fma2(pack2(v[2], v[3]), inv2, mag2), w2, w3);                                                  \
      uint32_t word = w0 + (w1 << (BITS)) + (w2 << (2 * (BITS))) + (w3 << (3 * (BITS))) - bias;               \
      if ((BITS) == 2) slot[g] = (uint8_t)word;                                                               \
      else if ((BITS) == 4) reinterpret_cast<uint16_t*>(slot)[g] = (uint16_t)word;                            \
      else reinterpret_cast<uint32_t*>(slot)[g] = word;                                                       \
      if (COUNT) {                                                                                            \
        if (one_sided) {                                                                                      \
          c0 += (v[0] > dhi) + (v[2] > dhi);                                                                  \
          c1 += (v[1] > dhi) + (v[3] > dhi);                                                                  \
        } else {                                                                                              \
          c0 += ((v[0] > dhi) || (v[0] < dlo)) + ((v[2] > dhi) || (v[2] < dlo));                              \
          c1 += ((v[1] > dhi) || (v[1] < dlo)) + ((v[3] > dhi) || (v[3] < dlo));                              \
        }                                                                                                     \
      }                                                                                                       \
    }                                                                                                         \
  }

constexpr int kSweepThreads = 512;

template <bool SIGMA>
__global__ void __launch_bounds__(kSweepThreads) compress_cta(const Plan pl, const CompressArgs a) {
  constexpr int DT = kBF16, NT = kSweepThreads;
  constexpr bool COUNT = SIGMA;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ double s_red[kMaxWarps * 4];
  __shared__ __align__(8) uint64_t s_full[kMaxStages];
  __shared__ uint32_t s_tiles[kMaxStages];
  __shared__ uint32_t s_abort, s_last;
  __shared__ float2 s_thr;
  __shared__ BlockCtl s_ctl;

  const uint32_t tid = threadIdx.x;
  const Team team = make_team(NT, s_red);
  const uint32_t nstage = pl.nstage, groups = pl.groups, bits = (uint32_t)pl.bits;
  const bool scan_on = pl.mode != kModeOff;
  uint32_t* sal = reinterpret_cast<uint32_t*>(smem + pl.sm_sal);
  uint32_t rp = 0;
  // Thread 0 requests the tiles and issues the loads: the first nstage tiles in one request, later ones one
  // at a time, the request running one tile ahead of its use.  Tiles come in ticket order.
  uint32_t next_ticket = 0, issued = 0;
  if (tid == 0) {
    for (uint32_t s = 0; s < nstage; ++s) mbar_init(&s_full[s], 1);
    fence_mbar_init();
    s_abort = 0;
    *cta_totals() = CtaTotals{0u, 0u, 0u, 0u};
    // (the ticket counter of this call was returned to zero by the call before the previous one, which had
    // completed before the previous kernel let this one start)
    if (a.early_ticket) next_ticket = (uint32_t)atomicAdd(&a.sc->ticket[a.parity], kStarted + nstage);
  }
  if (tid == 0 && scan_on) {  // (before the wait for the previous kernel, whose tail hides it)
    s_ctl.pl = pl;
    s_ctl.a = a;
    s_ctl.own = kNoTile;
  }
  dep_wait();     // the previous kernel on the stream has completed; global memory may be touched from here on
  dep_trigger();  // the next kernel on the stream may become resident as this one drains
  auto issue = [&](uint32_t s) {
    const uint32_t t = next_ticket;
    s_tiles[s] = t;
    if (t < pl.ntiles) {
      fence_proxy_async();
      mbar_expect_tx(&s_full[s], (uint32_t)pl.plane_bytes);
      bulk_g2s(smem + pl.sm_tile + (uint64_t)s * pl.stage_bytes, a.src + (uint64_t)t * pl.plane_bytes,
               (uint32_t)pl.plane_bytes, &s_full[s]);
      ++issued;
      next_ticket = issued < nstage ? t + 1u : (uint32_t)atomicAdd(&a.sc->ticket[a.parity], 1ull);
    }
  };
  if (tid == 0) {  // the first loads before anything else
    if (!a.early_ticket) next_ticket = (uint32_t)atomicAdd(&a.sc->ticket[a.parity], kStarted + nstage);
    for (uint32_t s = 0; s < nstage; ++s) issue(s);
  }
  const Dest d = make_dest(pl, a);
  if (tid == 0) {
    if (!d.fits && blockIdx.x == 0) report_error(a, kErrCapacity);
    if (scan_on) s_ctl.d = d;
  }
  __syncthreads();

  uint32_t s = 0, phase = 0;
  for (;;) {
    const uint32_t tile = s_tiles[s];
    if (tile >= pl.ntiles) break;
    bool ready = mbar_wait(&s_full[s], (phase >> s) & 1u, 1u << 20);
    ready = __all_sync(0xFFFFFFFFu, ready);
    phase ^= 1u << s;
    if (!ready) s_abort = 1;
    const uint8_t* plane = smem + pl.sm_tile + (uint64_t)s * pl.stage_bytes;
    const uint64_t gp = tile;

    // ---- sweep 1: minimum and maximum
    float lo = __int_as_float(0x7F800000), hi = __int_as_float(0xFF800000), lo1 = lo, hi1 = hi;
    if (ready) {
#pragma unroll 2
      for (uint32_t g = tid; g < groups; g += 2 * NT) {
        float v[4];
        lds_group(plane, g, v);
        lo = min_nan(lo, min_nan(min3_nan(v[0], v[1], v[2]), v[3]));
        hi = max_nan(hi, max_nan(max3_nan(v[0], v[1], v[2]), v[3]));
        if (g + NT < groups) {
          lds_group(plane, g + NT, v);
          lo1 = min_nan(lo1, min_nan(min3_nan(v[0], v[1], v[2]), v[3]));
          hi1 = max_nan(hi1, max_nan(max3_nan(v[0], v[1], v[2]), v[3]));
        }
      }
    }
    lo = min_nan(lo, lo1);
    hi = max_nan(hi, hi1);
    team_minmax(team, lo, hi, rp);  // one barrier: also tells every thread about an abort
    if (s_abort) break;
    const float range = __fsub_rn(hi, lo), nlo = -lo;
    if (!(fabsf(range) <= 3.402823466e38f) && tid == 0) report_error(a, kErrNonfinite);

    // ---- sweep 2: integer moments of the distances from lo, thresholds
    float dlo = 0.0f, dhi = 0.0f;
    bool one_sided = true, need_count = false;
    if (SIGMA) {
      const SigmaScale sc = sigma_scale(range);
      if (sc.applies) {  // (the same for every thread)
        uint32_t as = 0, aq = 0, ng = 0;
#pragma unroll 2
        for (uint32_t g = tid; g < groups; g += NT) {
          float v[4];
          lds_dist(plane, g, nlo, v);
          sigma_addends4(v[0], v[1], v[2], v[3], sc, as, aq);
          ++ng;
        }
        {  // the first warp adds up the warps' sums and works out what depends on them, for all
          int32_t pa = (int32_t)(as - ng * kMagicBits), pb = (int32_t)(aq - ng * kMagicBits);
          asm volatile("redux.sync.add.s32 %0, %0, %1;" : "+r"(pa) : "r"(0xFFFFFFFFu));
          asm volatile("redux.sync.add.s32 %0, %0, %1;" : "+r"(pb) : "r"(0xFFFFFFFFu));
          int2* r = reinterpret_cast<int2*>(red_half(team, rp));
          const uint32_t wl = tid & 31u;
          if (wl == 0) r[tid >> 5] = make_int2(pa, pb);
          __syncthreads();
          if (tid < 32u) {
            const int2 pr = wl < team.nwarps ? r[wl] : make_int2(0, 0);
            const long long Is = warp_sum_s32_wide(pr.x), Iq = warp_sum_s32_wide(pr.y);
            float tl, th;
            sigma_thresholds(Is, Iq, sc, pl.inv_hw, tl, th);
            if (tid == 0) s_thr = make_float2(tl, th);
          }
          __syncthreads();
          dlo = s_thr.x;
          dhi = s_thr.y;
        }
        need_count = range > dhi || 0.0f < dlo;  // otherwise no element can lie outside
        one_sided = !(0.0f < dlo);
      }
    }

    // ---- sweep 3: codes into the plane's slot (and the outlier count).  A plane that turns out
    // outlier-rich has its slot rewritten below.
    float inv, scale;
    quant_params(range, (1u << bits) - 1u, inv, scale);
    uint8_t* slot = d.dst + pl.slots_off + gp * pl.npay;
    uint32_t c0 = 0, c1 = 0;
    if (d.fits && pl.mode != kModeAll) {
      if (!need_count) {
        dhi = __int_as_float(0x7F800000);  // nothing is counted
        one_sided = true;
      }
      if (bits == 2u) FH_CTA_STORE_CODES(2)
      else if (bits == 4u) FH_CTA_STORE_CODES(4)
      else FH_CTA_STORE_CODES(8)
      const uint32_t code_bytes = groups * bits / 2u;
      for (uint32_t o = a4(code_bytes) + 4u * tid; o < pl.npay; o += 4u * NT) *reinterpret_cast<uint32_t*>(slot + o) = 0u;
      if (tid == 0)
        for (uint32_t o = code_bytes; o < a4(code_bytes); ++o) slot[o] = 0;
    } else if (SIGMA && need_count) {  // nothing may be stored: count only
      for (uint32_t g = tid; g < groups; g += NT) {
        float v[4];
        lds_dist(plane, g, nlo, v);
#pragma unroll
        for (int e = 0; e < 4; ++e) c0 += (v[e] > dhi) || (v[e] < dlo);
      }
    }
    uint32_t cls = kClsNormal, n_out = 0;
    if (SIGMA) {
      n_out = team_sum_u32(team, c0 + c1, rp);  // its barrier: every thread is done with the sweeps
      if ((uint64_t)n_out * pl.rho_den > (uint64_t)pl.rho_num * pl.HW) cls = kClsSalient;
    } else {
      if (pl.mode == kModeAll) cls = kClsSalient;
      if (pl.mode >= kModeChannel) cls = channel_class(pl, a, gp, n_out);
      __syncthreads();  // every thread is done with the sweeps
    }
    if (cls == kClsNormal) {
      if (tid == 0) {
        if (d.fits) store_table_entry(d, gp, (uint32_t)((pl.slots_off + gp * pl.npay) >> 4), cls | (n_out << 2), lo, scale);
        if (scan_on) scan_publish(a.scan, tile, 0u);
        issue(s);  // the stage is free: next load
      }
    } else {  // (the same for every thread) phase 1 of the block-wise path
      cta_tile_measure<DT, true>(&s_ctl, s_red, plane, sal, tile, cls | (n_out << 2));
      if (tid == 0) {
        issue(s);
        queue_push(&s_ctl, tile, s, s_tiles[s] >= pl.ntiles);
      }
    }
    s = s + 1 == nstage ? 0 : s + 1;
    // s_tiles[s] for the next iteration was written at least one barrier ago (nstage >= 2)
  }

  if (s_abort && tid == 0) {  // a load timed out: report, then wait (bounded) for copies still in flight
    report_error(a, kErrTimeout);
    for (uint32_t k = 0; k < nstage; ++k)
      if (s_tiles[k] < pl.ntiles) {
        mbar_wait(&s_full[k], 0u, 1u << 10);
        mbar_wait(&s_full[k], 1u, 1u << 10);
      }
  }
  if (scan_on) cta_finish<DT, true>(&s_ctl, s_red, smem + pl.sm_tile, sal, s_abort != 0u);
  cta_exit(pl, a, d, &s_last);
}

// -------------------------------------------------------------------------------------------------
// CTA-team kernel, register variant: planes of more than 1024 elements, up to kCtaMaxWarps * kCtaGroups groups.  One plane
// per tile; the CTA's warps (as few as hold the plane) take equal contiguous runs of its groups and keep them in
// registers, so the plane is read from its stage once.  Planes may start anywhere: the load takes in the 16-byte chunks
// around them.
//
// What every warp repeats per plane -- reductions, scalar steps, barriers: about 200 instructions -- is spread over up to
// 56 elements a lane, and what can wait does: the codes are computed and stored as if the plane were normal while the
// first warp works out the three-sigma thresholds, and the count of outliers is looked at behind the NEXT plane's
// first barrier, so that a plane costs three barriers.  A plane that turns out outlier-rich is still in its stage then;
// it is measured at the end of that turn, and phase 2 rewrites its slot.  PARTS: the plane has fewer rows of blocks than the CTA
// has warps (see fh_blocks.cuh; instances of their own, as the sweep of the others loses 5 % to the registers these take).
// -------------------------------------------------------------------------------------------------
constexpr int kCtaThreads = kCtaMaxWarps * 32;

// What the sweep only looks at now and then: the destination and, of thread 0, the next ticket, the number of loads issued and
// the last plane's minimum and scale, for its table entry.
struct CtaOwn {
  Dest d;
  uint32_t next_ticket, issued;
  float lo, scale;
};
// WORDS: bf16 runs are held as they lie in memory, with which 24 warps fit on an SM instead of 20 (28 without the plane's own
// statistics, and with random rounding, which reads the run again and takes 72 registers too).  That is taken for CTAs of 7, 11 and
// 12 warps, which come to three, two and two on an SM then and not to two, one and one, when there are planes for them (see
// word_runs): with few warps resident, the three barriers a plane are what such planes wait for.  us a call, 2 bits, before
// and now: 128 x 96 planes of 112 x 112 118.1 -> 108.0, with every eighth channel outlier-rich 250.2 -> 220.4, without statistics
// 73.2 -> 61.7, random rounding 249.3 -> 214.5; 64 x 32 of 140 x 140 46.3 -> 36.6, of 146 x 146 47.4 -> 39.9; 100 x 61 of
// 127 x 93 72.0 -> 68.1.  Elsewhere it is as many CTAs or little more, and with statistics the six instructions a group cost more than
// it gives: 56 x 56 (2 warps) 50.2 -> 55.6; 125 MB of 104 x 103 (6 warps) 53.8 -> 55.6, 119 x 120 (8) 55.8 -> 56.8, 126 x 128 (9)
// 52.7 -> 57.8, 152 x 153 (13) 69.1 -> 77.2, 158 x 158 (14) 64.0 -> 72.1.  (Not taken so far: without statistics and with random
// rounding it would pay at more widths, 13 warps 46.4 -> 35.2 and 148 -> 122.)
// What is not needed in every step is kept in shared memory then, since what does not fit the registers goes to local memory, for
// which the stages leave little L1.
template <bool WORDS>
struct Held {
  using T = float;
  static constexpr int N = 4;
};
template <>
struct Held<true> {
  using T = uint32_t;
  static constexpr int N = 2;
};
// (registers are dealt out by the threads that a CTA may have: 96, 80 or 72)
constexpr int cta_threads(bool words, int sigma) { return !words ? kCtaThreads : (sigma == 1 ? 768 : 896); }

template <int DT, int SIGMA, int K, int EDGE, bool PARTS, bool WORDS>
__global__ void __launch_bounds__(cta_threads(WORDS, SIGMA), 1) compress_cta_regs(const Plan pl, const CompressArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ double s_red[kMaxWarps * 4];
  __shared__ __align__(8) uint64_t s_full[2];
  __shared__ uint32_t s_tiles[2], s_abort, s_last, s_count[2];
  __shared__ float2 s_thr;
  __shared__ Cuts s_cut;
  __shared__ bool s_look;
  __shared__ BlockCtl s_ctl;
  __shared__ CtaOwn s_own;
  CtaOwn r_own;
  CtaOwn& own = WORDS ? s_own : r_own;

  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const Team team = make_cta_team(blockDim.x, s_red);
  const bool scan_on = pl.mode != kModeOff;
  uint32_t* sal = reinterpret_cast<uint32_t*>(smem + pl.sm_sal);
  uint32_t rp = 0;
  // Thread 0 requests the tiles and issues the loads: the first two in one request (one, when there are too few for every
  // CTA to get two), later ones one at a time, the request running one tile ahead of its use.  Tiles come in ticket order.
  if (tid == 0) {
    mbar_init(&s_full[0], 1);
    mbar_init(&s_full[1], 1);
    fence_mbar_init();
    s_abort = 0;
    s_count[0] = s_count[1] = 0;
    *cta_totals() = CtaTotals{0u, 0u, 0u, 0u};
    own.issued = 0;
    if (a.early_ticket) own.next_ticket = (uint32_t)atomicAdd(&a.sc->ticket[a.parity], kStarted + pl.nstage);
    if (scan_on) {  // (before the wait for the previous kernel, whose tail hides it)
      s_ctl.pl = pl;
      s_ctl.a = a;
      s_ctl.own = kNoTile;
    }
  }
  auto issue = [&](uint32_t s) {
    const uint32_t t = own.next_ticket;
    s_tiles[s] = t;
    if (t < pl.ntiles) {
      plane_load(pl, a.src, t, smem + (uint64_t)s * pl.stage_bytes, &s_full[s]);
      own.next_ticket = ++own.issued < pl.nstage ? t + 1u : (uint32_t)atomicAdd(&a.sc->ticket[a.parity], 1ull);
    }
  };
  // the previous kernel on the stream has completed; global memory may be touched from here on (the input is only read)
  if (!a.early_load) dep_wait();
  if (tid == 0) {  // the first loads before anything else
    if (!a.early_ticket) own.next_ticket = (uint32_t)atomicAdd(&a.sc->ticket[a.parity], kStarted + pl.nstage);
    issue(0);
    issue(1);
  }
  if (a.early_load) dep_wait();
  dep_trigger();  // the next kernel on the stream may become resident as this one drains
  if (!WORDS || tid == 0) own.d = make_dest(pl, a);
  if (tid == 0) {
    const Dest d = own.d;
    if (!d.fits && blockIdx.x == 0) report_error(a, kErrCapacity);
    if (scan_on) s_ctl.d = d;
  }
  __syncthreads();

  const uint32_t grain = plane_grain(pl);
  const uint32_t g0 = pl.groups * warp / team.nwarps, g1 = pl.groups * (warp + 1u) / team.nwarps;
  const int32_t n = (int32_t)(min(4u * g1, pl.HW) - 4u * g0);
  // the plane before, whose class is still open: its tile (kNoTile: none), and for its table entry minimum, scale
  uint32_t prev = kNoTile, prev_meta = 0;
  // Class of the plane before, behind a barrier that all its counts precede (every thread gets the same answer): a
  // normal plane is complete -- table entry, publication, its stage takes the next load --, another is to be measured.
  auto settle = [&](uint32_t s) -> bool {
    if (prev == kNoTile) return false;
    if (SIGMA) {
      const uint32_t n_out = s_count[s];
      prev_meta = ((uint64_t)n_out * pl.rho_den > (uint64_t)pl.rho_num * pl.HW ? kClsSalient : kClsNormal) | (n_out << 2);
    }
    if ((prev_meta & 3u) != kClsNormal) return true;
    if (tid == 0) {
      if (own.d.fits) store_table_entry(own.d, prev, (uint32_t)((pl.slots_off + (uint64_t)prev * pl.npay) >> 4), prev_meta, own.lo, own.scale);
      if (scan_on) scan_publish(a.scan, prev, 0u);
      issue(s);
    }
    return false;
  };
  auto measure = [&](uint32_t s) {
    cta_tile_measure<DT, PARTS>(&s_ctl, s_red, smem + (uint64_t)s * pl.stage_bytes + plane_head(pl, prev), sal, prev, prev_meta);
    if (tid == 0) {
      issue(s);
      queue_push(&s_ctl, prev, s, s_tiles[s] >= pl.ntiles);
    }
  };

  uint32_t s = 0, phase = 0;
  for (;;) {
    const uint32_t tile = s_tiles[s];
    if (tile >= pl.ntiles) break;
    const bool ready = mbar_wait(&s_full[s], (phase >> s) & 1u, 1u << 20);
    phase ^= 1u << s;
    typename Held<WORDS>::T x[K][Held<WORDS>::N];
    float lo, hi;
    const uint8_t* run = smem + (uint64_t)s * pl.stage_bytes + plane_head(pl, tile) + (uint64_t)g0 * (DT == kF32 ? 16u : 8u);
    run_load<DT, K, 32, EDGE>(run, lane, n, grain, x, lo, hi);
    if (!ready) s_abort = 1;
    team_minmax(team, lo, hi, rp);  // the first barrier
    if (s_abort) break;
    const bool open = settle(s ^ 1u);
    const float range = __fsub_rn(hi, lo);
    if (!(fabsf(range) <= 3.402823466e38f) && tid == 0) report_error(a, kErrNonfinite);
    const SigmaScale sc = sigma_scale(range);
    uint32_t as = 0, aq = 0;
    run_distances<DT, K, 32, EDGE, (SIGMA != 0)>(lane, n, lo, sc, x, as, aq);
    const bool rule = SIGMA && sc.applies;  // (the same for every thread)
    if (SIGMA) {
      int32_t pa = (int32_t)(as - (uint32_t)K * kMagicBits), pb = (int32_t)(aq - (uint32_t)K * kMagicBits);
      asm volatile("redux.sync.add.s32 %0, %0, %1;" : "+r"(pa) : "r"(0xFFFFFFFFu));
      asm volatile("redux.sync.add.s32 %0, %0, %1;" : "+r"(pb) : "r"(0xFFFFFFFFu));
      int2* r = reinterpret_cast<int2*>(red_half(team, rp));
      if (lane == 0) r[warp] = make_int2(pa, pb);
      __syncthreads();  // the second barrier
      if (warp == 0 && rule) {  // the first warp adds up the warps' sums and works out the thresholds, for all
        const int2 pr = lane < team.nwarps ? r[lane] : make_int2(0, 0);
        const long long Is = warp_sum_s32_wide(pr.x), Iq = warp_sum_s32_wide(pr.y);
        float tl, th;
        sigma_thresholds(Is, Iq, sc, pl.inv_hw, tl, th);
        if (lane == 0) {
          s_thr = make_float2(tl, th);
          if (WORDS) {
            s_look = range > th || 0.0f < tl;
            if (s_look) s_cut = element_cuts(lo, tl, th);
          }
        }
      }
      if (tid == 0) s_count[s ^ 1u] = 0;  // (settled by every thread before the barrier just passed)
    }
    float inv, scale;
    quant_params(range, (1u << pl.bits) - 1u, inv, scale);
    if (!WORDS || tid == 0) {  // (the plane before is settled, or is not a normal one)
      own.lo = lo;
      own.scale = scale;
    }
    uint32_t n_out = 0, cls = kClsNormal;
    if (!SIGMA) {
      if (pl.mode == kModeAll) cls = kClsSalient;
      if (pl.mode >= kModeChannel) cls = channel_class(pl, a, tile, n_out);
    }
    auto codes = [&]() {
      if (!own.d.fits || cls != kClsNormal) return;
      uint8_t* slot = own.d.dst + pl.slots_off + (uint64_t)tile * pl.npay;
      run_codes_any<DT, SIGMA, K, 32, EDGE>(pl, run, grain, lane, n, lo, inv, g0, tile, slot, x);
      pad_slot(pl, slot, tid, blockDim.x);
    };
    auto count = [&]() {
      if (!rule) return;
      __syncthreads();  // the third barrier: the thresholds
      const float dlo = s_thr.x, dhi = s_thr.y;
      if (WORDS ? s_look : range > dhi || 0.0f < dlo) {  // otherwise no element can lie outside
        uint32_t cnt;
        if constexpr (!WORDS) cnt = run_count<DT, K, 32, EDGE>(lane, n, dlo, dhi, x);
        else cnt = run_count<DT, K, 32, EDGE>(lane, n, own.lo, dlo, dhi, s_cut, x);
        asm volatile("redux.sync.add.u32 %0, %0, %1;" : "+r"(cnt) : "r"(0xFFFFFFFFu));
        if (lane == 0 && cnt) atomicAdd(&s_count[s], cnt);
      }
    };
    // (random rounding reads the run anew: with the distances out of the way there are registers for four groups at a time, whose
    // generators hide one another's latency: fp32, 2 bits, 64 x 64 planes of 112 x 112
    // 103.9 -> 91.6 us, of 56 x 56 33.6 -> 30.1)
    if (SIGMA == 2) {
      count();
      codes();
    } else {
      codes();
      count();
    }
    if (open) {  // the plane before, which is outlier-rich
      __syncthreads();
      measure(s ^ 1u);
    }
    prev = tile;
    prev_meta = cls | (n_out << 2);
    s ^= 1u;
    // (s_tiles of the next turn was written when the plane before was settled, behind the first barrier: a later one --
    // the second, with three-sigma statistics, or this one -- makes it known)
    if (!SIGMA || open) __syncthreads();
  }
  __syncthreads();
  if (!s_abort) {
    const bool open = settle(s ^ 1u);
    if (open) measure(s ^ 1u);
  }
  __syncthreads();
  if (s_abort && tid == 0) {  // a load timed out: report, then wait (bounded) for copies still in flight
    report_error(a, kErrTimeout);
    for (uint32_t k = 0; k < 2u; ++k)
      if (s_tiles[k] < pl.ntiles) {
        mbar_wait(&s_full[k], 0u, 1u << 10);
        mbar_wait(&s_full[k], 1u, 1u << 10);
      }
  }
  if (scan_on) cta_finish<DT, PARTS>(&s_ctl, s_red, smem, sal, s_abort != 0u);
  cta_exit(pl, a, own.d, &s_last);
}

}  // namespace fh

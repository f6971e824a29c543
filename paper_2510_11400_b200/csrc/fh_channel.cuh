// Channel-wide three-sigma statistics (salient_mode = CHANNEL): mu, sigma and the outlier count are taken
// over the N planes (n, c) of a channel c together, and the channel as a whole is normal or outlier-rich.
// Tensor-wide statistics (salient_mode = TENSOR) run through the same passes with the whole tensor as the
// one "channel"; a plane's class then follows from its own count.
// Three passes over the tensor, a team of lanes per plane (of at most 512 groups: larger ones go in pieces), results
// gathered per channel with atomics:
//   pass 0: minimum and maximum of the channel (the moments are taken of the distances from the minimum, and the
//           range fixes the scale of the integer sums);
//   pass 1: integer moment sums of the channel (exact, so the order of the atomics is immaterial);
//   pass 2: thresholds from the sums; outliers per plane (kept for the plane table) and per channel.
// The streaming kernel then reads a plane's class from its channel's count, so the tensor is read four times; what fits
// the L2 cache comes from there from the second time on.  A lane has 64 bytes in flight; the
// passes follow one another by programmatic launch; no memset between them (the streaming kernel's last CTA returns the
// statistics to zero).  Element by element with a warp per plane the three took 162 us for 32 x 96 bf16 planes of
// 112 x 112 (77 MB) and 27 us for 32 x 960 of 7 x 7; now 64 (16, 20 and 28) and 17 (5, 6 and 6), each kernel timed by itself.
#pragma once

#include "fh_device.cuh"

namespace fh {

// Order-preserving map float -> unsigned (finite values; -0.0 sorts below +0.0, and a distance from either is
// the same number).
__device__ __forceinline__ unsigned int float_key(float f) {
  const unsigned int b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key_float(unsigned int k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

// Group g of a plane as it lies there: four fp32 values, or two words of two bf16.  VEC: planes are whole groups on
// group-sized boundaries; otherwise positions past HW read as the plane's last element.  (The choice is made at compile
// time: a branch per load keeps the compiler from issuing the loads together.)
template <int DT, bool VEC>
__device__ __forceinline__ void load_group_raw(const uint8_t* plane, uint32_t g, uint32_t HW, uint32_t (&w)[4]) {
  if (VEC) {
    if (DT == kF32) {
      const uint4 t = __ldg(reinterpret_cast<const uint4*>(plane) + g);
      w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
    } else {
      const uint2 t = __ldg(reinterpret_cast<const uint2*>(plane) + g);
      w[0] = t.x; w[1] = t.y;
    }
    return;
  }
  uint32_t e[4];
#pragma unroll
  for (uint32_t k = 0; k < 4u; ++k) {
    const uint32_t i = min(g * 4u + k, HW - 1u);
    e[k] = DT == kF32 ? __ldg(reinterpret_cast<const uint32_t*>(plane) + i) : (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(plane) + i);
  }
  if (DT == kF32) {
#pragma unroll
    for (int k = 0; k < 4; ++k) w[k] = e[k];
  } else {
    w[0] = e[0] | e[1] << 16;
    w[1] = e[2] | e[3] << 16;
  }
}

constexpr uint32_t kChanPiece = 512;  // groups of a piece: their integer sums fit 32 bits

// Tensor-wide statistics have a single destination: the CTA's threads are combined in shared memory, and one of them issues the
// atomics.
template <int PASS>
__device__ __forceinline__ void channel_pass_whole(const ChannelArgs& a, float wlo, float whi, unsigned long long ws, unsigned long long wq,
                                                   float* s_lo, float* s_hi, unsigned long long* s_s, unsigned long long* s_q) {
  const uint32_t lane = threadIdx.x & 31u, full = 0xFFFFFFFFu;
  for (uint32_t o = 16; o > 0; o >>= 1) {
    wlo = fminf(wlo, __shfl_xor_sync(full, wlo, o));
    whi = fmaxf(whi, __shfl_xor_sync(full, whi, o));
  }
  ws = warp_sum_u64(ws);
  wq = warp_sum_u64(wq);
  const uint32_t warp = threadIdx.x >> 5;
  if (lane == 0) {
    s_lo[warp] = wlo;
    s_hi[warp] = whi;
    s_s[warp] = ws;
    s_q[warp] = wq;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (uint32_t k = 1; k < (uint32_t)kWarps; ++k) {
      wlo = fminf(wlo, s_lo[k]);
      whi = fmaxf(whi, s_hi[k]);
      ws += s_s[k];
      wq += s_q[k];
    }
    if (PASS == 0) {  // (every CTA of the grid owns at least one plane, so both values are numbers of the input)
      atomicMax(&a.chan->lo_inv, ~float_key(wlo));
      atomicMax(&a.chan->hi_key, float_key(whi));
    } else {
      atomicAdd(&a.chan->Is, ws);
      atomicAdd(&a.chan->Iq, wq);
    }
  }
}

template <int DT, int PASS, bool VEC>
__global__ void __launch_bounds__(kThreads, 4) channel_pass(const Plan pl, const ChannelArgs a) {
  const uint32_t tt = a.team, lane = threadIdx.x & 31u, tl = lane & (tt - 1u), full = 0xFFFFFFFFu;
  const bool whole = pl.mode == kModeTensor;
  __shared__ float s_lo[kWarps], s_hi[kWarps];
  __shared__ unsigned long long s_s[kWarps], s_q[kWarps];
  float wlo = __int_as_float(0x7F800000), whi = __int_as_float(0xFF800000);
  unsigned long long ws = 0, wq = 0;
  const uint32_t pieces = (pl.groups + kChanPiece - 1u) / kChanPiece;
  const uint64_t items = pl.P * pieces, step = (uint64_t)gridDim.x * (kThreads / tt);
  dep_trigger();
  dep_wait();
  for (uint64_t base = (uint64_t)blockIdx.x * (kThreads / tt); base < items; base += step) {  // (the warp stays together)
    const uint64_t item = base + threadIdx.x / tt;
    const bool there = item < items;
    const uint32_t p = !there ? 0u : (pieces == 1u ? (uint32_t)item : (uint32_t)(item / pieces));
    const uint32_t g0 = there ? (uint32_t)(item - (uint64_t)p * pieces) * kChanPiece : 0u, g1 = there ? min(pl.groups, g0 + kChanPiece) : 0u;
    const uint8_t* plane = a.src + p * pl.plane_bytes;
    ChanStat* cs = a.chan + (whole ? 0u : p % pl.C);
    float clo = 0.0f, dlo = 0.0f, dhi = 0.0f;
    SigmaScale sc = {};
    if (PASS > 0) {
      clo = key_float(~cs->lo_inv);
      sc = sigma_scale(__fsub_rn(key_float(cs->hi_key), clo));  // (not `applies`: a constant channel, or a range outside the rule's domain)
      if (PASS == 2) sigma_thresholds((long long)cs->Is, (long long)cs->Iq, sc, a.inv_nhw, dlo, dhi);
    }
    float lo = __int_as_float(0x7F800000), hi = __int_as_float(0xFF800000);
    uint32_t as = 0, aq = 0, n = 0;
    constexpr uint32_t U = DT == kF32 ? 4u : 8u;  // groups in flight: 64 bytes a lane
    for (uint32_t g = g0 + tl; g < g1; g += U * tt) {
      uint32_t w[U][4];
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) load_group_raw<DT, VEC>(plane, min(g + u * tt, g1 - 1u), pl.HW, w[u]);
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) {
        float v[4];
        if (DT == kF32) {
#pragma unroll
          for (int k = 0; k < 4; ++k) v[k] = __uint_as_float(w[u][k]);
        } else {
          v[0] = __uint_as_float(w[u][0] << 16); v[1] = __uint_as_float(w[u][0] & 0xFFFF0000u);
          v[2] = __uint_as_float(w[u][1] << 16); v[3] = __uint_as_float(w[u][1] & 0xFFFF0000u);
        }
        if (PASS == 0) {  // (an element read twice changes nothing; non-finite input is reported by the streaming kernel)
          lo = fminf(lo, fminf(fminf(v[0], v[1]), fminf(v[2], v[3])));
          hi = fmaxf(hi, fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])));
        } else {
          const uint32_t in = g + u * tt < g1 ? (VEC ? 4u : min(4u, pl.HW - 4u * (g + u * tt))) : 0u;
          float d[4];
#pragma unroll
          for (uint32_t k = 0; k < 4u; ++k) d[k] = k < in ? __fsub_rn(v[k], clo) : 0.0f;
          if (PASS == 1) {
            if (in) {
              sigma_addends(d, sc, as, aq);
              ++n;
            }
          } else {
#pragma unroll
            for (uint32_t k = 0; k < 4u; ++k) n += k < in && (d[k] > dhi || d[k] < dlo);
          }
        }
      }
    }
    if (PASS == 0) {
      for (uint32_t o = tt >> 1; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(full, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(full, hi, o));
      }
      wlo = fminf(wlo, lo);
      whi = fmaxf(whi, hi);
      if (there && tl == 0) {
        if (!whole) {
          atomicMax(&cs->lo_inv, ~float_key(lo));
          atomicMax(&cs->hi_key, float_key(hi));
        }
        if (g0 == 0u) a.plane_nout[p] = 0;
      }
    } else if (PASS == 1) {
      uint32_t s = sc.applies ? as - n * kMagicBits : 0u, q = sc.applies ? aq - n * kMagicBits : 0u;
      for (uint32_t o = tt >> 1; o > 0; o >>= 1) {
        s += __shfl_xor_sync(full, s, o);
        q += __shfl_xor_sync(full, q, o);
      }
      if (there && tl == 0) {
        ws += s;
        wq += q;
        if (!whole && sc.applies) {
          atomicAdd(&cs->Is, (unsigned long long)s);
          atomicAdd(&cs->Iq, (unsigned long long)q);
        }
      }
    } else {
      if (!sc.applies) n = 0;
      for (uint32_t o = tt >> 1; o > 0; o >>= 1) n += __shfl_xor_sync(full, n, o);
      if (there && tl == 0 && n) {
        if (pieces == 1u) a.plane_nout[p] = n;
        else atomicAdd(&a.plane_nout[p], n);
        if (!whole) atomicAdd(&cs->nout, (unsigned long long)n);  // the tensor-wide mode classifies by the plane's count
      }
    }
  }
  if (whole && PASS < 2) channel_pass_whole<PASS>(a, wlo, whi, ws, wq, s_lo, s_hi, s_s, s_q);
}

// The same for planes of more than 64 groups (a team is a whole warp then) that are whole groups: a warp takes a run of pieces in
// channel order, so that it works out a channel's scale and thresholds (a chain of loads, 64-bit arithmetic and a square
// root) once or twice and not once a piece, and sends its sums off at the channel's end.  The next loads are asked for before the
// present ones' elements are worked on.  What bounds it is the L2 cache's latency and rate.  A whole call, a piece at a time and
// now, us: bf16, 32 x 96 of 112 x 112 136.6 -> 131.4, 32 x 144 of 56 x 56 78.7 -> 76.7, 32 x 192 of 28 x 28 46.9 -> 43.9; fp32, 32 x 96
// of 112 x 112 172.5 -> 161.3.  (Planes that are not whole groups, loaded element by element, have no registers to load ahead:
// 47 x 33 66.9 -> 70.7; they stay with the kernel above.)
template <int DT, int PASS>
__global__ void __launch_bounds__(kThreads, 4) channel_pass_runs(const Plan pl, const ChannelArgs a) {
  constexpr uint32_t U = DT == kF32 ? 4u : 8u;  // groups a lane loads at a time: 64 bytes
  const uint32_t lane = threadIdx.x & 31u, full = 0xFFFFFFFFu, warp = threadIdx.x >> 5;
  const bool whole = pl.mode == kModeTensor;
  __shared__ float s_lo[kWarps], s_hi[kWarps];
  __shared__ unsigned long long s_s[kWarps], s_q[kWarps];
  const uint32_t pieces = (pl.groups + kChanPiece - 1u) / kChanPiece, part = ((pl.groups + pieces - 1u) / pieces + 31u) & ~31u;
  const uint32_t planes = whole ? (uint32_t)pl.P : pl.N;  // of a channel
  const uint64_t nw = (uint64_t)gridDim.x * kWarps, w0 = (uint64_t)blockIdx.x * kWarps + warp, items = pl.P * pieces;
  uint32_t left = (uint32_t)(items * (w0 + 1u) / nw - items * w0 / nw);  // pieces of the run
  uint32_t c, n, piece;
  {
    const uint32_t i = (uint32_t)(items * w0 / nw), q = i / pieces;
    piece = i - q * pieces;
    c = q / planes;
    n = q - c * planes;
  }
  float lo = __int_as_float(0x7F800000), hi = __int_as_float(0xFF800000);
  unsigned long long ws = 0, wq = 0;
  uint32_t nout = 0;
  uint32_t g = piece * part + lane, end = min(pl.groups, (piece + 1u) * part);
  uint64_t p = (uint64_t)n * (whole ? 1u : pl.C) + c;
  uint32_t buf[U][DT == kF32 ? 4 : 2], nxt[U][DT == kF32 ? 4 : 2];
  auto load = [&](uint32_t (&to)[U][DT == kF32 ? 4 : 2]) {
    const uint8_t* plane = a.src + p * pl.plane_bytes;
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      uint32_t t[4];
      load_group_raw<DT, true>(plane, min(g + u * 32u, end - 1u), pl.HW, t);
#pragma unroll
      for (int k = 0; k < (DT == kF32 ? 4 : 2); ++k) to[u][k] = t[k];
    }
  };
  dep_trigger();
  dep_wait();
  if (left) load(buf);
  float clo = 0.0f, dlo = 0.0f, dhi = 0.0f;
  SigmaScale sc = {};
  bool fresh = true;
  uint32_t as = 0, aq = 0, cnt = 0;
  while (left) {
    ChanStat* cs = a.chan + (whole ? 0u : c);
    const uint32_t g_now = g, end_now = end;
    const uint64_t p_now = p;
    const bool last = g - lane + U * 32u >= end;  // (of the piece)
    bool flush = false;
    if (PASS == 0 && g == 0u) a.plane_nout[p] = 0;  // (lane 0, ahead of the plane's first group)
    g += U * 32u;
    if (last) {
      --left;
      if (++piece == pieces) {
        piece = 0;
        if (++n == planes) {
          n = 0;
          ++c;
          flush = true;
        }
        p = (uint64_t)n * (whole ? 1u : pl.C) + c;
      }
      g = piece * part + lane;
      end = min(pl.groups, (piece + 1u) * part);
      flush |= left == 0u;
    }
    if (left) load(nxt);
    if (PASS > 0 && fresh) {
      clo = key_float(~cs->lo_inv);
      sc = sigma_scale(__fsub_rn(key_float(cs->hi_key), clo));  // (not `applies`: a constant channel, or a range outside the rule's domain)
      if (PASS == 2) sigma_thresholds((long long)cs->Is, (long long)cs->Iq, sc, a.inv_nhw, dlo, dhi);
      fresh = false;
    }
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      float v[4];
      if (DT == kF32) {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = __uint_as_float(buf[u][k]);
      } else {
        v[0] = __uint_as_float(buf[u][0] << 16); v[1] = __uint_as_float(buf[u][0] & 0xFFFF0000u);
        v[2] = __uint_as_float(buf[u][1] << 16); v[3] = __uint_as_float(buf[u][1] & 0xFFFF0000u);
      }
      if (PASS == 0) {  // (an element read twice changes nothing; non-finite input is reported by the streaming kernel)
        lo = fminf(lo, fminf(fminf(v[0], v[1]), fminf(v[2], v[3])));
        hi = fmaxf(hi, fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])));
      } else {
        const bool in = g_now + u * 32u < end_now;
        float d[4];
#pragma unroll
        for (uint32_t k = 0; k < 4u; ++k) d[k] = __fsub_rn(v[k], clo);
        if (PASS == 1) {
          if (in) {
            sigma_addends(d, sc, as, aq);
            ++cnt;
          }
        } else {
#pragma unroll
          for (uint32_t k = 0; k < 4u; ++k) cnt += in && (d[k] > dhi || d[k] < dlo);
        }
      }
    }
    if (last) {
      if (PASS == 1) {  // (a lane's sums of a piece fit 32 bits)
        if (sc.applies) {
          ws += as - cnt * kMagicBits;
          wq += aq - cnt * kMagicBits;
        }
        as = aq = cnt = 0;
      } else if (PASS == 2) {
        asm volatile("redux.sync.add.u32 %0, %0, %1;" : "+r"(cnt) : "r"(full));
        if (!sc.applies) cnt = 0;
        if (lane == 0 && cnt) {
          if (pieces == 1u) a.plane_nout[p_now] = cnt;
          else atomicAdd(&a.plane_nout[p_now], cnt);
        }
        nout += cnt;
        cnt = 0;
      }
    }
    if (flush && !whole) {
      if (PASS == 0) {
        const uint32_t kl = __reduce_max_sync(full, ~float_key(lo)), kh = __reduce_max_sync(full, float_key(hi));
        if (lane == 0) {
          atomicMax(&cs->lo_inv, kl);
          atomicMax(&cs->hi_key, kh);
        }
        lo = __int_as_float(0x7F800000);
        hi = __int_as_float(0xFF800000);
      } else if (PASS == 1) {
        ws = warp_sum_u64(ws);
        wq = warp_sum_u64(wq);
        if (lane == 0 && sc.applies) {
          atomicAdd(&cs->Is, ws);
          atomicAdd(&cs->Iq, wq);
        }
        ws = wq = 0;
      } else {
        if (lane == 0 && nout) atomicAdd(&cs->nout, (unsigned long long)nout);
        nout = 0;
      }
      fresh = true;
    }
#pragma unroll
    for (uint32_t u = 0; u < U; ++u)
#pragma unroll
      for (int k = 0; k < (DT == kF32 ? 4 : 2); ++k) buf[u][k] = nxt[u][k];
  }
  if (whole && PASS < 2) channel_pass_whole<PASS>(a, lo, hi, ws, wq, s_lo, s_hi, s_s, s_q);
}

}  // namespace fh

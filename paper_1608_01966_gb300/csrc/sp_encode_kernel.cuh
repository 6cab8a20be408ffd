// Frame encoder kernel: colour frames -> reduction -> gray -> adaptive
// Gaussian threshold -> packed input bits.
//
// The work is integer arithmetic on every pixel, so instructions issued per
// pixel bound it before memory does.  One warp walks a strip of 240 output
// columns downwards, a row at a time, and keeps everything in registers; no
// barrier and no shared image.  Lane l holds the 8 pixels 8 (l - 1) .. 8 (l -
// 1) + 7 of the strip; lanes 0 and 31 are the halo (at most 6 columns on each
// side), lanes 1..30 produce output.  Per row:
//   1. 8 gray pixels, a byte each: the luma of f x f block means, or the bytes
//      as they are; pixels outside the image replicate its edge (a byte
//      permute chosen once per lane; rows are clamped).  The source rows come
//      through a ring in shared memory that each lane fills for itself a few
//      rows ahead (cp.async), so a warp has several rows in flight without
//      holding them in registers;
//   2. the vertical binomial window as a cascade of 2 half [1 1] steps: a step
//      adds the previous row's value, so a row costs one add per step and two
//      pixels share a 32-bit add for the first 8 steps (255 * 2^8 < 2^16);
//   3. the horizontal binomial window on those 16-bit sums: neighbours' words
//      by shuffles, two taps per 16-bit dot product, 6 products a pixel at
//      window 11, the rounding constant and the offset in the accumulator;
//   4. the vertical steps past the 8th, on 32-bit sums (the two directions
//      commute);
//   5. the comparison's sign bits, gathered into the lane's 8 output bits.
// The weighted sum, its rounding and the comparison are exact integers as in
// the definition: g + offset > floor((s + h) / 2^k) iff (g + offset) 2^k > s + h.
//
// 128 frames of 960 x 540 RGB, window 11: 86 us, 26 warp instructions per 32
// pixels at 1.15 times the rows (halo); gray and vertical sums of a band in shared
// memory, three barriers apart (sp_encode_band.cu), 211 us and 101.  64 frames of
// 1920 x 1080 halved: 94 us (4.3 TB/s) against 529.  4 warps a scheduler at 128
// registers; at 96 registers (5 warps) the cascade spills: 105 and 204 us.
#pragma once

#include "sp_encode_rule.h"
#include "sp_encode_strip.cuh"

namespace sp {
namespace enc {

constexpr uint32_t kWarps = 2;     // independent warps of a CTA
constexpr uint32_t kStrip = kEncodeStrip;  // output columns of a strip: lanes 1..30
constexpr uint32_t kAll = 0xffffffffu;

// Luma (77 R + 150 G + 29 B + 128) >> 8 of four pixels, given the sums before
// the shift (16 bits each): their second bytes.
__device__ __forceinline__ uint32_t pack_luma(uint32_t l0, uint32_t l1, uint32_t l2, uint32_t l3) {
  return __byte_perm(__byte_perm(l0, l1, 0x0051), __byte_perm(l2, l3, 0x0051), 0x5410);
}

// Gray of four RGB pixels held in three little-endian words
// (R0 G0 B0 R1 | G1 B1 R2 G2 | B2 R3 G3 B3).
__device__ __forceinline__ uint32_t gray4_rgb(uint32_t w0, uint32_t w1, uint32_t w2) {
  constexpr uint32_t k0 = 77u | (150u << 8) | (29u << 16);  // byte 3 weighs 0
  constexpr uint32_t k3 = k0 << 8;                          // byte 0 weighs 0
  return pack_luma(__dp4a(w0, k0, 128u), __dp4a(__byte_perm(w0, w1, 0x0543), k0, 128u),
                   __dp4a(__byte_perm(w1, w2, 0x0432), k0, 128u), __dp4a(w2, k3, 128u));
}

// Add word m of a source row's 8 F pixels (CH channels) to the block sums:
// every (pixel, channel) that owns bytes of the word gets one dot product.
template <int CH, int F>
__device__ __forceinline__ void add_word(uint32_t (&s)[8][CH], int m, uint32_t w) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      uint32_t mask = 0u;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int b = 4 * m + k;
        if (b / (F * CH) == i && b % CH == c) mask |= 1u << (8 * k);
      }
      if (mask) s[i][c] = __dp4a(w, mask, s[i][c]);
    }
  }
}

// The 8 gray bytes of the block sums: channel means rounded half up, luma.
template <int CH, int F>
__device__ __forceinline__ uint2 gray8_sums(const uint32_t (&s)[8][CH]) {
  constexpr uint32_t area = F * F, half = area / 2u;
  uint32_t g[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (CH == 1)
      g[i] = ((s[i][0] + half) / area) << 8;  // where pack_luma looks
    else
      g[i] = 77u * ((s[i][0] + half) / area) + 150u * ((s[i][CH > 1 ? 1 : 0] + half) / area) +
             29u * ((s[i][CH > 1 ? 2 : 0] + half) / area) + 128u;
  }
  return make_uint2(pack_luma(g[0], g[1], g[2], g[3]), pack_luma(g[4], g[5], g[6], g[7]));
}

// Two horizontal weights of window B starting at tap i (0 past either end),
// as the low two bytes of a dot product operand; `hi`: the weights' high bytes
// (only window 13 has any).
template <int B>
__host__ __device__ constexpr uint32_t weight2(int i, bool hi) {
  uint32_t r = 0;
  for (int k = 0; k < 2; ++k) {
    const int j = i + k;
    const uint32_t w = j >= 0 && j < B ? binom(B - 1, j) : 0u;
    r |= (hi ? w >> 8 : w & 255u) << (8 * k);
  }
  return r;
}

// The binomial window of row sums v (8 + 4 HW pixels as 16-bit pairs, this
// lane's first pixel at pixel 2 HW) around this lane's pixel T, plus c.
template <int B, int HW, int T>
__device__ __forceinline__ uint32_t window_sum(const uint32_t (&v)[4 + 2 * HW], uint32_t c) {
  constexpr int s = T - (B - 1) / 2 + 2 * HW;  // first tap's pixel
  constexpr int m0 = s / 2, m1 = (s + B - 1) / 2;
  uint32_t hi = 0u;
#pragma unroll
  for (int m = m0; m <= m1; ++m) {
    c = __dp2a_lo(v[m], weight2<B>(2 * m - s, false), c);
    if (weight2<B>(2 * m - s, true)) hi = __dp2a_lo(v[m], weight2<B>(2 * m - s, true), hi);
  }
  return B > 11 ? c + (hi << 8) : c;
}

// Window B, CH channels, reduction F; A8: source rows, frames and the strips'
// first pixels lie on 8-byte boundaries and output rows are whole bytes.
template <int B, int CH, int F, bool A8>
__global__ void __launch_bounds__(kWarps * 32, 8) sp_encode_kernel(const EncodeArgs a) {
  constexpr int H = (B - 1) / 2;
  constexpr int K16 = 2 * H < 8 ? 2 * H : 8;  // vertical steps on 16-bit sums
  constexpr int K32 = 2 * H - K16;            // and on 32-bit ones
  constexpr int HW = (H + 1) / 2;             // words of a neighbour lane
  constexpr int SH = 4 * H;                   // log2 of the window's weight
  __shared__ uint2 s_gray[kWarps][8][32];     // gray rows until their output row comes
  // the ring of source rows: a stage is one source row of this lane's 8 F
  // pixels (and the word that an unaligned row spills into); kAhead stages
  constexpr int kWords = 2 * F * CH, kSlots = kWords + (A8 ? 0 : 1);
  constexpr int kAhead = F == 1 ? 4 : 6;
  __shared__ __align__(8) uint32_t s_raw[kWarps][kAhead][kSlots * 32];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t u = blockIdx.x * kWarps + warp;
  if (u >= a.units) return;
  const uint32_t strip = u % a.strips, v0 = u / a.strips;
  const uint32_t chunk = v0 % a.chunks, frame = v0 / a.chunks;
  const int y0 = (int)(chunk * a.rows), y1 = min((int)a.Hr, y0 + (int)a.rows);
  const int x = (int)(strip * kStrip) + 8 * ((int)lane - 1);
  const int W = (int)a.Wr;  // at least 8
  // the 8 pixels read, [xb, xb + 8), and where each of this lane's (clamped)
  // pixels lies among them
  const int xb = min(max(x, 0), W - 8);
  uint32_t sel[2] = {0u, 0u};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int j = min(max(min(max(x + i, 0), W - 1) - xb, 0), 7);
    sel[i >> 2] |= (uint32_t)j << (4 * (i & 3));
  }
  const uint8_t* f0 = a.src + (uint64_t)frame * a.src_stride;
  const uint8_t* f1 = f0 + a.frame_bytes;
  const uint64_t row_bytes = (uint64_t)a.W * CH;
  const uint8_t* fx = f0 + (uint64_t)((uint32_t)xb * F * CH);
  auto clamp_row = [&](int i) { return (uint32_t)min(max(y0 - H + i, 0), (int)a.Hr - 1); };
  const int n = y1 - y0 + 2 * H;
  int fetch_row = 0, fetch_dy = 0, fetch_slot = 0, use_slot = 0;
  auto fetch = [&]() {
    if (fetch_row < n) {
      const uint8_t* p = fx + ((uint64_t)clamp_row(fetch_row) * F + (uint32_t)fetch_dy) * row_bytes;
      uint32_t* dst = &s_raw[warp][fetch_slot][0];
      if (A8) {
#pragma unroll
        for (int k = 0; k < kWords / 2; ++k)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(
                           (uint32_t)__cvta_generic_to_shared(dst + 2 * (k * 32 + lane))),
                       "l"(p + 8 * k)
                       : "memory");
      } else {
        const uint32_t mis = (uint32_t)(reinterpret_cast<uintptr_t>(p) & 3u);
        const uint8_t* q = p - mis;
        if (q >= f0) {
          // whole words; the last one stops at the frame's end
#pragma unroll
          for (int k = 0; k < kSlots; ++k) {
            const uint8_t* w = q + 4 * k;
            if (k < kWords || mis) {
              const uint32_t take = f1 - w >= 4 ? 4u : (uint32_t)(f1 - w);
              asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(
                               (uint32_t)__cvta_generic_to_shared(dst + k * 32 + lane)),
                           "l"(w), "r"(take)
                           : "memory");
            }
          }
        } else {
          // the frame starts inside the first word: its bytes one by one
          for (int k = 0; k < kSlots; ++k) {
            uint32_t w = 0u;
            for (int b = 0; b < 4; ++b) {
              const uint8_t* s = q + 4 * k + b;
              if (s >= p && s < p + 4 * kWords) w |= (uint32_t)__ldg(s) << (8 * b);
            }
            dst[k * 32 + lane] = w;
          }
        }
      }
      if (F == 1 || ++fetch_dy == F) {
        fetch_dy = 0;
        ++fetch_row;
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    fetch_slot = fetch_slot + 1 == kAhead ? 0 : fetch_slot + 1;
  };
  // the oldest stage's words (source row dy of gray row i)
  auto next_stage = [&](uint32_t (&w)[kWords], int i, int dy) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kAhead - 1) : "memory");
    const uint32_t* src = &s_raw[warp][use_slot][0];
    if (A8) {
#pragma unroll
      for (int k = 0; k < kWords / 2; ++k) {
        const uint2 t = *reinterpret_cast<const uint2*>(src + 2 * (k * 32 + lane));
        w[2 * k] = t.x;
        w[2 * k + 1] = t.y;
      }
    } else {
      const uint32_t low = (uint32_t)reinterpret_cast<uintptr_t>(fx) +
                           (clamp_row(i) * F + (uint32_t)dy) * (uint32_t)row_bytes;
      const uint32_t sh = 8u * (low & 3u);
      uint32_t prev = src[lane];
#pragma unroll
      for (int k = 0; k < kWords; ++k) {
        const uint32_t next = src[(k + 1) * 32 + lane];  // unused bits where the row is aligned
        w[k] = __funnelshift_r(prev, next, sh);
        prev = next;
      }
    }
    use_slot = use_slot + 1 == kAhead ? 0 : use_slot + 1;
  };
  auto gray_row = [&](int i) -> uint2 {
    uint32_t w[kWords];
    uint2 g;
    if (F == 1) {
      next_stage(w, i, 0);
      if (CH == 1)
        g = make_uint2(w[0], w[1]);
      else
        g = make_uint2(gray4_rgb(w[0], w[1], w[CH > 1 ? 2 : 0]),
                       gray4_rgb(w[CH > 1 ? 3 : 0], w[CH > 1 ? 4 : 0], w[CH > 1 ? 5 : 0]));
      fetch();
    } else {
      uint32_t s[8][CH];
#pragma unroll
      for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int c = 0; c < CH; ++c) s[q][c] = 0u;
#pragma unroll
      for (int dy = 0; dy < F; ++dy) {
        next_stage(w, i, dy);
#pragma unroll
        for (int m = 0; m < kWords; ++m) add_word<CH, F>(s, m, w[m]);
        fetch();
      }
      g = gray8_sums<CH, F>(s);
    }
    return make_uint2(__byte_perm(g.x, g.y, sel[0]), __byte_perm(g.x, g.y, sel[1]));
  };

  uint32_t p16[K16][4], p32[K32 > 0 ? K32 : 1][8];
#pragma unroll
  for (int k = 0; k < K16; ++k)
#pragma unroll
    for (int w = 0; w < 4; ++w) p16[k][w] = 0u;
#pragma unroll
  for (int k = 0; k < (K32 > 0 ? K32 : 1); ++k)
#pragma unroll
    for (int t = 0; t < 8; ++t) p32[k][t] = 0u;
  // what every window sum starts from: the rounding term, and where the
  // comparison fits 32 bits (window <= 11) the offset, each step past the
  // horizontal one doubling it
  constexpr uint32_t kHalf = 1u << (SH - 1);
  const uint32_t c0 = (uint32_t)((B > 11 ? (int32_t)kHalf
                                         : (int32_t)kHalf - a.offset * (1 << (SH < 24 ? SH : 0))) /
                                 (1 << K32));
  const bool bytes = A8 || (W & 7) == 0;  // a lane's 8 bits are a byte of the output
  uint32_t* out = a.out + (uint64_t)frame * a.out_stride;
  const bool mine = lane >= 1u && lane <= 30u && x < W;
#pragma unroll
  for (int k = 0; k < kAhead; ++k) fetch();
#pragma unroll 2
  for (int i = 0; i < n; ++i) {
    // 1. gray
    const uint2 g = gray_row(i);
    s_gray[warp][i & 7][lane] = g;
    // 2. vertical steps on 16-bit pairs
    uint32_t v[4 + 2 * HW];
    v[HW] = __byte_perm(g.x, 0u, 0x4140);
    v[HW + 1] = __byte_perm(g.x, 0u, 0x4342);
    v[HW + 2] = __byte_perm(g.y, 0u, 0x4140);
    v[HW + 3] = __byte_perm(g.y, 0u, 0x4342);
#pragma unroll
    for (int k = 0; k < K16; ++k)
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const uint32_t t = v[HW + w] + p16[k][w];
        p16[k][w] = v[HW + w];
        v[HW + w] = t;
      }
    if (i < K16) continue;  // the first K16 rows only fill the cascade
    // 3. horizontal window
#pragma unroll
    for (int w = 0; w < HW; ++w) {
      v[w] = __shfl_up_sync(kAll, v[4 + w], 1);
      v[HW + 4 + w] = __shfl_down_sync(kAll, v[HW + w], 1);
    }
    uint32_t s[8];
    s[0] = window_sum<B, HW, 0>(v, c0);
    s[1] = window_sum<B, HW, 1>(v, c0);
    s[2] = window_sum<B, HW, 2>(v, c0);
    s[3] = window_sum<B, HW, 3>(v, c0);
    s[4] = window_sum<B, HW, 4>(v, c0);
    s[5] = window_sum<B, HW, 5>(v, c0);
    s[6] = window_sum<B, HW, 6>(v, c0);
    s[7] = window_sum<B, HW, 7>(v, c0);
    // 4. the remaining vertical steps
#pragma unroll
    for (int k = 0; k < K32; ++k)
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const uint32_t z = s[t] + p32[k][t];
        p32[k][t] = s[t];
        s[t] = z;
      }
    if (i < 2 * H) continue;
    // 5. output row y0 + i - 2 H, whose gray row came H rows ago
    const uint2 gc = s_gray[warp][(i - H) & 7][lane];
    uint32_t m = 0u;
#pragma unroll
    for (int t = 7; t >= 0; --t) {
      const uint32_t gt = ((t < 4 ? gc.x : gc.y) >> (8 * (t & 3))) & 255u;
      const uint32_t d = B > 11 ? (s[t] >> SH) - gt - (uint32_t)a.offset
                                : s[t] - (gt << (SH < 32 ? SH : 0));
      m = __funnelshift_l(d, m, 1);  // the sign bit: 1 where the pixel is above
    }
    const uint32_t at = (uint32_t)(y0 + i - 2 * H) * (uint32_t)W + (uint32_t)x;
    if (bytes) {
      if (mine) reinterpret_cast<uint8_t*>(out)[at >> 3] = (uint8_t)m;
    } else {
      // rows that do not start at a byte: four lanes' bits as one word, OR'ed
      // into the (zeroed) words they straddle
      if (!mine)
        m = 0u;
      else if (x + 8 > W)
        m &= (1u << (W - x)) - 1u;
      const uint32_t m1 = __shfl_down_sync(kAll, m, 1), m2 = __shfl_down_sync(kAll, m, 2),
                     m3 = __shfl_down_sync(kAll, m, 3);
      if ((lane & 3u) == 1u && mine) {
        const uint32_t w = m | (m1 << 8) | (lane < 29u ? (m2 << 16) | (m3 << 24) : 0u);
        const uint32_t sh = at & 31u, lo = w << sh, hi = sh ? w >> (32u - sh) : 0u;
        if (lo) atomicOr(out + (at >> 5), lo);
        if (hi) atomicOr(out + (at >> 5) + 1u, hi);
      }
    }
  }
  // the unused high bytes of the last word
  if (bytes && strip + 1u == a.strips && chunk + 1u == a.chunks && lane == 0u)
    for (uint32_t b = (uint32_t)W * a.Hr / 8u; b < a.n_words * 4u; ++b)
      reinterpret_cast<uint8_t*>(out)[b] = 0u;
}

// f is 1 or 2; a8: see the kernel.  Unaligned RGB rows take the strip kernel up
// to window 7 only (encode_in_strips).
template <int B>
cudaError_t launch_block(const EncodeArgs& a, bool a8, cudaStream_t st) {
  const uint32_t grid = (a.units + kWarps - 1u) / kWarps, threads = kWarps * 32;
  if (a.ch == 3u && a8) {
    if (a.f == 1u)
      sp_encode_kernel<B, 3, 1, true><<<grid, threads, 0, st>>>(a);
    else
      sp_encode_kernel<B, 3, 2, true><<<grid, threads, 0, st>>>(a);
  } else if (a.ch == 3u) {
    if constexpr (B <= 7) {
      if (a.f == 1u)
        sp_encode_kernel<B, 3, 1, false><<<grid, threads, 0, st>>>(a);
      else
        sp_encode_kernel<B, 3, 2, false><<<grid, threads, 0, st>>>(a);
    } else {
      return cudaErrorNotSupported;
    }
  } else if (a.f == 1u) {
    if (a8)
      sp_encode_kernel<B, 1, 1, true><<<grid, threads, 0, st>>>(a);
    else
      sp_encode_kernel<B, 1, 1, false><<<grid, threads, 0, st>>>(a);
  } else {
    sp_encode_kernel<B, 1, 2, false><<<grid, threads, 0, st>>>(a);
  }
  return cudaGetLastError();
}

extern template cudaError_t launch_block<3>(const EncodeArgs&, bool, cudaStream_t);
extern template cudaError_t launch_block<5>(const EncodeArgs&, bool, cudaStream_t);
extern template cudaError_t launch_block<7>(const EncodeArgs&, bool, cudaStream_t);
extern template cudaError_t launch_block<9>(const EncodeArgs&, bool, cudaStream_t);
extern template cudaError_t launch_block<11>(const EncodeArgs&, bool, cudaStream_t);
extern template cudaError_t launch_block<13>(const EncodeArgs&, bool, cudaStream_t);

}  // namespace enc
}  // namespace sp

// Frame encoder, band kernel: colour frames -> reduction -> gray -> adaptive
// Gaussian threshold -> packed input bits, for the calls that strips are slower
// on (sp_encode_rule.h): reductions by 3 and more, strips filled badly or with
// rows slow to read, and outputs narrower than a strip kernel's lane.
//
// One CTA encodes a band of output rows of one frame.  It owns the output
// words whose first pixel lies in the band; the last of them may run into
// the next rows, so the CTA also computes those.  Three phases, all in
// shared memory and all integer arithmetic:
//   A. gray image of the band's rows plus a halo of (block-1)/2 rows above
//      and below (rows outside the image replicate the edge rows), each
//      pixel the luma of its reduced (block-mean) colour;
//   B. vertical binomial sums V of the band's rows, computed for
//      (block-1)/2 extra columns on each side that replicate the edge
//      columns, so phase C needs no clamping;
//   C. one warp per output word: each lane applies the horizontal binomial
//      sum to V at its pixel, rounds the local mean, compares, and the warp
//      ballot is the word; when rows are a whole number of words, a lane
//      takes four adjacent pixels from vector loads of V and eight lanes
//      OR their nibbles into a word.
// Reading the source bounds it: f^2 source pixels a pixel, and the halo rows
// once per CTA of up to 32 rows.
#include "sp_encode_strip.cuh"

#include <algorithm>
#include <atomic>

namespace sp {

extern std::atomic<uint64_t> g_launches;

namespace {

constexpr int kEncThreads = 512;
constexpr uint32_t kEncSmemTarget = 100u << 10;  // two CTAs per SM
constexpr uint32_t kEncSmemMax = 200u << 10;

struct BandArgs {
  const uint8_t* src;
  uint64_t src_stride;  // bytes between frames
  uint32_t W, ch, f;    // source width, channels, reduction factor
  uint32_t Wr, Hr;      // output size
  int32_t offset;
  uint32_t* out;
  uint64_t out_stride;  // words between encoded frames
  uint32_t n_words;
  uint32_t band_rows;   // output rows per CTA
  uint32_t g_pitch;     // bytes per gray row in shared memory
  uint32_t g_bytes;     // bytes of the gray area (16-byte multiple)
  uint32_t v_pitch;     // words per V row: >= Wr + block + 2, a multiple of 4
  uint32_t vec4;        // f == 1 and 4-byte aligned rows: four pixels per load
  uint32_t vecf;        // f % 4 == 0 and 4-byte aligned rows: whole words per block row
};

__device__ __forceinline__ uint32_t reduced_gray(const BandArgs& a, const uint8_t* fs,
                                                 uint32_t gy, uint32_t x) {
  if (a.f == 1u) {
    const uint8_t* px = fs + ((uint64_t)gy * a.W + x) * a.ch;
    if (a.ch == 1u) return __ldg(px);
    return (77u * __ldg(px) + 150u * __ldg(px + 1) + 29u * __ldg(px + 2) + 128u) >> 8;
  }
  uint32_t s0 = 0, s1 = 0, s2 = 0;
  for (uint32_t dy = 0; dy < a.f; ++dy) {
    const uint8_t* row = fs + ((uint64_t)(gy * a.f + dy) * a.W + (uint64_t)x * a.f) * a.ch;
    for (uint32_t dx = 0; dx < a.f; ++dx) {
      const uint8_t* px = row + dx * a.ch;
      s0 += __ldg(px);
      if (a.ch == 3u) {
        s1 += __ldg(px + 1);
        s2 += __ldg(px + 2);
      }
    }
  }
  const uint32_t area = a.f * a.f, half = area / 2u;
  const uint32_t r = (s0 + half) / area;
  if (a.ch == 1u) return r;
  const uint32_t g = (s1 + half) / area, b = (s2 + half) / area;
  return (77u * r + 150u * g + 29u * b + 128u) >> 8;
}

// reduced_gray for f % 4 == 0 from aligned words: a block row of f pixels is
// 3f/4 words (RGB, repeating every three words) or f/4 words (gray), whose
// channel bytes are summed with byte dot products.
__device__ __forceinline__ uint32_t reduced_gray_words(const BandArgs& a, const uint8_t* fs,
                                                       uint32_t gy, uint32_t x) {
  const uint32_t* base = reinterpret_cast<const uint32_t*>(fs);
  const uint32_t wpr = a.W * a.ch / 4u;  // words per source row
  const uint32_t nw = a.f * a.ch / 4u;   // words per block row
  uint32_t s0 = 0, s1 = 0, s2 = 0;
  for (uint32_t dy = 0; dy < a.f; ++dy) {
    const uint32_t* w = base + (uint64_t)(gy * a.f + dy) * wpr + (uint64_t)x * nw;
    if (a.ch == 1u) {
      for (uint32_t m = 0; m < nw; ++m) s0 = __dp4a(__ldg(w + m), 0x01010101u, s0);
    } else {
      for (uint32_t m = 0; m < nw; m += 3) {
        const uint32_t w0 = __ldg(w + m), w1 = __ldg(w + m + 1), w2 = __ldg(w + m + 2);
        s0 = __dp4a(w0, 0x01000001u, __dp4a(w1, 0x00010000u, __dp4a(w2, 0x00000100u, s0)));
        s1 = __dp4a(w0, 0x00000100u, __dp4a(w1, 0x01000001u, __dp4a(w2, 0x00010000u, s1)));
        s2 = __dp4a(w0, 0x00010000u, __dp4a(w1, 0x00000100u, __dp4a(w2, 0x01000001u, s2)));
      }
    }
  }
  const uint32_t area = a.f * a.f, half = area / 2u;
  const uint32_t r = (s0 + half) / area;
  if (a.ch == 1u) return r;
  const uint32_t g = (s1 + half) / area, b = (s2 + half) / area;
  return (77u * r + 150u * g + 29u * b + 128u) >> 8;
}

// Luma of four RGB pixels held in three little-endian words
// (R0 G0 B0 R1 | G1 B1 R2 G2 | B2 R3 G3 B3), packed as four bytes.
__device__ __forceinline__ uint32_t luma4(uint32_t w0, uint32_t w1, uint32_t w2) {
  constexpr uint32_t kW = 77u | (150u << 8) | (29u << 16);  // byte 3 weighs 0
  const uint32_t g0 = __dp4a(w0, kW, 128u) >> 8;
  const uint32_t g1 = __dp4a(__byte_perm(w0, w1, 0x0543), kW, 128u) >> 8;
  const uint32_t g2 = __dp4a(__byte_perm(w1, w2, 0x0432), kW, 128u) >> 8;
  const uint32_t g3 = __dp4a(w2 >> 8, kW, 128u) >> 8;
  return g0 | (g1 << 8) | (g2 << 16) | (g3 << 24);
}

// Binomial-weighted sum of B values v[0..B-1]: the weights are symmetric,
// so pairs are added first and multiplied once (half the multiplies).
template <int B, typename F>
__device__ __forceinline__ uint32_t binomial_sum(F v) {
  constexpr int kHalf = (B - 1) / 2;
  uint32_t s = binom(B - 1, kHalf) * v(kHalf);
#pragma unroll
  for (int j = 0; j < kHalf; ++j) s += binom(B - 1, j) * (v(j) + v(B - 1 - j));
  return s;
}

// Advance a flat position (r, x) over rows of width w by `step` = sr rows + sx.
__device__ __forceinline__ void advance(uint32_t& r, uint32_t& x, uint32_t sr, uint32_t sx,
                                        uint32_t w) {
  r += sr;
  x += sx;
  if (x >= w) {
    x -= w;
    ++r;
  }
}

template <int B>
__global__ void __launch_bounds__(kEncThreads, 2) sp_encode_band_kernel(const BandArgs a) {
  constexpr uint32_t kHalf = (B - 1) / 2;
  constexpr uint32_t kShift = 2 * (B - 1);
  constexpr uint32_t kRowsPerItem = 4;  // phase B: rows of V per work item
  extern __shared__ __align__(16) uint8_t enc_smem[];
  const uint32_t frame = blockIdx.y;
  const uint32_t y0 = blockIdx.x * a.band_rows;
  if (y0 >= a.Hr) return;
  const uint32_t y1 = min(a.Hr, y0 + a.band_rows);
  const uint32_t n_px = a.Wr * a.Hr;
  const uint32_t w_lo = (uint32_t)(((uint64_t)y0 * a.Wr + 31u) >> 5);
  const uint32_t w_hi = min(a.n_words, (uint32_t)(((uint64_t)y1 * a.Wr + 31u) >> 5));
  if (w_lo >= w_hi) return;  // the band's words start in an earlier band
  const uint32_t p_last = min(w_hi * 32u, n_px) - 1u;
  const uint32_t nV = p_last / a.Wr - y0 + 1u;  // rows of V this CTA needs
  const uint32_t nG = nV + 2u * kHalf;
  uint8_t* G = enc_smem;
  uint32_t* V = reinterpret_cast<uint32_t*>(enc_smem + a.g_bytes);
  const uint8_t* fs = a.src + (uint64_t)frame * a.src_stride;
  const uint32_t tid = threadIdx.x;

  // A. gray rows y0 - half .. y0 + nV - 1 + half, edge rows replicated.
  // Items are taken kUnroll at a time with all their loads issued first, so
  // each thread keeps several source words in flight.
  constexpr int kUnroll = 4;
  auto clamp_row = [&](uint32_t r) {
    int gy = (int)y0 - (int)kHalf + (int)r;
    return (uint32_t)(gy < 0 ? 0 : (gy >= (int)a.Hr ? (int)a.Hr - 1 : gy));
  };
  const uint32_t* fw = reinterpret_cast<const uint32_t*>(fs);
  if (a.vec4) {
    // four pixels per item from aligned words (f == 1, W % 4 == 0)
    const uint32_t q = a.Wr >> 2;
    uint32_t r = tid / q, k = tid - r * q;
    const uint32_t sr = kEncThreads / q, sk = kEncThreads - sr * q;
    while (r < nG) {
      uint32_t ru[kUnroll], ku[kUnroll], w0[kUnroll], w1[kUnroll], w2[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        ru[u] = r;
        ku[u] = k;
        advance(r, k, sr, sk, q);
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        w0[u] = w1[u] = w2[u] = 0u;
        if (ru[u] < nG) {
          const uint32_t gy = clamp_row(ru[u]);
          if (a.ch == 3u) {
            const uint32_t* w = fw + (uint64_t)gy * q * 3u + 3u * ku[u];
            w0[u] = __ldg(w);
            w1[u] = __ldg(w + 1);
            w2[u] = __ldg(w + 2);
          } else {
            w0[u] = __ldg(fw + (uint64_t)gy * q + ku[u]);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u)
        if (ru[u] < nG)
          *reinterpret_cast<uint32_t*>(G + ru[u] * a.g_pitch + 4u * ku[u]) =
              a.ch == 3u ? luma4(w0[u], w1[u], w2[u]) : w0[u];
    }
  } else if (a.vecf && a.f == 4u) {
    // 4 x 4 blocks from aligned words: 3 words (RGB) or 1 word (gray) per block row
    const uint32_t wpr = a.W * a.ch / 4u;
    uint32_t r = tid / a.Wr, x = tid - r * a.Wr;
    const uint32_t sr = kEncThreads / a.Wr, sx = kEncThreads - sr * a.Wr;
    constexpr int kU = kUnroll / 2;
    while (r < nG) {
      uint32_t ru[kU], xu[kU], w[kU][12];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        ru[u] = r;
        xu[u] = x;
        advance(r, x, sr, sx, a.Wr);
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
#pragma unroll
        for (int m = 0; m < 12; ++m) w[u][m] = 0u;
        if (ru[u] < nG) {
          const uint32_t gy = clamp_row(ru[u]);
          const uint32_t nw = a.ch;  // words per block row: 4 * ch / 4
#pragma unroll
          for (int dy = 0; dy < 4; ++dy) {
            const uint32_t* row = fw + (uint64_t)(gy * 4u + dy) * wpr + (uint64_t)xu[u] * nw;
            w[u][3 * dy] = __ldg(row);
            if (a.ch == 3u) {
              w[u][3 * dy + 1] = __ldg(row + 1);
              w[u][3 * dy + 2] = __ldg(row + 2);
            }
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        if (ru[u] >= nG) continue;
        uint32_t gray;
        if (a.ch == 3u) {
          uint32_t s0 = 0, s1 = 0, s2 = 0;
#pragma unroll
          for (int dy = 0; dy < 4; ++dy) {
            const uint32_t q0 = w[u][3 * dy], q1 = w[u][3 * dy + 1], q2 = w[u][3 * dy + 2];
            s0 = __dp4a(q0, 0x01000001u, __dp4a(q1, 0x00010000u, __dp4a(q2, 0x00000100u, s0)));
            s1 = __dp4a(q0, 0x00000100u, __dp4a(q1, 0x01000001u, __dp4a(q2, 0x00010000u, s1)));
            s2 = __dp4a(q0, 0x00010000u, __dp4a(q1, 0x00000100u, __dp4a(q2, 0x01000001u, s2)));
          }
          gray = (77u * ((s0 + 8u) >> 4) + 150u * ((s1 + 8u) >> 4) + 29u * ((s2 + 8u) >> 4) +
                  128u) >> 8;
        } else {
          uint32_t s0 = 0;
#pragma unroll
          for (int dy = 0; dy < 4; ++dy) s0 = __dp4a(w[u][3 * dy], 0x01010101u, s0);
          gray = (s0 + 8u) >> 4;
        }
        G[ru[u] * a.g_pitch + xu[u]] = (uint8_t)gray;
      }
    }
  } else {
    uint32_t r = tid / a.Wr, x = tid - r * a.Wr;
    const uint32_t sr = kEncThreads / a.Wr, sx = kEncThreads - sr * a.Wr;
    for (; r < nG; advance(r, x, sr, sx, a.Wr)) {
      const uint32_t gy = clamp_row(r);
      G[r * a.g_pitch + x] = (uint8_t)(a.vecf ? reduced_gray_words(a, fs, gy, x)
                                               : reduced_gray(a, fs, gy, x));
    }
  }
  __syncthreads();
  // B. vertical sums over B gray rows, for columns -half .. Wr - 1 + half;
  // an item is kRowsPerItem consecutive rows of one column
  {
    const uint32_t vw = a.v_pitch;
    const uint32_t groups = (nV + kRowsPerItem - 1) / kRowsPerItem;
    uint32_t rg = tid / vw, c = tid - rg * vw;
    const uint32_t sr = kEncThreads / vw, sc = kEncThreads - sr * vw;
    for (; rg < groups; advance(rg, c, sr, sc, vw)) {
      int x = (int)c - (int)kHalf;
      x = x < 0 ? 0 : (x >= (int)a.Wr ? (int)a.Wr - 1 : x);
      const uint32_t r0 = rg * kRowsPerItem;
      const uint8_t* col = G + r0 * a.g_pitch + x;
      uint32_t g[kRowsPerItem + B - 1];
#pragma unroll
      for (uint32_t j = 0; j < kRowsPerItem + B - 1; ++j)
        g[j] = r0 + j < nG ? (uint32_t)col[j * a.g_pitch] : 0u;
#pragma unroll
      for (uint32_t t = 0; t < kRowsPerItem; ++t) {
        const uint32_t s = binomial_sum<B>([&](int j) { return g[t + j]; });
        if (r0 + t < nV) V[(r0 + t) * vw + c] = s;
      }
    }
  }
  __syncthreads();
  const uint32_t lane = tid & 31u, warp = tid >> 5;
  constexpr uint32_t kWarps = kEncThreads / 32;
  uint32_t* out = a.out + (uint64_t)frame * a.out_stride;
  if (a.Wr % 32u == 0u) {
    // C'. words are whole row segments: a lane takes four adjacent pixels
    // (vector loads of V), eight lanes make one word
    constexpr uint32_t kVec = (B + 3 + 3) / 4;  // 16-byte loads covering B + 3 columns
    const uint32_t q_row = a.Wr >> 2;
    const uint32_t n_items = (y1 - y0) * q_row;  // a multiple of 8
    uint32_t i = tid;
    uint32_t r = i / q_row, q = i - r * q_row;
    const uint32_t sr = kEncThreads / q_row, sq = kEncThreads - sr * q_row;
    const uint32_t n_round = (n_items + 31u) & ~31u;
    for (; i < n_round; i += kEncThreads, advance(r, q, sr, sq, q_row)) {
      uint32_t m = 0;
      if (i < n_items) {
        const uint4* vr = reinterpret_cast<const uint4*>(V + r * a.v_pitch + 4u * q);
        uint32_t v[4 * kVec];
#pragma unroll
        for (uint32_t k = 0; k < kVec; ++k) {
          const uint4 t = vr[k];
          v[4 * k] = t.x;
          v[4 * k + 1] = t.y;
          v[4 * k + 2] = t.z;
          v[4 * k + 3] = t.w;
        }
        const uint32_t g4 = *reinterpret_cast<const uint32_t*>(G + (r + kHalf) * a.g_pitch + 4u * q);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const uint32_t s = binomial_sum<B>([&](int j) { return v[t + j]; });
          const uint32_t mean = (s + (1u << (kShift - 1))) >> kShift;
          const int g = (int)((g4 >> (8 * t)) & 255u);
          m |= (g + a.offset > (int)mean ? 1u : 0u) << t;
        }
      }
      uint32_t word = m << (4u * (lane & 7u));
      word |= __shfl_xor_sync(0xffffffffu, word, 1);
      word |= __shfl_xor_sync(0xffffffffu, word, 2);
      word |= __shfl_xor_sync(0xffffffffu, word, 4);
      if ((lane & 7u) == 0u && i < n_items) out[w_lo + i / 8u] = word;
    }
    return;
  }
  // C. one warp per owned word; (y, x) of each lane's pixel kept incrementally
  uint32_t w = w_lo + warp;
  uint32_t p = w * 32u + lane;
  uint32_t y = p / a.Wr, x = p - y * a.Wr;
  const uint32_t sy = (kWarps * 32u) / a.Wr, sx = kWarps * 32u - sy * a.Wr;
  for (; w < w_hi; w += kWarps, p += kWarps * 32u, advance(y, x, sy, sx, a.Wr)) {
    bool bit = false;
    if (p < n_px) {
      const uint32_t r = y - y0;
      const uint32_t* vr = V + r * a.v_pitch + x;  // vr[i] is column x + i - half
      const uint32_t s = binomial_sum<B>([&](int i) { return vr[i]; });
      const uint32_t mean = (s + (1u << (kShift - 1))) >> kShift;
      const int g = (int)G[(r + kHalf) * a.g_pitch + x];
      bit = g + a.offset > (int)mean;
    }
    const uint32_t m = __ballot_sync(0xffffffffu, bit);
    if (lane == 0) out[w] = m;
  }
}

uint32_t plan_smem(uint32_t block, uint32_t Wr, uint32_t th, uint32_t* g_pitch,
                   uint32_t* g_bytes, uint32_t* v_pitch) {
  const uint32_t half = (block - 1) / 2;
  const uint32_t v_rows = th + 1u + 30u / Wr;  // owned words reach at most 31 pixels past
  const uint32_t g_rows = v_rows + 2u * half;
  *g_pitch = (Wr + 3u) & ~3u;
  *g_bytes = (g_rows * *g_pitch + 15u) & ~15u;
  *v_pitch = (Wr + block + 2u + 3u) & ~3u;  // 16-byte rows; the vector loads of
                                             // four pixels read up to Wr + block + 1
  return *g_bytes + v_rows * *v_pitch * 4u;
}

template <int B>
cudaError_t launch_band(const BandArgs& a, uint32_t n, uint32_t smem, cudaStream_t st) {
  const uint32_t bands = (a.Hr + a.band_rows - 1u) / a.band_rows;
  sp_encode_band_kernel<B><<<dim3(bands, n), kEncThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

// Allow every kernel instance the planned shared memory on the current device.
cudaError_t encode_band_init() {
  cudaError_t e = cudaSuccess;
  auto set = [&](const void* k) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEncSmemMax);
  };
  set((const void*)sp_encode_band_kernel<3>);
  set((const void*)sp_encode_band_kernel<5>);
  set((const void*)sp_encode_band_kernel<7>);
  set((const void*)sp_encode_band_kernel<9>);
  set((const void*)sp_encode_band_kernel<11>);
  set((const void*)sp_encode_band_kernel<13>);
  return e;
}

cudaError_t launch_encode_band(const EncodeArgs& e, uint32_t block, cudaStream_t st) {
  BandArgs a{};
  a.src = e.src;
  a.src_stride = e.src_stride;
  a.W = e.W;
  a.ch = e.ch;
  a.f = e.f;
  a.Wr = e.Wr;
  a.Hr = e.Hr;
  a.offset = e.offset;
  a.out = e.out;
  a.out_stride = e.out_stride;
  a.n_words = e.n_words;
  a.vec4 = (e.f == 1u && e.W % 4u == 0u && e.src_stride % 4u == 0u &&
            reinterpret_cast<uintptr_t>(e.src) % 4u == 0u)
               ? 1u
               : 0u;
  a.vecf = (e.f % 4u == 0u && e.W % 4u == 0u && e.src_stride % 4u == 0u &&
            reinterpret_cast<uintptr_t>(e.src) % 4u == 0u) ? 1u : 0u;
  uint32_t th = 32;
  for (; th > 1; th /= 2)
    if (plan_smem(block, a.Wr, th, &a.g_pitch, &a.g_bytes, &a.v_pitch) <= kEncSmemTarget) break;
  const uint32_t smem = plan_smem(block, a.Wr, th, &a.g_pitch, &a.g_bytes, &a.v_pitch);
  a.band_rows = std::min(th, a.Hr);
  cudaError_t err;
  switch (block) {
    case 3: err = launch_band<3>(a, e.n_frames, smem, st); break;
    case 5: err = launch_band<5>(a, e.n_frames, smem, st); break;
    case 7: err = launch_band<7>(a, e.n_frames, smem, st); break;
    case 9: err = launch_band<9>(a, e.n_frames, smem, st); break;
    case 11: err = launch_band<11>(a, e.n_frames, smem, st); break;
    default: err = launch_band<13>(a, e.n_frames, smem, st); break;
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return err;
}

}  // namespace sp

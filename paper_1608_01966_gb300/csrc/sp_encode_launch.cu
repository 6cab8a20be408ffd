// Launch shape of the frame encoder: the reading mode, strips and row chunks.
#include "sp_encode_kernel.cuh"

#include <algorithm>
#include <atomic>

namespace sp {

extern std::atomic<uint64_t> g_launches;

cudaError_t launch_encode(EncodeArgs a, uint32_t block, cudaStream_t st) {
  const bool a8 = reinterpret_cast<uintptr_t>(a.src) % 8u == 0u && a.src_stride % 8u == 0u &&
                  (uint64_t)a.W * a.ch % 8u == 0u && a.Wr % 8u == 0u;
  a.strips = (a.Wr + enc::kStrip - 1u) / enc::kStrip;
  // Which kernel.  Blocks of 3 x 3 pixels and more: a strip's halo rows cost f
  // times as many source rows each, so the band kernel, whose CTAs share them,
  // reads less (128 frames of 960 x 540, f 4: 56 us against 136).  Below that a
  // strip kernel's time goes with the strips walked, the band kernel's with
  // the pixels, so strips have to be filled, to a percentage that depends on how
  // costly a strip's rows are to read and on the block (a chunk walks block + 3
  // rows besides its own).  us, strip / band, n frames of h rows: aligned f 1
  // width 96 b 11 n 128 h 400 27 / 36, 120 b 13 n 24 h 270 RGB 14.7 / 12.7, 160 b
  // 3 n 6 h 270 9.2 / 8.1 but n 24 8.5 / 10.4; aligned f 2 gray 160 b 7 n 96 h 100
  // 17 / 25, b 13 30 / 29, RGB 160 b 13 43 / 32, n 96 h 270 59 / 58, n 128 h 400 b
  // 11 68 / 119; unaligned (plus a clear of the output) f 1 150 b 7 n 24 h 100
  // 10.3 / 9.4, 205 b 3 n 6 h 270 11.5 / 10.5, 230 10.7 / 10.8, gray 481 b 13 n 24
  // h 100 19 / 23, RGB 481 b 7 17 / 21, b 13 27 / 23; f 2 gray 150 b 7 12.8 / 14.7,
  // b 13 19 / 17, 481 b 13 33 / 41, RGB 481 b 7 39 / 38, b 13 62 / 44, but one frame
  // 16 / 37; full strips, 960 x 540 RGB f 1, n 128: 84 / 211.
  const bool tall = block > 7u;
  const uint64_t image_rows = (uint64_t)a.n_frames * a.Hr;
  const uint32_t filled = (uint32_t)((uint64_t)a.Wr * 100u / ((uint64_t)a.strips * enc::kStrip));
  uint32_t need;  // percent; above 100: never
  if (a8) {
    if (a.f == 1u)
      need = image_rows < 4096u ? 70u : (tall ? 60u : 40u);
    else
      need = tall && image_rows < 25000u ? 85u : (a.ch == 1u ? 50u : 60u);
  } else if (a.ch == 1u) {
    if (a.strips > 1u)  // f 2, 252 b 11: n 30 h 200 33 / 29, n 128 h 400 97 / 142
      need = tall && a.f == 2u && image_rows < 25000u ? 65u : 50u;
    else
      need = a.f == 1u ? (tall ? 101u : 95u) : (tall ? 95u : 60u);
  } else if (a.f == 1u) {
    need = tall ? 101u : (a.strips > 1u ? 60u : 95u);
  } else {
    // at most 304 warps of 4 rows: two per SM
    const uint64_t warps = (uint64_t)a.n_frames * a.strips * ((a.Hr + 3u) / 4u);
    need = tall || warps > 304u ? 101u : (a.strips > 1u ? 65u : 85u);
  }
  if (!a8 && a.f == 1u && a.W % 4u == 0u && a.src_stride % 4u == 0u &&
      reinterpret_cast<uintptr_t>(a.src) % 4u == 0u) {
    // rows of whole words: the band kernel reads four pixels at a time (us,
    // strip / band, b 7: gray 300 n 12 h 100 9.6 / 8.8, n 60 h 270 19 / 21, RGB
    // 27 / 23, 404 n 40 19 / 23, 644 n 40 h 360 27 / 37)
    need = std::max(need, image_rows < 4096u ? 101u : (a.ch == 1u ? 60u : 80u));
  }
  if (a.f >= 3u || a.Wr < 8u || filled < need) return launch_encode_band(a, block, st);
  // Rows per chunk: every chunk reads block - 1 rows besides its own, a chunk
  // per warp; the fewest rows walked by the warps of a full machine in whole
  // waves (16 warps resident per SM, at 128 registers a thread)
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const uint64_t resident = 16ull * (uint64_t)std::max(1, sms);
  uint64_t best = ~0ull;
  a.rows = a.Hr;
  for (uint32_t chunks = 1; chunks <= a.Hr; ++chunks) {
    const uint32_t rows = (a.Hr + chunks - 1u) / chunks;
    if (chunks > 1u && rows < 4u) break;
    const uint64_t units = (uint64_t)a.n_frames * a.strips * ((a.Hr + rows - 1u) / rows);
    const uint64_t cost = (units + resident - 1u) / resident * (rows + block + 3u);
    if (cost < best) {
      best = cost;
      a.rows = rows;
    }
  }
  a.chunks = (a.Hr + a.rows - 1u) / a.rows;
  const uint64_t units = (uint64_t)a.n_frames * a.strips * a.chunks;
  if (units > 0x7fffffffull) return cudaErrorInvalidValue;
  a.units = (uint32_t)units;
  if (a.Wr % 8u != 0u) {
    // rows that start inside a byte are OR'ed into words
    e = cudaMemset2DAsync(a.out, a.out_stride * 4u, 0, (size_t)a.n_words * 4u, a.n_frames, st);
    if (e != cudaSuccess) return e;
  }
  switch (block) {
    case 3: e = enc::launch_block<3>(a, a8, st); break;
    case 5: e = enc::launch_block<5>(a, a8, st); break;
    case 7: e = enc::launch_block<7>(a, a8, st); break;
    case 9: e = enc::launch_block<9>(a, a8, st); break;
    case 11: e = enc::launch_block<11>(a, a8, st); break;
    default: e = enc::launch_block<13>(a, a8, st); break;
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return e;
}

}  // namespace sp

// Launch shape of the frame encoder: the reading mode, strips and row chunks.
#include "sp_encode_kernel.cuh"
#include "sp_encode_rule.h"

#include <algorithm>
#include <atomic>

namespace sp {

extern std::atomic<uint64_t> g_launches;

cudaError_t launch_encode(EncodeArgs a, uint32_t block, cudaStream_t st) {
  const bool a8 = reinterpret_cast<uintptr_t>(a.src) % 8u == 0u && a.src_stride % 8u == 0u &&
                  (uint64_t)a.W * a.ch % 8u == 0u && a.Wr % 8u == 0u;
  a.strips = (a.Wr + kEncodeStrip - 1u) / kEncodeStrip;
  // asked for where it is needed: the two calls take half a microsecond
  int sms = 0;
  auto ask_sms = [&]() {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e != cudaSuccess ? e : cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  };
  cudaError_t e = cudaSuccess;
  if (!a8 && a.ch == 3u && a.f == 2u && (e = ask_sms()) != cudaSuccess) return e;
  const bool words = a.src_stride % 4u == 0u && reinterpret_cast<uintptr_t>(a.src) % 4u == 0u;
  if (!encode_in_strips({a.W, a.ch, a.f, a.Wr, a.Hr, block, a.n_frames, a8, words, (uint32_t)sms}))
    return launch_encode_band(a, block, st);
  if (sms == 0 && (e = ask_sms()) != cudaSuccess) return e;
  // Rows per chunk: every chunk reads block - 1 rows besides its own, a chunk
  // per warp; the fewest rows walked by the warps of a full machine in whole
  // waves (16 warps resident per SM, at 128 registers a thread)
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

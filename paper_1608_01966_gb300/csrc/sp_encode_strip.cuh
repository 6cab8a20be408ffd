// The frame encoder's kernel arguments and launchers (strip kernels in
// sp_encode_kernel.cuh, one translation unit per pair of window sizes; band
// kernels in sp_encode_band.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sp {

// Weights of the encoder's window: row n of Pascal's triangle.
__host__ __device__ constexpr uint32_t binom(uint32_t n, uint32_t k) {
  uint64_t r = 1;
  for (uint32_t i = 1; i <= k; ++i) r = r * (n - k + i) / i;
  return (uint32_t)r;
}

struct EncodeArgs {
  const uint8_t* src;
  uint64_t src_stride;   // bytes between frames
  uint64_t frame_bytes;  // bytes of one frame
  uint32_t W, ch, f;     // source width, channels, reduction factor
  uint32_t Wr, Hr;       // output size
  int32_t offset;        // -256..256
  uint32_t* out;
  uint64_t out_stride;   // words between encoded frames
  uint32_t n_words;
  uint32_t n_frames;
  uint32_t strips, chunks, rows;  // strips of a row, row chunks of a frame, rows per chunk
  uint32_t units;                 // n_frames * chunks * strips, one per warp
};

// Encode a.n_frames frames with window size `block` (odd, 3..13) on st;
// strips, chunks, rows and units are filled in here.
cudaError_t launch_encode(EncodeArgs a, uint32_t block, cudaStream_t st);

// The same by bands of rows in shared memory (sp_encode_band.cu): any
// reduction and width.
cudaError_t encode_band_init();  // once per device, before its first launch
cudaError_t launch_encode_band(const EncodeArgs& a, uint32_t block, cudaStream_t st);

}  // namespace sp

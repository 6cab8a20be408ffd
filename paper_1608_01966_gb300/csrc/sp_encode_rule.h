// Which of the encoder's two kernels takes a call: plain C++, no device code.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace sp {

constexpr uint32_t kEncodeStrip = 240;  // output columns of a strip (one warp)

struct EncodeShape {
  uint32_t W, ch, f;    // source width, channels, reduction factor
  uint32_t Wr, Hr;      // output size
  uint32_t block;       // window size
  uint32_t n_frames;
  bool a8;              // rows, frames and strips on 8-byte boundaries, output rows whole bytes
  bool words;           // rows and frames on 4-byte boundaries
  uint32_t sms;         // of unaligned RGB halved; else it may be 0
};

// Whether the strip kernel takes the call (else the band kernel).  Blocks of 3 x
// 3 pixels and more: a strip's halo rows cost f times as many source rows each,
// so the band kernel, whose CTAs share them, reads less (128 frames of 960 x
// 540, f 4: 56 us against 136).  Below that a
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
inline bool encode_in_strips(const EncodeShape& e) {
  const uint32_t strips = (e.Wr + kEncodeStrip - 1u) / kEncodeStrip;
  const bool tall = e.block > 7u;
  const uint64_t image_rows = (uint64_t)e.n_frames * e.Hr;
  const uint32_t filled = (uint32_t)((uint64_t)e.Wr * 100u / ((uint64_t)strips * kEncodeStrip));
  uint32_t need;  // percent; above 100: never
  if (e.a8) {
    if (e.f == 1u)
      need = image_rows < 4096u ? 70u : (tall ? 60u : 40u);
    else
      need = tall && image_rows < 25000u ? 85u : (e.ch == 1u ? 50u : 60u);
  } else if (e.ch == 1u) {
    if (strips > 1u)  // f 2, 252 b 11: n 30 h 200 33 / 29, n 128 h 400 97 / 142
      need = tall && e.f == 2u && image_rows < 25000u ? 65u : 50u;
    else
      need = e.f == 1u ? (tall ? 101u : 95u) : (tall ? 95u : 60u);
  } else if (e.f == 1u) {
    need = tall ? 101u : (strips > 1u ? 60u : 95u);
  } else {
    // at most two warps of 4 rows per SM
    const uint64_t warps = (uint64_t)e.n_frames * strips * ((e.Hr + 3u) / 4u);
    need = tall || warps > 2ull * e.sms ? 101u : (strips > 1u ? 65u : 85u);
  }
  if (!e.a8 && e.f == 1u && e.W % 4u == 0u && e.words) {
    // rows of whole words: the band kernel reads four pixels at a time (us,
    // strip / band, b 7: gray 300 n 12 h 100 9.6 / 8.8, n 60 h 270 19 / 21, RGB
    // 27 / 23, 404 n 40 19 / 23, 644 n 40 h 360 27 / 37)
    need = std::max(need, image_rows < 4096u ? 101u : (e.ch == 1u ? 60u : 80u));
  }
  return e.f <= 2u && e.Wr >= 8u && filled >= need;
}

}  // namespace sp

// Frame encoder on the GPU (Section 2 and "Adaptive Video Encoder" in
// Section 3.1): colour frames -> reduction -> gray -> adaptive Gaussian
// threshold -> packed input bits, in one kernel (sp_encode_strip.cuh), plus
// the sp_encoder_* ABI.
#include "sp_internal.h"

#include "sp_encode_strip.cuh"

#include <algorithm>
#include <chrono>
#include <thread>

using namespace sp::rt;

namespace {

constexpr uint32_t kEncChunkFrames = 32;          // frames per encode + SP step
constexpr uint64_t kEncStageBytes = 64ull << 20;  // host path: raw bytes per chunk

struct EncPlan {
  uint32_t Wr = 0, Hr = 0, n_words = 0;
  uint64_t src_bytes = 0;
};

sp_status validate_encoder(const sp_encoder_config* c, EncPlan* p) {
  if (!c) return fail(SP_EINVAL, "NULL encoder config");
  if (c->src_w == 0 || c->src_h == 0 || c->src_w > 65535u || c->src_h > 65535u)
    return fail(SP_EINVAL, "source size %ux%u outside 1..65535", c->src_w, c->src_h);
  if (c->channels != 1 && c->channels != 3)
    return fail(SP_EINVAL, "channels %u (1 or 3)", c->channels);
  if (c->reduce < 1 || c->reduce > 8) return fail(SP_EINVAL, "reduce %u outside 1..8", c->reduce);
  if (c->block < 3 || c->block > 13 || c->block % 2 == 0)
    return fail(SP_EINVAL, "block %u (odd, 3..13)", c->block);
  if (c->reserved[0] || c->reserved[1]) return fail(SP_EINVAL, "reserved fields must be zero");
  const uint32_t Wr = c->src_w / c->reduce, Hr = c->src_h / c->reduce;
  if (Wr == 0 || Hr == 0) return fail(SP_EINVAL, "reduction leaves an empty frame");
  if ((uint64_t)Wr * Hr >= (1ull << 31)) return fail(SP_EINVAL, "output frame too large");
  p->Wr = Wr;
  p->Hr = Hr;
  p->n_words = (uint32_t)(((uint64_t)Wr * Hr + 31u) / 32u);
  p->src_bytes = (uint64_t)c->src_w * c->src_h * c->channels;
  // the widest output the encoder takes (a row of V sums of the widest
  // window in 200 KB of shared memory set this bound; results never depended on it)
  const uint32_t g_rows = 2u + 30u / Wr + (c->block - 1u), v_rows = 2u + 30u / Wr;
  const uint64_t smem = (uint64_t)((g_rows * ((Wr + 3u) & ~3u) + 15u) & ~15u) +
                        (uint64_t)v_rows * ((Wr + c->block + 5u) & ~3u) * 4u;
  if (smem > (200u << 10)) return fail(SP_EINVAL, "output width %u too large", Wr);
  return SP_OK;
}

}  // namespace

struct sp_encoder {
  sp_encoder_config cfg{};
  EncPlan plan;
  int device = 0;
  uint32_t timeout_ms = 10000;
  cudaStream_t stream = nullptr, s_in = nullptr, s_out = nullptr;
  cudaEvent_t ev_h2d[kSlots] = {}, ev_comp[kSlots] = {}, ev_d2h[kSlots] = {}, ev_tail = nullptr;
  uint32_t* d_bits = nullptr;  // kEncChunkFrames encoded frames
  uint8_t* d_raw = nullptr;    // host path: [kSlots][chunk][src_bytes]
  uint32_t raw_chunk = 0;
  uint32_t* d_masks = nullptr;  // host path: [kSlots][kEncChunkFrames][mask_words]
  uint32_t mask_words = 0;
};

namespace {

void free_encoder(sp_encoder* e) {
  if (!e) return;
  DeviceGuard g(e->device);
  if (e->stream) cudaStreamSynchronize(e->stream);
  if (e->s_in) cudaStreamSynchronize(e->s_in);
  if (e->s_out) cudaStreamSynchronize(e->s_out);
  for (int i = 0; i < kSlots; ++i) {
    if (e->ev_h2d[i]) cudaEventDestroy(e->ev_h2d[i]);
    if (e->ev_comp[i]) cudaEventDestroy(e->ev_comp[i]);
    if (e->ev_d2h[i]) cudaEventDestroy(e->ev_d2h[i]);
  }
  if (e->ev_tail) cudaEventDestroy(e->ev_tail);
  if (e->d_bits) cudaFree(e->d_bits);
  if (e->d_raw) cudaFree(e->d_raw);
  if (e->d_masks) cudaFree(e->d_masks);
  if (e->stream) cudaStreamDestroy(e->stream);
  if (e->s_in) cudaStreamDestroy(e->s_in);
  if (e->s_out) cudaStreamDestroy(e->s_out);
  delete e;
}

sp_status enqueue_encode(sp_encoder* e, const uint8_t* d_src, uint32_t n, uint64_t src_stride,
                         uint32_t* d_bits, uint64_t bits_stride, cudaStream_t st) {
  const EncPlan& p = e->plan;
  sp::EncodeArgs a{};
  a.W = e->cfg.src_w;
  a.ch = e->cfg.channels;
  a.f = e->cfg.reduce;
  a.Wr = p.Wr;
  a.Hr = p.Hr;
  // gray and mean lie in 0..255: past these the offset decides alone
  a.offset = std::max(-256, std::min(256, e->cfg.offset));
  a.n_words = p.n_words;
  a.frame_bytes = p.src_bytes;
  a.src_stride = src_stride;
  a.out_stride = bits_stride;
  for (uint32_t f0 = 0; f0 < n; f0 += 65535u) {
    a.n_frames = std::min(n - f0, 65535u);
    a.src = d_src + (uint64_t)f0 * src_stride;
    a.out = d_bits + (uint64_t)f0 * bits_stride;
    SP_CUDA(sp::launch_encode(a, e->cfg.block, st));
  }
  return SP_OK;
}

cudaStream_t pick_stream(sp_encoder* e, void* stream) {
  return stream ? static_cast<cudaStream_t>(stream) : e->stream;
}

sp_status check_handle(sp_encoder* e, sp_handle* h, uint32_t* mask_words) {
  sp_info info{};
  const sp_status s = sp_get_info(h, &info);
  if (s != SP_OK) return s;
  if (info.input_bits != (uint64_t)e->plan.Wr * e->plan.Hr)
    return fail(SP_EINVAL, "the SP takes %llu input bits, the encoder makes %ux%u",
                (unsigned long long)info.input_bits, e->plan.Wr, e->plan.Hr);
  if (info.device != e->device) return fail(SP_EINVAL, "encoder and SP on different devices");
  *mask_words = info.mask_words;
  return SP_OK;
}

sp_status ensure_bits(sp_encoder* e) {
  if (!e->d_bits)
    SP_CUDA(device_malloc((void**)&e->d_bits, (size_t)kEncChunkFrames * e->plan.n_words * 4));
  return SP_OK;
}

}  // namespace

SP_API sp_status sp_encoder_config_init(sp_encoder_config* cfg) {
  if (!cfg) return fail(SP_EINVAL, "NULL argument");
  *cfg = sp_encoder_config{};
  cfg->src_w = 960;
  cfg->src_h = 540;
  cfg->channels = 3;
  cfg->reduce = 1;
  cfg->block = 11;
  cfg->offset = 2;
  return SP_OK;
}

SP_API sp_status sp_encoder_create(const sp_encoder_config* cfg, sp_encoder** out) {
  if (!out) return fail(SP_EINVAL, "NULL argument");
  *out = nullptr;
  EncPlan plan;
  sp_status s = validate_encoder(cfg, &plan);
  if (s != SP_OK) return s;
  sp_encoder* e = new sp_encoder();
  e->cfg = *cfg;
  e->plan = plan;
  e->timeout_ms = default_timeout_ms();
  cudaError_t err = cudaGetDevice(&e->device);
  if (err == cudaSuccess) err = sp::encode_band_init();
  if (err == cudaSuccess) err = cudaStreamCreateWithFlags(&e->stream, cudaStreamNonBlocking);
  if (err != cudaSuccess) {
    free_encoder(e);
    return fail(SP_ECUDA, "encoder set-up: %s", cudaGetErrorString(err));
  }
  *out = e;
  return SP_OK;
}

SP_API void sp_encoder_destroy(sp_encoder* e) { free_encoder(e); }

SP_API sp_status sp_encoder_get_info(const sp_encoder* e, sp_encoder_info* out) {
  if (!e || !out) return fail(SP_EINVAL, "NULL argument");
  out->out_w = e->plan.Wr;
  out->out_h = e->plan.Hr;
  out->out_bits = (uint64_t)e->plan.Wr * e->plan.Hr;
  out->out_words = e->plan.n_words;
  out->src_bytes = e->plan.src_bytes;
  return SP_OK;
}

SP_API sp_status sp_encode_device(sp_encoder* e, const uint8_t* d_src, uint32_t n_frames,
                                  uint64_t src_stride, uint32_t* d_bits, uint64_t bits_stride,
                                  void* stream) {
  if (!e || ((!d_src || !d_bits) && n_frames)) return fail(SP_EINVAL, "NULL argument");
  if (n_frames == 0) return SP_OK;
  if (src_stride < e->plan.src_bytes) return fail(SP_EINVAL, "source stride below the frame size");
  if (bits_stride < e->plan.n_words) return fail(SP_EINVAL, "bit stride below %u words", e->plan.n_words);
  if (reinterpret_cast<uintptr_t>(d_bits) % 4u) return fail(SP_EINVAL, "d_bits not 4-byte aligned");
  DeviceGuard g(e->device);
  return enqueue_encode(e, d_src, n_frames, src_stride, d_bits, bits_stride, pick_stream(e, stream));
}

SP_API sp_status sp_encode_compute_device(sp_encoder* e, sp_handle* h, const uint8_t* d_src,
                                          uint32_t n_frames, uint64_t src_stride, int learn,
                                          uint32_t* d_active_masks, void* stream) {
  if (!e || !h || (!d_src && n_frames)) return fail(SP_EINVAL, "NULL argument");
  if (n_frames == 0) return SP_OK;
  if (src_stride < e->plan.src_bytes) return fail(SP_EINVAL, "source stride below the frame size");
  if (reinterpret_cast<uintptr_t>(d_active_masks) % 4u)
    return fail(SP_EINVAL, "d_active_masks not 4-byte aligned");
  uint32_t mw = 0;
  sp_status s = check_handle(e, h, &mw);
  if (s != SP_OK) return s;
  DeviceGuard g(e->device);
  s = ensure_bits(e);
  if (s != SP_OK) return s;
  cudaStream_t st = pick_stream(e, stream);
  for (uint32_t f0 = 0; f0 < n_frames; f0 += kEncChunkFrames) {
    const uint32_t nf = std::min(n_frames - f0, kEncChunkFrames);
    s = enqueue_encode(e, d_src + (uint64_t)f0 * src_stride, nf, src_stride, e->d_bits,
                       e->plan.n_words, st);
    if (s != SP_OK) return s;
    s = sp_compute_frames_device(h, e->d_bits, nf, e->plan.n_words, learn,
                                 d_active_masks ? d_active_masks + (uint64_t)f0 * mw : nullptr, st);
    if (s != SP_OK) return s;
  }
  return SP_OK;
}

SP_API sp_status sp_encode_compute(sp_encoder* e, sp_handle* h, const uint8_t* h_src,
                                   uint32_t n_frames, int learn, uint32_t* h_active_masks) {
  if (!e || !h || (!h_src && n_frames)) return fail(SP_EINVAL, "NULL argument");
  if (n_frames == 0) return SP_OK;
  uint32_t mw = 0;
  sp_status s = check_handle(e, h, &mw);
  if (s != SP_OK) return s;
  DeviceGuard g(e->device);
  s = ensure_bits(e);
  if (s != SP_OK) return s;
  const uint64_t fb = e->plan.src_bytes;
  if (!e->d_raw) {
    e->raw_chunk = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(kEncChunkFrames, kEncStageBytes / fb));
    SP_CUDA(device_malloc((void**)&e->d_raw, (size_t)kSlots * e->raw_chunk * fb));
    SP_CUDA(cudaStreamCreateWithFlags(&e->s_in, cudaStreamNonBlocking));
    SP_CUDA(cudaStreamCreateWithFlags(&e->s_out, cudaStreamNonBlocking));
    SP_CUDA(cudaEventCreateWithFlags(&e->ev_tail, cudaEventDisableTiming));
    for (int i = 0; i < kSlots; ++i) {
      SP_CUDA(cudaEventCreateWithFlags(&e->ev_h2d[i], cudaEventDisableTiming));
      SP_CUDA(cudaEventCreateWithFlags(&e->ev_comp[i], cudaEventDisableTiming));
      SP_CUDA(cudaEventCreateWithFlags(&e->ev_d2h[i], cudaEventDisableTiming));
      SP_CUDA(cudaEventRecord(e->ev_comp[i], e->stream));
      SP_CUDA(cudaEventRecord(e->ev_d2h[i], e->stream));
    }
  }
  if (h_active_masks && mw > e->mask_words) {
    if (e->d_masks) {
      SP_CUDA(cudaStreamSynchronize(e->s_out));
      cudaFree(e->d_masks);
      e->d_masks = nullptr;
    }
    SP_CUDA(device_malloc((void**)&e->d_masks, (size_t)kSlots * e->raw_chunk * mw * 4));
    e->mask_words = mw;
  }
  const uint32_t chunk = e->raw_chunk;
  for (uint32_t f0 = 0, ci = 0; f0 < n_frames; f0 += chunk, ++ci) {
    const int slot = (int)(ci % kSlots);
    const uint32_t nf = std::min(n_frames - f0, chunk);
    uint8_t* raw = e->d_raw + (size_t)slot * chunk * fb;
    uint32_t* masks = h_active_masks ? e->d_masks + (size_t)slot * chunk * mw : nullptr;
    // copy in once the work that read this slot two chunks ago is done
    SP_CUDA(cudaStreamWaitEvent(e->s_in, e->ev_comp[slot], 0));
    SP_CUDA(cudaMemcpyAsync(raw, h_src + (uint64_t)f0 * fb, (size_t)nf * fb,
                            cudaMemcpyHostToDevice, e->s_in));
    SP_CUDA(cudaEventRecord(e->ev_h2d[slot], e->s_in));
    SP_CUDA(cudaStreamWaitEvent(e->stream, e->ev_h2d[slot], 0));
    SP_CUDA(cudaStreamWaitEvent(e->stream, e->ev_d2h[slot], 0));
    s = sp_encode_compute_device(e, h, raw, nf, fb, learn, masks, e->stream);
    if (s != SP_OK) return s;
    SP_CUDA(cudaEventRecord(e->ev_comp[slot], e->stream));
    if (h_active_masks) {
      SP_CUDA(cudaStreamWaitEvent(e->s_out, e->ev_comp[slot], 0));
      SP_CUDA(cudaMemcpyAsync(h_active_masks + (uint64_t)f0 * mw, masks, (size_t)nf * mw * 4,
                              cudaMemcpyDeviceToHost, e->s_out));
      SP_CUDA(cudaEventRecord(e->ev_d2h[slot], e->s_out));
    }
  }
  // the SP's stream (now the encoder's) waits for the last copy out, so the
  // handle's bounded wait covers everything
  SP_CUDA(cudaEventRecord(e->ev_tail, e->s_out));
  SP_CUDA(cudaStreamWaitEvent(e->stream, e->ev_tail, 0));
  return sp_sync(h);
}

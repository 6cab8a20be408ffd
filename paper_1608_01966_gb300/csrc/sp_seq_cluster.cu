// Frame sequences of one Spatial Pooler in a single persistent launch: the
// SP state lives in the shared memory of one thread-block cluster for the
// whole sequence.
//
// A sequence with learning is inherently serial (frame t+1 reads the
// permanences frame t wrote), so one SP is bound by the latency of a frame's
// chain, not by bandwidth.  A cluster of Q CTAs loads the state once -- CTA q
// owns columns [q*Cq, (q+1)*Cq) -- and loops over the frames.  16 compute
// warps walk the chain; four helper warps keep everything else off it (the
// next frame's input band by cp.async into the other of two buffers, the
// masks and overlap records, clearing what later frames count into).  A frame:
//
//   1. the band of input words the CTA's pools cover is waited for;
//   2. Alg. 1, each warp its own columns; counts of at least min_overlap go to
//      shared memory as 16-bit values; CTA barrier;
//   3. the CTA pushes its counts to every other CTA of the cluster (st.async,
//      completing on the receiver's mbarrier) and waits for theirs: one
//      one-way trip, where a cluster barrier followed by reads of remote
//      memory costs a barrier and a round trip;
//   4. global inhibition: a histogram of all counts in shared memory, barrier,
//      then every warp finds the k-th largest count (32 bins a step from the
//      largest count down) and all winners of its CTA by itself; local
//      inhibition: every column is ranked against its neighbours' counts by a
//      few lanes of the warp that owns it, barrier;
//   5. Section 1.1: the CTA's i-th winner is learnt by warp i % 16 (winners
//      are neighbours, so dealing them out is what keeps one warp from doing
//      them all), the frame's band still in place; barrier.
//
// A cluster of one CTA (small SPs) has no step 3: its warps add their counts
// to the histogram as they publish them.
//
// us per learning frame, with a cluster barrier and remote reads in place of
// step 3, one warp deciding for the CTA and every CTA ranking all columns of
// local inhibition / as here: 1024 x 256 on 960 x 540 4.9 / 3.0 (window), 4096 x
// 64 local of radius 4 37.3 / 6.7 (window), 4096 x 256 13.9 (a kernel per frame:
// the pools do not fit) / 6.7 (windowL2), 256 x 16 2.60 / 2.02 (one CTA).
//
// Three forms of the state:
//   pools     input indices and fp32 permanences in shared memory; a column's
//             pool is read four synapses per lane (S % 4 == 0), several
//             columns side by side in a warp when pools are small;
//   window    (frames a multiple of 32 pixels wide whose ascending pools fit
//             64 x 64 boxes) a 64 x 64 bitmap of each column's connected
//             synapses: a column is 64 row segments of funnel shift, AND and
//             population count, whatever its pool's size.  Band rows are
//             padded to an odd number of words, so that the 32 rows a warp
//             reads lie in 32 banks.  Permanences and 16-bit positions of the
//             synapses in their boxes are kept beside it in shared memory;
//   windowL2  the same without them: learning reads the pools and permanences
//             of the frame's winners from global memory (L2).
//
// Non-unit boosts make the overlaps fp32 values: then every CTA publishes its
// boosted overlaps, a cluster barrier orders them, and every CTA gathers all
// of them and runs Alg. 2 on its own.
//
// Counts are double-buffered by frame parity: a CTA sends frame t+2's counts
// only after it has received frame t+1's from everyone, and those are sent
// after the sender is done with frame t's.
//
// Waits are bounded (a.wait_ns of %globaltimer, 1 s by default): when one
// expires, the CTA learns nothing from that frame and its loop ends at the next
// B1.  Every CTA reaches the cluster barrier at the end (the others after their
// own limit).  There each CTA tells how many frames' counts it has sent, so one
// that gave up knows what is still on its way to its shared memory and waits
// for just that before it leaves.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>

#include "../../include/sp.h"
#include "sp_device.cuh"
#include "sp_kernels.cuh"

namespace cg = cooperative_groups;

namespace sp {

extern std::atomic<uint64_t> g_launches;

namespace {

using dev::kFull;
using dev::learn_one;

constexpr uint32_t kSeqWarps = kSeqThreads / 32;   // compute warps
constexpr uint32_t kSeqHelpers = 128;              // threads of the helper warps
constexpr int kSeqCols = 4;   // window forms: columns a warp counts side by side
constexpr unsigned long long kSeqDrainNs = 1000000000ull;  // bound of drain_counts' waits
constexpr uint32_t kBoxWords = 128;  // bitmap words of a 64 x 64 box

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

// Wait (at most about `ns`; ONCE: only look) for the phase with this parity;
// with CLUSTER, what other CTAs of the cluster sent with it is visible after.
template <bool CLUSTER, bool ONCE = false>
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, unsigned long long ns) {
  uint32_t ok;
  if (ONCE) {
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0u;
  }
  unsigned long long t0 = 0;
  for (uint32_t i = 0;; ++i) {
    if (CLUSTER)
      asm volatile(
          "{\n.reg .pred p;\n"
          "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
          "selp.b32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(smem_u32(bar)), "r"(parity)
          : "memory");
    else
      asm volatile(
          "{\n.reg .pred p;\n"
          "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
          "selp.b32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(smem_u32(bar)), "r"(parity)
          : "memory");
    if (ok) return true;
    if ((i & 63u) == 0u) {
      const unsigned long long t = now_ns();
      if (i == 0u)
        t0 = t;
      else if (t - t0 > ns)
        return false;
    }
  }
}

// The shared::cluster address of `saddr` (this CTA's shared memory) in CTA `rank`.
__device__ __forceinline__ uint32_t peer_addr(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}

__device__ __forceinline__ void send16(uint32_t dst, const uint4& v, uint32_t bar) {
  asm volatile(
      "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, "
      "[%5];\n" ::"r"(dst),
      "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
      : "memory");
}

// This helper thread's share of copying `rows` rows of `len` consecutive words
// from src to a band whose rows are `pitch` words apart; its arrival on bar
// follows its copies.
__device__ __forceinline__ void copy_band(uint32_t* dst, const uint32_t* src, uint32_t rows,
                                          uint32_t len, uint32_t pitch, uint64_t* bar) {
  const uint32_t h = threadIdx.x - kSeqThreads;
  const uint32_t dr = kSeqHelpers / len, dx = kSeqHelpers - dr * len;
  uint32_t r = h / len, x = h - r * len;
  const uint32_t n = rows * len;
  for (uint32_t i = h; i < n; i += kSeqHelpers) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(dst + r * pitch + x)),
                 "l"(src + i)
                 : "memory");
    r += dr;
    x += dx;
    if (x >= len) {
      x -= len;
      ++r;
    }
  }
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void compute_sync() {
  asm volatile("bar.sync 2, %0;\n" ::"n"(kSeqThreads) : "memory");
}

// What the other CTAs of the cluster still send to a CTA whose wait for counts
// gave up, by one of its warps: it sent *sent frames' counts (`bytes` each to
// every other CTA), and its barriers expect as many from every other; those
// were waited for but the last.  A CTA sends a frame's counts after it has
// everyone's of the frame before, so the others sent one frame less, as many,
// or one more.  (Shared-memory addresses and a loop over the two barriers: as
// pointers and straight code this cost the loop over the frames 2 %.)
__device__ __forceinline__ void drain_counts(uint32_t cnt_bar, uint32_t sent, uint32_t bytes) {
  uint32_t n, m, Q;
  asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(n) : "r"(sent) : "memory");
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;\n" : "=r"(Q));
  const uint32_t lane = threadIdx.x & 31u;
  const bool peer = lane < Q;  // at most kSeqMaxCluster
  asm volatile("ld.shared::cluster.u32 %0, [%1];\n"
               : "=r"(m)
               : "r"(peer_addr(sent, peer ? lane : 0u))
               : "memory");
  const uint32_t fewer = __popc(__ballot_sync(kFull, peer && m < n));
  const uint32_t more = __popc(__ballot_sync(kFull, peer && m > n));
  if (lane != 0u) return;
  for (uint32_t k = 0; k < 2u; ++k) {  // frames n - 1 and n
    if (k ? more == 0u : n == 0u) continue;
    const uint32_t f = n + k - 1u, bar = cnt_bar + 8u * (f & 1u), miss = (k ? more : fewer) * bytes;
    if (k)  // not armed yet: what is on its way
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(miss)
                   : "memory");
    else if (miss)  // armed for everyone's: less what nobody will send
      asm volatile("mbarrier.complete_tx.relaxed.cluster.shared::cta.b64 [%0], %1;\n" ::"r"(bar),
                   "r"(miss)
                   : "memory");
    const unsigned long long t0 = now_ns();
    uint32_t ok = 0u;
    while (!ok && now_ns() - t0 < kSeqDrainNs)
      asm volatile(
          "{\n.reg .pred p;\n"
          "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
          "selp.b32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(bar), "r"((f >> 1) & 1u)
          : "memory");
  }
}

// Words of one frame's histogram: bins 0..S, bin 0 the largest count.
__host__ __device__ __forceinline__ uint32_t hist_words(uint32_t S) { return (S + 4u) & ~3u; }

// Shared-memory layout of one CTA (all offsets in 4-byte words).
struct SeqLayout {
  uint32_t bits, at, org, idx, perm, boost, band, cnt, hist, mask, dirty, ov, all, shist, smask, total;
  __host__ __device__ SeqLayout(uint32_t form, uint32_t Q, uint32_t Cq, uint32_t S,
                                uint32_t band_max, uint32_t C) {
    const uint32_t CqS = Cq * S;
    uint32_t o = 0;
    auto part = [&](uint32_t words) {
      const uint32_t at0 = o;
      o += (words + 3u) & ~3u;  // 16-byte aligned parts
      return at0;
    };
    const bool window = form != kSeqPools;
    bits = part(window ? Cq * kBoxWords : 0u);
    at = part(window ? Cq : 0u);
    org = part(window ? Cq : 0u);
    // pools: 32-bit indices; window: 16-bit positions in the box
    idx = part(form == kSeqPools ? CqS : (form == kSeqWindow ? (CqS + 1u) / 2u : 0u));
    perm = part(form != kSeqWindowL2 ? CqS : 0u);
    boost = part(Cq);
    band = part(2u * band_max);
    mask = part(3u * (Cq / 32u));            // three frames' winner masks in turn
    dirty = part(Cq / 32u);
    const uint32_t rest = o;
    cnt = part(2u * (Q * Cq / 2u));          // [2][Q * Cq] 16-bit counts
    hist = part(3u * hist_words(S));         // three frames' histograms in turn
    const uint32_t unit_end = o;
    o = rest;  // non-unit boosts use the same memory for fp32 overlaps
    ov = part(2u * Cq);
    all = part(C);
    shist = part((S + 1u) > 256u ? (S + 1u) : 256u);
    smask = part(2u * ((C + 31u) / 32u));    // mask words, and tied columns
    o = o > unit_end ? o : unit_end;
    total = o;
  }
};

template <int N>
struct IntC {
  static constexpr int value = N;
};

// ONCE: a bound of less than a microsecond, which the clock may not resolve, is
// no wait at all; its own instance, since a choice between two mbarrier
// instructions in the chain of a frame took 3 % (1024 x 256).
template <uint32_t FORM, bool ONCE>
__global__ void __launch_bounds__(kSeqThreads + kSeqHelpers, 1) sp_seq_cluster_kernel(const SeqArgs a) {
  constexpr bool kWindow = FORM != kSeqPools;
  constexpr bool kPermSmem = FORM != kSeqWindowL2;
  constexpr uint32_t kAll = kSeqThreads + kSeqHelpers;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ uint32_t sh[2 * kSeqWarps];
  // non-unit boosts: select_threshold's; else [0] is set once a wait has given
  // up, [1] is the number of frames whose counts this CTA has sent
  __shared__ uint32_t s2[2];
  __shared__ uint32_t s_n;                 // winners listed in this frame
  __shared__ uint16_t s_list[kSeqThreads];  // their columns in this CTA
  __shared__ __align__(8) uint64_t s_band_bar[2], s_cnt_bar[2];

  const uint32_t q = cluster.block_rank(), Q = cluster.num_blocks();
  const uint32_t t = threadIdx.x;
  const uint32_t warp = t >> 5, lane = t & 31u;
  const bool helper = t >= kSeqThreads;
  const uint32_t C = a.C, S = a.S, Cq = a.Cq;
  const uint32_t c0 = q * Cq;
  const uint32_t nc = C > c0 ? min(Cq, C - c0) : 0u;
  const uint32_t mw = Cq / 32u;  // mask words of this CTA
  const SeqLayout L(FORM, Q, Cq, S, a.band_max, C);
  uint32_t* s_bits = sm + L.bits;
  uint32_t* s_at = sm + L.at;
  uint32_t* s_org = sm + L.org;
  uint32_t* s_idx = sm + L.idx;
  uint16_t* s_pos = reinterpret_cast<uint16_t*>(sm + L.idx);
  float* s_perm = reinterpret_cast<float*>(sm + L.perm);
  float* s_boost = reinterpret_cast<float*>(sm + L.boost);
  uint32_t* s_band = sm + L.band;
  uint32_t* s_dirty = sm + L.dirty;
  const uint32_t hw = hist_words(S);
  const uint32_t cnt_words = Q * Cq / 2u;  // 32-bit words of one frame's counts
  const uint64_t g0 = (uint64_t)c0 * S;
  const bool fast = a.unit_boost != 0u;  // counts are the overlaps
  const bool global = a.inhibition == 0u;

  // Column ownership of the count.  A warp counts P columns side by side,
  // L32 = 32 / P lanes each (pools of a few synapses); its i-th own column is
  //   lc = ((i / P) * kSeqWarps + warp) * P + i % P,   i < own.
  const uint32_t lp = kWindow ? 0u : seq_pool_groups(S, Cq);  // log2 P
  const uint32_t P = 1u << lp, ll = 5u - lp, L32 = 1u << ll;
  const uint32_t passes = (Cq + (kSeqWarps << lp) - 1u) / (kSeqWarps << lp);
  const uint32_t own = passes << lp;  // at most 32 (Cq <= kSeqThreads)
  auto own_col = [&](uint32_t i) {
    return (((i >> lp) * kSeqWarps + warp) << lp) + (i & (P - 1u));
  };

  // ---- prologue: barriers, this CTA's state and input band -------------------
  if (t == 0) {
    s_n = 0u;
    s2[0] = s2[1] = 0u;
    mbar_init(&s_band_bar[0], kSeqHelpers);
    mbar_init(&s_band_bar[1], kSeqHelpers);
    mbar_init(&s_cnt_bar[0], 1);
    mbar_init(&s_cnt_bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  for (uint32_t i = t; i < nc; i += kAll) s_boost[i] = __ldg(a.boost + c0 + i);
  for (uint32_t i = t; i < mw; i += kAll) s_dirty[i] = 0u;
  for (uint32_t i = t; i < 3u * hw; i += kAll) sm[L.hist + i] = 0u;
  for (uint32_t i = t; i < 3u * mw; i += kAll) sm[L.mask + i] = 0u;
  for (uint32_t i = t; i < 2u * cnt_words; i += kAll) sm[L.cnt + i] = 0u;
  // band words no copy writes (rows past the frame, row padding) are read
  // under empty bitmap bits only; they are set once all the same
  for (uint32_t i = t; i < 2u * a.band_max; i += kAll) s_band[i] = 0u;
  if (FORM == kSeqPools) {
    const uint32_t nCS = nc * S;
    if ((S & 3u) == 0u) {
      const uint4* gi = reinterpret_cast<const uint4*>(a.idx + g0);
      const uint4* gp = reinterpret_cast<const uint4*>(a.perm + g0);
      for (uint32_t i = t; i < nCS / 4u; i += kAll) {
        reinterpret_cast<uint4*>(s_idx)[i] = __ldg(gi + i);
        reinterpret_cast<uint4*>(s_perm)[i] = gp[i];
      }
    } else {
      for (uint32_t i = t; i < nCS; i += kAll) {
        s_idx[i] = __ldg(a.idx + g0 + i);
        s_perm[i] = a.perm[g0 + i];
      }
    }
  }
  __syncthreads();
  // exact quotient by the frame width: with m = ceil(2^32 / W) the estimate
  // floor(id m / 2^32) is the quotient or one more (id < 2^32, m W - 2^32 < W)
  const uint32_t inv_w = kWindow ? 0xffffffffu / a.win_w + 1u : 0u;
  auto row_of = [&](uint32_t id) {
    const uint32_t r = __umulhi(id, inv_w);
    return r * a.win_w > id ? r - 1u : r;
  };
  // position of synapse id in its column's box: (bitmap word << 5) | bit
  auto box_pos = [&](uint32_t id, uint32_t org) {
    const uint32_t d = id - (org >> 16) * a.win_w;
    const uint32_t r = row_of(d), jx = d - r * a.win_w - (org & 0xffffu);
    return ((4u * (r & 31u) + 2u * (r >> 5) + (jx >> 5)) << 5) | (jx & 31u);
  };
  // learning left pending by the previous call; the columns' boxes and bitmaps;
  // the smallest and largest value that the CTA's band must cover (input
  // indices; window forms: box rows)
  if (!helper) {
    uint32_t mn = 0xffffffffu, mx = 0u;
    for (uint32_t i = 0; i < own; ++i) {
      const uint32_t lc = own_col(i);
      if (lc >= nc) continue;
      const uint32_t c = c0 + lc;
      const bool pend = a.pend_mask && ((__ldg(a.pend_mask + (c >> 5)) >> (c & 31u)) & 1u);
      if (kWindow) {
        // kBatch synapses a lane at a time, loaded before the first is used (a
        // pool of up to 256 is read once)
        constexpr int kBatch = 8;
        const uint64_t e0 = g0 + (uint64_t)lc * S;
        uint32_t id[kBatch];
        float pm[kBatch];
        auto load_batch = [&](uint32_t s0) {
#pragma unroll
          for (int j = 0; j < kBatch; ++j) {
            const uint32_t s = min(s0 + 32u * j, S - 1u);
            id[j] = __ldg(a.idx + e0 + s);
            pm[j] = a.perm[e0 + s];
          }
        };
        uint32_t x0 = 0xffffffffu, y0 = 0xffffffffu;
        for (uint32_t s0 = lane; s0 < S; s0 += 32u * kBatch) {
          load_batch(s0);
#pragma unroll
          for (int j = 0; j < kBatch; ++j) {
            const uint32_t y = row_of(id[j]);
            x0 = min(x0, id[j] - y * a.win_w);
            y0 = min(y0, y);
          }
        }
        x0 = __reduce_min_sync(kFull, x0);
        y0 = __reduce_min_sync(kFull, y0);
        const uint32_t org = (y0 << 16) | x0;
        if (lane == 0u) s_org[lc] = org;
        mn = min(mn, y0);
        mx = max(mx, y0 + 63u);
        uint32_t* wb = s_bits + lc * kBoxWords;
        reinterpret_cast<uint4*>(wb)[lane] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        for (uint32_t s0 = lane; s0 < S; s0 += 32u * kBatch) {
          if (S > 32u * kBatch) load_batch(s0);
#pragma unroll
          for (int j = 0; j < kBatch; ++j) {
            const uint32_t s = s0 + 32u * j;
            if (s < S) {
              const uint32_t pos = box_pos(id[j], org);
              float p = pm[j];
              if (pend) p = learn_one(p, dev::input_bit(a.pend_x, id[j]), a.inc, a.dec);
              if (kPermSmem) {
                s_pos[lc * S + s] = (uint16_t)pos;
                s_perm[lc * S + s] = p;
              } else if (pend) {
                a.perm[e0 + s] = p;
              }
              if (p >= a.thr) atomicOr(wb + (pos >> 5), 1u << (pos & 31u));
            }
          }
        }
      } else {
        const uint32_t* row = s_idx + lc * S;
        for (uint32_t s = lane; s < S; s += 32u) {
          const uint32_t id = row[s];
          mn = min(mn, id);
          mx = max(mx, id);
          if (pend)
            s_perm[lc * S + s] =
                learn_one(s_perm[lc * S + s], dev::input_bit(a.pend_x, id), a.inc, a.dec);
        }
      }
      if (pend && kPermSmem && lane == 0u) atomicOr(s_dirty + (lc >> 5), 1u << (lc & 31u));
    }
    mn = __reduce_min_sync(kFull, mn);
    mx = __reduce_max_sync(kFull, mx);
    if (lane == 0u) {
      sh[warp] = mn;
      sh[kSeqWarps + warp] = mx;
    }
  }
  __syncthreads();
  // the band: brows rows of blen words from word w_lo of the frame, `pitch` apart
  uint32_t w_lo = 0u, brows = 0u, blen = 1u, pitch = 1u, y_lo = 0u;
  {
    uint32_t m0 = 0xffffffffu, m1 = 0u;
    for (uint32_t w = 0; w < kSeqWarps; ++w) {
      m0 = min(m0, sh[w]);
      m1 = max(m1, sh[kSeqWarps + w]);
    }
    if (m0 <= m1 && kWindow) {  // else a CTA without columns
      y_lo = m0;
      w_lo = m0 * a.wpr;
      brows = min(m1 + 1u, a.n_words / a.wpr) - m0;
      blen = a.wpr;
      pitch = a.wpr | 1u;
    } else if (m0 <= m1) {
      w_lo = m0 >> 5;
      brows = 1u;
      blen = (m1 >> 5) + 1u - w_lo;
    }
  }
  if (helper) {
    copy_band(s_band, a.frames + w_lo, brows, blen, pitch, &s_band_bar[0]);
  } else if (kWindow) {
    for (uint32_t lc = t; lc < nc; lc += kSeqThreads) {
      const uint32_t org = s_org[lc];
      s_at[lc] = ((((org >> 16) - y_lo) * pitch + ((org & 0xffffu) >> 5)) << 5) | (org & 31u);
    }
  }
  // barriers initialized, counts cleared and bitmaps built in every CTA
  // before anyone sends
  cluster.sync();

  bool ok = true;  // this thread's waits so far
  uint32_t f = 0;
  if (helper) {
    for (; f < a.n_frames; ++f) {
      const uint32_t par = f & 1u;
      if (__syncthreads_or(0)) {  // B1: frame f counted, frame f - 1 done with
        ok = false;
        if (fast) break;
      }
      const uint32_t h = t - kSeqThreads;
      if (fast && Q > 1u && h == 0u) {
        mbar_expect(&s_cnt_bar[par], (Q - 1u) * Cq * 2u);
        s2[1] = f + 1u;
      }
      if (f + 1u < a.n_frames)
        copy_band(s_band + (par ^ 1u) * a.band_max, a.frames + (uint64_t)(f + 1u) * a.stride + w_lo,
                  brows, blen, pitch, &s_band_bar[par ^ 1u]);
      if (!fast) cluster.sync();  // every CTA's overlaps of frame f are published
      // the masks of frame f - 1; the mask of frame f + 1 and the histogram of
      // frame f + 2 cleared (their last readers passed B1)
      const uint32_t* pm = sm + L.mask + ((f + 2u) % 3u) * mw;
      uint32_t* zm = sm + L.mask + ((f + 1u) % 3u) * mw;
      for (uint32_t i = h; i < mw; i += kSeqHelpers) {
        if (f > 0u && a.masks_out && c0 / 32u + i < a.mask_words)
          a.masks_out[(uint64_t)(f - 1u) * a.mask_words + c0 / 32u + i] = pm[i];
        zm[i] = 0u;
      }
      if (fast && global) {
        uint32_t* zh = sm + L.hist + ((f + 2u) % 3u) * hw;
        for (uint32_t i = h; i < hw; i += kSeqHelpers) zh[i] = 0u;
      }
      if (a.ov_all) {
        const uint16_t* cnt = reinterpret_cast<const uint16_t*>(sm + L.cnt + par * cnt_words) + c0;
        const float* ov = reinterpret_cast<const float*>(sm + L.ov) + par * Cq;
        for (uint32_t i = h; i < nc; i += kSeqHelpers)
          a.ov_all[(uint64_t)f * C + c0 + i] = fast ? __uint2float_rn((uint32_t)cnt[i]) : ov[i];
      }
    }
  } else {
    // a warp's columns' bitmaps and band positions stay in registers when it
    // has few columns
    const bool reg_bits = kWindow && passes <= (uint32_t)kSeqCols;
    const uint32_t row32 = 32u * pitch;
    uint4 bm[kSeqCols];
    uint32_t off[kSeqCols], shf[kSeqCols];
    // column j past p0 of this warp (a valid one: results past nc are dropped)
    auto col_at = [&](uint32_t p0, int j) {
      return min((p0 + (uint32_t)j) * kSeqWarps + warp, nc - 1u);
    };
    auto load_bits = [&](uint32_t lc) {
      return reinterpret_cast<const uint4*>(s_bits + lc * kBoxWords)[lane];
    };
    if (reg_bits && nc) {
#pragma unroll
      for (int j = 0; j < kSeqCols; ++j) {
        const uint32_t lc = col_at(0u, j), at = s_at[lc];
        bm[j] = load_bits(lc);
        off[j] = (at >> 5) + lane * pitch;
        shf[j] = at & 31u;
      }
    }
    // what does not change from frame to frame: the CTA this warp sends to, and
    // in local inhibition the lane's column and its clipped window
    uint32_t peer_cnt = 0u, peer_bar = 0u;
    if (Q > 1u && warp < Q) {
      peer_cnt = peer_addr(smem_u32(reinterpret_cast<uint16_t*>(sm + L.cnt) + c0), warp);
      peer_bar = peer_addr(smem_u32(&s_cnt_bar[0]), warp);
    }
    uint32_t lg = 5u;  // log2 of the lanes that share a column
    for (uint32_t n_own = 1u; n_own < own; n_own <<= 1) --lg;
    const uint32_t loc_i = lane >> lg, loc_g = lane & ((1u << lg) - 1u), loc_lc = own_col(loc_i);
    const bool loc_ok = !global && loc_i < own && loc_lc < nc;
    uint32_t loc_x = 0u, loc_y = 0u;
    if (loc_ok) {
      loc_y = (c0 + loc_lc) / a.gw;
      loc_x = c0 + loc_lc - loc_y * a.gw;
    }
    const uint32_t parts2 = (S + 63u) / 64u;
    const float inv_parts2 = 1.0f / (float)parts2;
    uint32_t slot = 0u;  // f % 3
    for (; f < a.n_frames; ++f, slot = slot == 2u ? 0u : slot + 1u) {
      const uint32_t par = f & 1u, phase = (f >> 1) & 1u;
      const uint32_t* band = s_band + par * a.band_max;
      uint32_t* s_cnt32 = sm + L.cnt + par * cnt_words;
      uint16_t* s_cnt = reinterpret_cast<uint16_t*>(s_cnt32);  // [Q * Cq], column order
      uint32_t* hist = sm + L.hist + slot * hw;
      uint32_t* smask_f = sm + L.mask + slot * mw;
      float* ov_pub = reinterpret_cast<float*>(sm + L.ov) + par * Cq;
      if (ok) ok = mbar_wait<false, ONCE>(&s_band_bar[par], phase, a.wait_ns);

      // ---- Alg. 1 for this warp's columns ---------------------------------------
      // every load of a step is issued before its first use: no branch
      // separates the columns a warp counts side by side
      uint32_t top = 0u;  // largest count seen by this thread
      auto publish = [&](uint32_t lc, uint32_t raw) {
        const uint32_t v = raw >= a.min_overlap ? raw : 0u;
        if (!fast) {
          ov_pub[lc] = dev::boosted(raw, a.min_overlap, s_boost[lc]);
          return;
        }
        s_cnt[c0 + lc] = (uint16_t)v;
        if (Q == 1u && global && v != 0u) {
          atomicAdd(hist + v, 1u);
          top = max(top, v);
        }
      };
      auto count_window = [&](uint32_t p0) {
        uint32_t n[kSeqCols], a0[kSeqCols][3], a1[kSeqCols][3];
        if (!reg_bits) {
#pragma unroll
          for (int j = 0; j < kSeqCols; ++j) {
            const uint32_t lc = col_at(p0, j), at = s_at[lc];
            bm[j] = load_bits(lc);
            off[j] = (at >> 5) + lane * pitch;
            shf[j] = at & 31u;
          }
        }
#pragma unroll
        for (int j = 0; j < kSeqCols; ++j) {
          const uint32_t* p = band + off[j];
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            a0[j][i] = p[i];
            a1[j][i] = p[row32 + i];
          }
        }
#pragma unroll
        for (int j = 0; j < kSeqCols; ++j)
          n[j] = __popc(__funnelshift_r(a0[j][0], a0[j][1], shf[j]) & bm[j].x) +
                 __popc(__funnelshift_r(a0[j][1], a0[j][2], shf[j]) & bm[j].y) +
                 __popc(__funnelshift_r(a1[j][0], a1[j][1], shf[j]) & bm[j].z) +
                 __popc(__funnelshift_r(a1[j][1], a1[j][2], shf[j]) & bm[j].w);
        uint32_t mine = 0u;
#pragma unroll
        for (int j = 0; j < kSeqCols; ++j) {
          const uint32_t r = __reduce_add_sync(kFull, n[j]);
          mine = lane == (uint32_t)j ? r : mine;
        }
        const uint32_t lc = (p0 + lane) * kSeqWarps + warp;
        if (lane < (uint32_t)kSeqCols && lc < nc) publish(lc, mine);
      };
      // U groups of P columns side by side
      auto count_pools = [&](uint32_t p0, auto u) {
        constexpr int U = decltype(u)::value;
        uint32_t n[U], row[U];
        const uint32_t sub = lane >> ll, sl = lane & (L32 - 1u);
#pragma unroll
        for (int j = 0; j < U; ++j) {
          n[j] = 0u;
          row[j] = min((((p0 + j) * kSeqWarps + warp) << lp) + sub, nc - 1u) * S;
        }
        auto bit = [&](uint32_t w, uint32_t id, float p) {
          return p >= a.thr ? (w >> (id & 31u)) & 1u : 0u;
        };
        if ((S & 3u) == 0u) {
          for (uint32_t v = sl; v < (S >> 2); v += L32) {
            uint4 id[U], w[U];
            float4 pm[U];
#pragma unroll
            for (int j = 0; j < U; ++j) {
              id[j] = reinterpret_cast<const uint4*>(s_idx + row[j])[v];
              pm[j] = reinterpret_cast<const float4*>(s_perm + row[j])[v];
            }
#pragma unroll
            for (int j = 0; j < U; ++j)
              w[j] = make_uint4(band[(id[j].x >> 5) - w_lo], band[(id[j].y >> 5) - w_lo],
                                band[(id[j].z >> 5) - w_lo], band[(id[j].w >> 5) - w_lo]);
#pragma unroll
            for (int j = 0; j < U; ++j)
              n[j] += bit(w[j].x, id[j].x, pm[j].x) + bit(w[j].y, id[j].y, pm[j].y) +
                      bit(w[j].z, id[j].z, pm[j].z) + bit(w[j].w, id[j].w, pm[j].w);
          }
        } else {
          for (uint32_t s = sl; s < S; s += L32) {
            uint32_t id[U], w[U];
            float pm[U];
#pragma unroll
            for (int j = 0; j < U; ++j) {
              id[j] = s_idx[row[j] + s];
              pm[j] = s_perm[row[j] + s];
            }
#pragma unroll
            for (int j = 0; j < U; ++j) w[j] = band[(id[j] >> 5) - w_lo];
#pragma unroll
            for (int j = 0; j < U; ++j) n[j] += bit(w[j], id[j], pm[j]);
          }
        }
        if (P == 1u) {
          uint32_t mine = 0u;
#pragma unroll
          for (int j = 0; j < U; ++j) {
            const uint32_t r = __reduce_add_sync(kFull, n[j]);
            mine = lane == (uint32_t)j ? r : mine;
          }
          const uint32_t lc = (p0 + lane) * kSeqWarps + warp;
          if (lane < (uint32_t)U && lc < nc) publish(lc, mine);
        } else {
          for (uint32_t o = 1u; o < L32; o <<= 1) {
#pragma unroll
            for (int j = 0; j < U; ++j) n[j] += __shfl_xor_sync(kFull, n[j], o);
          }
          // lane j of a column's lanes publishes the j-th group's count
          uint32_t mine = n[0];
#pragma unroll
          for (int j = 1; j < U; ++j) mine = sl == (uint32_t)j ? n[j] : mine;
          const uint32_t lc = (((p0 + sl) * kSeqWarps + warp) << lp) + sub;
          if (sl < (uint32_t)U && lc < nc) publish(lc, mine);
        }
      };
      if (nc) {
        if (kWindow) {
          for (uint32_t p0 = 0; p0 < passes; p0 += kSeqCols) count_window(p0);
        } else {
          uint32_t p0 = 0;
          for (; p0 + 3u <= passes; p0 += 4u) count_pools(p0, IntC<4>{});
          for (; p0 < passes; p0 += 2u) count_pools(p0, IntC<2>{});
        }
      }
      if (fast && global && Q == 1u) {
        top = __reduce_max_sync(kFull, top);
        if (lane == 0u && top) atomicMax(hist, top);
      }
      // B1: every warp's counts are in place
      if (__syncthreads_or(!ok ? 1 : 0)) {
        ok = false;
        if (fast) break;  // else the cluster barriers below are still to be met
      }

      if (fast) {
        // ---- all counts to every CTA --------------------------------------------
        if (Q > 1u) {
          if (warp < Q && warp != q) {
            const uint32_t dst = peer_cnt + par * cnt_words * 4u, bar = peer_bar + par * 8u;
            for (uint32_t u = lane; u < Cq / 8u; u += 32u)
              send16(dst + u * 16u, reinterpret_cast<const uint4*>(s_cnt + c0)[u], bar);
          }
          if (ok) ok = mbar_wait<true, ONCE>(&s_cnt_bar[par], phase, a.wait_ns);
          if (!ok) atomicSub(&s_n, 1u << 20);  // read as below 0: nothing is learnt from it
        }
        if (global) {
          if (Q > 1u) {
            for (uint32_t i = t; i < cnt_words; i += kSeqThreads) {
              const uint32_t w = s_cnt32[i], v0 = w & 0xffffu, v1 = w >> 16;
              if (v0) atomicAdd(hist + v0, 1u);
              if (v1) atomicAdd(hist + v1, 1u);
              top = max(top, max(v0, v1));
            }
            top = __reduce_max_sync(kFull, top);
            if (lane == 0u && top) atomicMax(hist, top);
            compute_sync();
          }
          // warp m decides the CTA's columns 32m .. 32m + 31
          if (warp < mw) {
            // T = the k-th largest count (0 when at most k columns count);
            // `need` of the `ties` columns at it win, in column order
            uint32_t T, need, ties;
            const uint32_t v = s_cnt[c0 + 32u * warp + lane];
            dev::warp_kth_count(hist, a.k, T, need, ties);
            const bool tie = T != 0u && v == T;
            bool win = T != 0xffffffffu && v > T;
            const uint32_t tw = __ballot_sync(kFull, tie);
            if (tw) {
              uint32_t before = 0u;  // tied columns below this warp's
              if (ties > need) {
                const uint4* cv = reinterpret_cast<const uint4*>(s_cnt);
                const uint32_t lim = (c0 + 32u * warp) / 8u, TT = T | (T << 16);
                auto eq2 = [&](uint32_t w) {
                  const uint32_t x = w ^ TT;
                  return ((x & 0xffffu) == 0u ? 1u : 0u) + ((x >> 16) == 0u ? 1u : 0u);
                };
#pragma unroll 4
                for (uint32_t i = lane; i < lim; i += 32u) {
                  const uint4 w = cv[i];
                  before += eq2(w.x) + eq2(w.y) + eq2(w.z) + eq2(w.w);
                }
                before = __reduce_add_sync(kFull, before);
              }
              win = win || (tie && before + __popc(tw & ((1u << lane) - 1u)) < need);
            }
            const uint32_t w = __ballot_sync(kFull, win);
            if (lane == 0u) smask_f[warp] = w;
          }
        } else {
          // local: G lanes share a column, each ranking it against every G-th
          // row of its clipped (2r + 1)^2 neighbourhood.  A neighbour beats it
          // with a higher count, or with an equal one and a lower index: rows
          // above and columns to the left win ties
          const uint32_t lc = loc_lc, c = c0 + lc, G = 1u << lg, g = loc_g;
          const uint32_t v = loc_ok ? s_cnt[c] : 0u;
          uint32_t beaten = 0u;
          if (v != 0u && a.k != 0u) {
            const uint32_t x = loc_x, y = loc_y, r = a.radius;
            const uint32_t x0 = x >= r ? x - r : 0u, x1 = min(a.gw - 1u, x + r);
            const uint32_t y0 = y >= r ? y - r : 0u, y1 = min(a.gh - 1u, y + r);
            // two columns a word: (count | 0x8000) - limit keeps its top bit
            // where the count reaches the limit (counts are below 0x8000)
            uint32_t two = 0u;  // a 16-bit sum per half
            for (uint32_t jj = y0 + g; jj <= y1; jj += G) {
              if (jj == y) {
                for (uint32_t ii = x0; ii <= x1; ++ii)
                  beaten += s_cnt[jj * a.gw + ii] >= (ii < x ? v : v + 1u) ? 1u : 0u;
                continue;
              }
              const uint32_t lim = jj < y ? v : v + 1u, lim2 = lim | (lim << 16);
              const uint32_t i0 = jj * a.gw + x0, i1 = jj * a.gw + x1;
              const uint32_t w0 = i0 >> 1, w1 = i1 >> 1;
              auto reach = [&](uint32_t w) {
                return (((s_cnt32[w] | 0x80008000u) - lim2) >> 15) & 0x00010001u;
              };
              const uint32_t first = (i0 & 1u) ? 0x00010000u : 0x00010001u;
              const uint32_t final = (i1 & 1u) ? 0x00010001u : 0x00000001u;
              if (w0 == w1) {
                two += reach(w0) & first & final;
              } else {
                two += (reach(w0) & first) + (reach(w1) & final);
#pragma unroll 4
                for (uint32_t w = w0 + 1u; w < w1; ++w) two += reach(w);
              }
            }
            beaten += (two & 0xffffu) + (two >> 16);
          }
          for (uint32_t o = 1u; o < G; o <<= 1) beaten += __shfl_xor_sync(kFull, beaten, o);
          if (g == 0u && v != 0u && beaten < a.k)
            atomicOr(smask_f + (lc >> 5), 1u << (lc & 31u));
          compute_sync();
        }
      } else {
        // ---- non-unit boosts: gather all overlaps through DSMEM -------------------
        cluster.sync();  // every CTA's overlaps of frame f are published
        uint32_t* s_all = sm + L.all;
        uint32_t* s_smask = sm + L.smask;
        uint32_t nz = 0;
#pragma unroll 4
        for (uint32_t i = t; i < C; i += kSeqThreads) {
          const uint32_t owner = i / Cq;
          const float* src = cluster.map_shared_rank(ov_pub, owner);
          const uint32_t v = __float_as_uint(src[i - owner * Cq]);
          s_all[i] = v;
          nz += v != 0u;
        }
        for (uint32_t i = t; i < a.mask_words; i += kSeqThreads) s_smask[i] = 0u;
        if (global) {
          uint32_t e0, e1, nz_tot, z, Tb, nd;
          dev::block_scan2<kSeqWarps>(nz, 0u, e0, e1, nz_tot, z, sh);
          dev::select_threshold<kSeqThreads>(s_all, C, a.k, nz_tot, nullptr, 0u, sm + L.shist, sh,
                                             s2, Tb, nd);
          dev::mark_global<kSeqThreads>(s_all, C, Tb, nd, s_smask, s_smask + a.mask_words, nullptr);
        } else {
          compute_sync();
          dev::mark_local<kSeqThreads>(s_all, 0u, C, a.gw, a.gh, a.radius, a.k, s_smask, nullptr,
                                       sh);
        }
        compute_sync();
        if (warp < mw && lane == 0u)
          smask_f[warp] = c0 / 32u + warp < a.mask_words ? s_smask[c0 / 32u + warp] : 0u;
      }

      // ---- the winners' list (in no order), duty cycles ---------------------------
      if (warp < mw) {
        __syncwarp();
        const uint32_t w = smask_f[warp], lc = 32u * warp + lane;
        if (a.duty && lc < nc) {
          const float d = a.duty[c0 + lc], act = (w >> lane) & 1u ? 1.0f : 0.0f;
          a.duty[c0 + lc] = __fadd_rn(d, __fdiv_rn(__fsub_rn(act, d), a.duty_period));
        }
        if (a.learn && w != 0u) {
          uint32_t at = 0u;
          if (lane == 0u) at = atomicAdd(&s_n, (uint32_t)__popc(w));
          at = __shfl_sync(kFull, at, 0) + __popc(w & ((1u << lane) - 1u));
          if ((w >> lane) & 1u) s_list[at & (kSeqThreads - 1u)] = (uint16_t)lc;
        }
      }
      if (!a.learn) continue;
      compute_sync();
      // ---- learning: the listed winners' synapses, 32 J of one column a unit,
      // units dealt to the warps; a unit's loads are issued before the first is
      // used.  Few winners: small units, so that their chains are short
      const uint32_t n_win = (uint32_t)max((int)s_n, 0);
      auto learn = [&](auto jc, uint32_t parts, float inv_parts) {
        constexpr int J = decltype(jc)::value;
        const uint32_t units = n_win * parts;
        for (uint32_t u = warp; u < units; u += kSeqWarps) {
          // u / parts: both below 2^16, half a unit from the next quotient
          const uint32_t i = __float2uint_rz(((float)u + 0.5f) * inv_parts);
          const uint32_t s0 = (u - i * parts) * 32u * J + lane;
          const uint32_t lc = s_list[i];
          uint32_t* wb = s_bits + lc * kBoxWords;
          uint32_t at = 0u, org = 0u;
          if (kWindow) {
            at = s_at[lc];
            org = s_org[lc];
          }
          const uint64_t e0 = g0 + (uint64_t)lc * S;
          uint32_t id[J], bit[J];
          float p[J];
#pragma unroll
          for (int j = 0; j < J; ++j) {
            const uint32_t s = min(s0 + 32u * j, S - 1u);
            id[j] = FORM == kSeqPools ? s_idx[lc * S + s]
                                      : (kPermSmem ? (uint32_t)s_pos[lc * S + s]
                                                   : __ldg(a.idx + e0 + s));
            p[j] = kPermSmem ? s_perm[lc * S + s] : __ldcg(a.perm + e0 + s);
          }
#pragma unroll
          for (int j = 0; j < J; ++j) {
            if (FORM == kSeqPools) {
              bit[j] = (band[(id[j] >> 5) - w_lo] >> (id[j] & 31u)) & 1u;
            } else {
              if (!kPermSmem) id[j] = box_pos(id[j], org);
              const uint32_t r = (id[j] >> 7) + ((id[j] & 64u) >> 1);
              const uint32_t x = (at & 31u) + (id[j] & 63u);  // word parity and bit: the pixel
              bit[j] = (band[(at >> 5) + r * pitch + (x >> 5)] >> (x & 31u)) & 1u;
            }
          }
#pragma unroll
          for (int j = 0; j < J; ++j) {
            const uint32_t s = s0 + 32u * j;
            const float np = learn_one(p[j], bit[j], a.inc, a.dec);
            if (s < S) {
              if (kPermSmem)
                s_perm[lc * S + s] = np;
              else
                __stcg(a.perm + e0 + s, np);
              if (kWindow && (np >= a.thr) != (p[j] >= a.thr))
                atomicXor(wb + (id[j] >> 5), 1u << (id[j] & 31u));
            }
          }
          if (kPermSmem && lane == 0u && s0 == 0u) atomicOr(s_dirty + (lc >> 5), 1u << (lc & 31u));
        }
      };
      if (parts2 == 1u || n_win * S <= 2048u) {
        learn(IntC<2>{}, parts2, inv_parts2);
      } else {
        constexpr int J = kPermSmem ? 8 : 4;  // the box positions of 8 would spill
        const uint32_t parts = (S + 32u * J - 1u) / (32u * J);
        learn(IntC<J>{}, parts, 1.0f / (float)parts);
      }
      compute_sync();  // the next count reads what other warps learnt
      if (t == 0u) s_n = 0u;
      if (reg_bits && nc) {
#pragma unroll
        for (int j = 0; j < kSeqCols; ++j) {
          const uint32_t lc = col_at(0u, j);
          if ((smask_f[lc >> 5] >> (lc & 31u)) & 1u) bm[j] = load_bits(lc);
        }
      }
    }
  }
  if (!ok) {
    s2[0] = 1u;
    if (a.err) atomicExch(a.err, 1u);
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  // ---- the last frame's outputs, and the permanence rows that changed ------------
  const uint32_t last = a.n_frames - 1u;
  const uint32_t* lmask = sm + L.mask + (last % 3u) * mw;
  for (uint32_t i = t; i < mw; i += kAll) {
    const uint32_t w = c0 / 32u + i;
    if (w < a.mask_words) {
      if (a.masks_out) a.masks_out[(uint64_t)last * a.mask_words + w] = lmask[i];
      a.mask_last[w] = lmask[i];
    }
  }
  {
    const uint16_t* cnt = reinterpret_cast<const uint16_t*>(sm + L.cnt + (last & 1u) * cnt_words);
    const float* ov = reinterpret_cast<const float*>(sm + L.ov) + (last & 1u) * Cq;
    for (uint32_t i = t; i < nc; i += kAll)
      a.ov_out[c0 + i] = fast ? __uint2float_rn((uint32_t)cnt[c0 + i]) : ov[i];
  }
  if (kPermSmem) {
    for (uint32_t lc = warp; lc < nc; lc += kAll / 32u) {
      if (!((s_dirty[lc >> 5] >> (lc & 31u)) & 1u)) continue;
      float* gp = a.perm + g0 + (uint64_t)lc * S;
      for (uint32_t s = lane; s < S; s += 32) gp[s] = s_perm[lc * S + s];
    }
  }
  cluster.sync();  // every CTA's mask of the last frame is final, and its last counts are sent
  if (warp == kSeqWarps && s2[0] && fast) drain_counts(smem_u32(s_cnt_bar), smem_u32(&s2[1]), Cq * 2u);
  if (q == 0u && warp == 0u) {
    // ascending list of the last frame's winners, 32 mask words at a time
    uint32_t total = 0u;
    for (uint32_t b = 0; b < a.mask_words; b += 32u) {
      const uint32_t w = b + lane, owner = w / mw;
      uint32_t m = 0u;
      if (w < a.mask_words) m = cluster.map_shared_rank(lmask, owner)[w - owner * mw];
      const uint32_t n = __popc(m);
      uint32_t inc = n;
#pragma unroll
      for (uint32_t o = 1; o < 32u; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += y;
      }
      uint32_t pos = total + inc - n;
      for (; m != 0u; m &= m - 1u) a.result[1 + pos++] = w * 32u + (uint32_t)(__ffs(m) - 1);
      total += __shfl_sync(kFull, inc, 31);
    }
    if (lane == 0u) a.result[0] = total;
  }
  // no CTA may exit while another can still read or write its shared memory
  cluster.sync();
}

// One warp per column.
__global__ void __launch_bounds__(256) sp_pool_scan_kernel(const uint32_t* idx, uint32_t C,
                                                           uint32_t S, uint32_t W, uint32_t* out) {
  const uint32_t c = blockIdx.x * 8u + (threadIdx.x >> 5), lane = threadIdx.x & 31u;
  if (c >= C) return;
  const uint32_t* p = idx + (uint64_t)c * S;
  const bool box = W % 32u == 0u && S <= 4096u;
  uint32_t lo = 0xffffffffu, hi = 0u, x0 = 0xffffffffu, x1 = 0u;
  bool ascending = true;
  for (uint32_t s = lane; s < S; s += 32u) {
    const uint32_t id = p[s];
    lo = min(lo, id);
    hi = max(hi, id);
    if (s + 1u < S) ascending = ascending && p[s + 1u] > id;
    if (box) {
      const uint32_t x = id % W;
      x0 = min(x0, x);
      x1 = max(x1, x);
    }
  }
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
  x0 = __reduce_min_sync(kFull, x0);
  x1 = __reduce_max_sync(kFull, x1);
  ascending = __all_sync(kFull, ascending);
  if (lane == 0u) {
    const uint32_t y0 = lo / W, y1 = hi / W;
    const bool fits = box && ascending && x1 - x0 < 64u && y1 - y0 < 64u && x0 <= 0xffffu &&
                      y0 <= 0xffffu;
    out[c] = lo;
    out[C + c] = hi;
    out[2u * C + c] = fits ? y0 : 0xffffffffu;
  }
}

using SeqKernel = void (*)(const SeqArgs);

template <bool ONCE>
SeqKernel seq_kernel(uint32_t form) {
  return form == kSeqPools ? sp_seq_cluster_kernel<kSeqPools, ONCE>
                           : (form == kSeqWindow ? sp_seq_cluster_kernel<kSeqWindow, ONCE>
                                                 : sp_seq_cluster_kernel<kSeqWindowL2, ONCE>);
}

}  // namespace

cudaError_t launch_pool_scan(const uint32_t* idx, uint32_t C, uint32_t S, uint32_t W,
                             uint32_t* out, cudaStream_t stream) {
  sp_pool_scan_kernel<<<(C + 7u) / 8u, 256, 0, stream>>>(idx, C, S, W, out);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

size_t seq_smem_bytes(uint32_t form, uint32_t Q, uint32_t C, uint32_t S, uint32_t Cq,
                      uint32_t band_max) {
  return (size_t)SeqLayout(form, Q, Cq, S, band_max, C).total * 4u;
}

cudaError_t seq_kernel_init(uint32_t form, size_t smem_bytes) {
  for (const SeqKernel k : {seq_kernel<false>(form), seq_kernel<true>(form)}) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t seq_max_active_clusters(uint32_t form, uint32_t Q, size_t smem_bytes, int* out) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(Q, 1, 1);
  cfg.blockDim = dim3(kSeqThreads + kSeqHelpers, 1, 1);
  cfg.dynamicSmemBytes = smem_bytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = Q;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaOccupancyMaxActiveClusters(out, seq_kernel<false>(form), &cfg);
}

cudaError_t launch_seq(const SeqArgs& a, uint32_t form, uint32_t Q, size_t smem_bytes,
                       cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(Q, 1, 1);
  cfg.blockDim = dim3(kSeqThreads + kSeqHelpers, 1, 1);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = Q;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, a.wait_ns < 1000u ? seq_kernel<true>(form) : seq_kernel<false>(form), a);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return e;
}

}  // namespace sp

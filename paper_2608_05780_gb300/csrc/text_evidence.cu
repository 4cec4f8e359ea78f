// Text-row evidence (Sec. 3.2, "Evidence Decomposition"):
//   tok[h, m]   = sum_{text rows i} exp(s_im - LSE_i),  s = scale q_i k_m (Eq. 8),
//   frame[h, t] = sum_{m in frame t} tok[h, m],
// with LSE the probe's saved row normaliser (Eq. 11). Text rows attend to
// every visual key of their video (dense causal), so every (text row, visual
// key) pair enters; after a probe with per-row block masks only the pairs whose
// bit is set do (their LSE entries are staged once per block of the unit's
// keys, -inf where the row does not keep the block). The probabilities are
// formed again from q, k and LSE: spilling the text rows' logits from the probe
// and reading them back (940 MB each way on 65,664 tokens) cost more.
//
// Work unit: 128 visual keys of a video, one KV group, a part of its heads. A
// persistent grid (one CTA per SM) walks the units; every role runs on across
// unit borders on its own, so only a CTA's first unit pays the fill. A step is
// one head and one text tile (the video's text rows cut evenly into tiles of
// at most 128 rows, or 256 where some video of the call has more than 128):
//   warps 0-15  four groups of 128 threads, one thread per key (TMEM lane), each
//               with a TMEM buffer of its own (two groups at 256 columns); the
//               heads go round the groups, so that four (two) heads are in
//               flight. A thread adds exp2(s scale log2e - LSE log2e) over its head's
//               text rows and writes tok[h, key]; frame sums by shuffles (and
//               shared memory for N_v > 32)
//   warp 16     TMA: the unit's key tile K_g into a 2-deep ring, Q_h of each
//               text tile into a ring of the head's MMA warp (128B swizzle)
//   warps 17/18 MMA, every other head each: S^T = K_g Q_h^T (tcgen05, bf16 in,
//               fp32 in TMEM; M = 128 keys, N = the tile's text rows). Issuing
//               blocks while the tensor pipe is busy, so one warp's waits fall
//               into the other's MMAs
//   warp 19     the steps' LSEs, negated in log2 units, to shared memory (two
//               steps ahead); it arrives on the same barrier as the step's MMA
// What bounds it: per (text row, key) pair one ex2 on the XU pipe (32 per clock
// and SM) and 2 d tensor flops. A tcgen05.mma with A and B in shared memory
// takes at least 64 clocks whatever its N (measured: 72 at N = 32, 69 at N =
// 128), so one wide text tile per head is cheaper than several narrow ones;
// the waits of a step (about 150 clocks each even when they are over) are
// hidden only behind other heads' sums, hence the groups.
// A pair of columns is one packed fma, two ex2 and one packed add. The evidence
// call that forms the sums (this kernel and the maps, 28 heads in 4 groups, d =
// 128) took 419 us on the 8-video batch, 116 on 65,664 tokens, 37 on 16,512 and 19
// on 4,160 with one CTA per (128 keys, KV group), one thread per key and two CTAs
// per SM; with this kernel 351, 87, 31 and 16. The LSE warp needs two steps'
// loads in flight: with one, serialised by a branch, the kernel takes 6 to 40% more.
// Every (head, key) has one writer and a fixed summation order. Every wait is
// bounded; on timeout the CTA records EVISEL_ETIMEOUT and drains its copies
// and MMAs. The key warps never leave their loop early; after a timeout they
// only skip the work.
#include <cstdint>
#include <cuda_runtime.h>

#include "evisel_internal.h"
#include "sm103_ptx.cuh"

namespace evisel {
namespace {

constexpr int kRows = 128;                       // keys of a unit (TMEM lanes)
constexpr int kMaxText = 256;                    // text rows of a step
constexpr int kUnitTable = 64;                   // units of a CTA looked up before the roles start
constexpr int kMaxBlocks = 8;                    // mask blocks of a unit's keys (16 tokens at least)
constexpr int kGroups = 4;                       // groups of key threads: heads in flight
constexpr int kKeyWarps = kGroups * kRows / 32;
constexpr int kWarpProducer = kKeyWarps;
constexpr int kWarpMma = kKeyWarps + 1;
constexpr int kMmaWarps = 2;
constexpr int kWarpLse = kWarpMma + kMmaWarps;
constexpr int kThreads = 32 * (kWarpLse + 1);
constexpr int kTmemCols = 512;

template <int D>
struct TeCfg {
  static constexpr int KB = D / 64;
  static constexpr int BOX = kRows * 128;        // one TMA box: 128 rows x 64 columns
  static constexpr int K_BYTES = KB * BOX;
  static constexpr int KS = 2;                   // K ring stages
  static constexpr int QS = 4;                   // Q stages of 128 rows (2 of 256): half of them per MMA warp
  static constexpr int NB = 4;                   // S buffers (2 of them used at 256 columns)
  static constexpr int OFF_K = 0;
  static constexpr int OFF_Q = KS * K_BYTES;
  static constexpr int OFF_LSE = OFF_Q + QS * K_BYTES;              // per S buffer [blocks of the keys][its columns] fp32
  static constexpr int OFF_RED = OFF_LSE + kMaxBlocks * kTmemCols * 4;   // [kKeyWarps] fp32
  static constexpr int OFF_UNIT = OFF_RED + kKeyWarps * 4;          // [kUnitTable] Unit
  static constexpr int OFF_BAR = OFF_UNIT + kUnitTable * 48;
  static constexpr int B_KF = 0, B_KE = B_KF + KS, B_QF = B_KE + KS, B_QE = B_QF + QS, B_SF = B_QE + QS,
                       B_SE = B_SF + NB, B_DRAIN = B_SE + NB;
  static constexpr int N_BARS = B_DRAIN + kMmaWarps;
  static constexpr int OFF_MISC = OFF_BAR + N_BARS * 8;
  static constexpr int SMEM_BYTES = OFF_MISC + 16 + 1024;
  static_assert(SMEM_BYTES <= 232448, "shared memory budget");
};

__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  const bool ok = ptx::mbar_wait(bar, parity, abort_flag, kWaitTimeoutNs);
  return __all_sync(0xffffffffu, ok);
}

__device__ __forceinline__ void record_failure(volatile int* abort_flag, int* status) {
  *abort_flag = 1;
  atomicExch(status, kStatusTimeout);
}

// Heads [h0, h0 + nh) of KV group g against the keys [col0, col0 + 128)
// of a video, in nh heads x n_tt text tiles of tile_rows rows.
struct Unit {
  int col0, vis_start, n_vis, n_text, vis_off, frame_off;
  int g, h0, nh, n_tt, tile_rows, pad;
};

__device__ __forceinline__ Unit unit_of(const TextEvidenceLaunch& L, int u) {
  Unit x;
  const EvChunk ch = L.chunks[u % L.n_chunks];
  const int gi = u / L.n_chunks;                 // the units of one (group, part) are adjacent: they share Q
  x.g = gi / L.head_split;
  const int part = gi % L.head_split, gq = L.hq / L.hkv;
  const int lo = gq * part / L.head_split, hi = gq * (part + 1) / L.head_split;
  x.h0 = x.g * gq + lo;
  x.nh = hi - lo;
  const VideoInfo& vi = L.videos[ch.video];
  x.col0 = ch.col0;
  x.vis_start = vi.vis_start;
  x.n_vis = vi.n_vis;
  x.n_text = vi.n_text;
  x.vis_off = vi.vis_off;
  x.frame_off = vi.frame_off;
  x.n_tt = (x.n_text + L.text_cols - 1) / L.text_cols;
  x.pad = 0;
  x.tile_rows = x.n_tt > 0 ? ((x.n_text + x.n_tt - 1) / x.n_tt + 15) & ~15 : 0;   // at most text_cols
  return x;
}

// Sum of one (head, key) over the text rows that keep the key's block, from q
// and k in global memory. A dropped pair's -inf entry does not hide a NaN or
// +inf logit, so a masked sum that came out NaN is formed again here: rare and
// slow, where testing every pair took 13 us of 318 (24,576 tokens, 28 heads, 250
// text rows) and testing every step 7.
__device__ __noinline__ float kept_sum(const TextEvidenceLaunch& L, const Unit& x, int h, int key) {
  const int D = L.head_dim, blk = (x.col0 + key) / L.keep_block;
  const int64_t row0 = x.vis_start + x.n_vis;
  const uint32_t* words = L.keep + (static_cast<int64_t>(h) * L.keep_words + (blk >> 5)) * L.n_tok + row0;
  const uint4* k = reinterpret_cast<const uint4*>(
      static_cast<const uint16_t*>(L.k) + (static_cast<int64_t>(x.vis_start + x.col0 + key) * L.hkv + x.g) * D);
  float sum = 0.f;
  for (int r = 0; r < x.n_text && !isnan(sum); ++r) {
    if (!((__ldg(words + r) >> (blk & 31)) & 1u)) continue;
    const uint4* q = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(L.q) + ((row0 + r) * L.hq + h) * D);
    float s = 0.f;
    for (int c = 0; c < D / 8; ++c) {
      const uint4 a = __ldg(q + c), b = __ldg(k + c);
      const uint32_t av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        s = fmaf(__uint_as_float(av[i] << 16), __uint_as_float(bv[i] << 16), s);
        s = fmaf(__uint_as_float(av[i] & 0xffff0000u), __uint_as_float(bv[i] & 0xffff0000u), s);
      }
    }
    const float lse = __ldg(L.lse + static_cast<int64_t>(h) * L.n_tok + row0 + r);
    sum += ptx::ex2(fmaf(s, L.scale_log2, -1.4426950408889634f * lse));
  }
  return sum;
}

// kKeep: the probe ran with per-row block masks.
template <int D, bool kKeep>
__global__ void __launch_bounds__(kThreads, 1) text_evidence_kernel(const __grid_constant__ TextEvidenceLaunch L) {
  using C = TeCfg<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = ptx::smem_addr(smem);
  auto bar = [&](int i) { return sbase + C::OFF_BAR + 8u * i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_MISC + 4);
  float* lse_s = reinterpret_cast<float*>(smem + C::OFF_LSE);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_units = L.n_chunks * L.hkv * L.head_split;
  const int nb = kTmemCols / L.text_cols;          // S buffers = groups in use
  const int nblk = kKeep ? kRows / L.keep_block : 1;   // mask blocks of a unit's keys
  // The n-th Q tile of MMA warp w is in stage w spw + n % spw, phase n / spw:
  // every barrier has one waiter, which sees each of its phases (a parity wait
  // must never run two phases ahead).
  const int spw = nb / kMmaWarps;                  // Q stages per MMA warp
  const int q_block = L.text_cols * 128, q_bytes = C::KB * q_block;
  // S buffer b of the CTA's n-th head is n % nb; buffer_free waits until the
  // step before in it has been summed (every step of every role passes here once).
  uint32_t used = 0u, odd = 0u;                    // per buffer: any step yet, parity of their number
  auto buffer_free = [&](int b) {
    const bool free_ = !((used >> b) & 1u) || warp_wait(bar(C::B_SE + b), ((odd >> b) & 1u) ^ 1u, abort_flag);
    used |= 1u << b;
    odd ^= 1u << b;
    return free_;
  };

  // The CTA's units, looked up in parallel: two dependent global loads per unit
  // and role would cost more than a short unit's sums.
  Unit* table = reinterpret_cast<Unit*>(smem + C::OFF_UNIT);
  static_assert(sizeof(Unit) == 48 && C::OFF_UNIT % 16 == 0, "unit table");
  if (threadIdx.x >= 64 && threadIdx.x < 64 + kUnitTable) {
    const int i = threadIdx.x - 64, u = blockIdx.x + i * gridDim.x;
    if (u < n_units) table[i] = unit_of(L, u);
  }
  auto unit_at = [&](int u) -> Unit {
    const int i = (u - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x);
    return i < kUnitTable ? table[i] : unit_of(L, u);
  };
  if (threadIdx.x == 0) {
    for (int i = 0; i < C::N_BARS; ++i)
      ptx::mbar_init(bar(i), i >= C::B_SF && i < C::B_SF + C::NB   ? 2u     // the MMA's commit and the LSE warp
                             : i >= C::B_SE && i < C::B_SE + C::NB ? kRows / 32u   // the four warps of a group
                             : i >= C::B_KE && i < C::B_KE + C::KS ? static_cast<uint32_t>(kMmaWarps)
                                                                   : 1u);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc<kTmemCols>(ptx::smem_addr(tmem_slot));
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;

  if (warp == kWarpProducer) {
    const uint64_t pol_q = ptx::l2_policy_evict_last();   // the video's text Q is read by every key tile
    const uint64_t pol_k = ptx::l2_policy_evict_first();  // a key tile is read once per KV group and part
    uint32_t leader = 0;
    int nk = 0, nh = 0;                          // K tiles issued, heads so far
    int nq[kMmaWarps] = {};                      // Q tiles issued to each MMA warp
    for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x) {
      const Unit x = unit_at(u);
      if (x.n_tt == 0) continue;                 // a video without text rows: nothing to load
      const int ks = nk % C::KS;
      if (nk >= C::KS && !warp_wait(bar(C::B_KE + ks), ((nk - C::KS) / C::KS) & 1, abort_flag)) {
        ok = false;
        break;
      }
      if (ptx::elect_one(leader)) {
        ptx::mbar_arrive_expect_tx(bar(C::B_KF + ks), C::K_BYTES);
#pragma unroll
        for (int kb = 0; kb < C::KB; ++kb)
          ptx::tma_load_3d(sbase + C::OFF_K + ks * C::K_BYTES + kb * C::BOX, &L.tm_k, bar(C::B_KF + ks), kb * 64, x.g,
                           x.vis_start + x.col0, pol_k);
      }
      __syncwarp();
      ++nk;
      const int text0 = x.vis_start + x.n_vis;
      for (int hh = 0; ok && hh < x.nh; ++hh, ++nh) {
        const int w = nh & (kMmaWarps - 1);
        for (int tt = 0; tt < x.n_tt; ++tt) {
          const int n = w ? nq[1] : nq[0];
          const int qs = w * spw + n % spw;
          if (n >= spw && !warp_wait(bar(C::B_QE + qs), (n / spw - 1) & 1, abort_flag)) {
            ok = false;
            break;
          }
          const int boxes = x.tile_rows > kRows ? 2 : 1;   // 2 only in 256-row stages
          if (ptx::elect_one(leader)) {
            ptx::mbar_arrive_expect_tx(bar(C::B_QF + qs), boxes * C::K_BYTES);
            for (int bx = 0; bx < boxes; ++bx)
#pragma unroll
              for (int kb = 0; kb < C::KB; ++kb)
                ptx::tma_load_3d(sbase + C::OFF_Q + qs * q_bytes + kb * q_block + bx * C::BOX, &L.tm_q,
                                 bar(C::B_QF + qs), kb * 64, x.h0 + hh, text0 + tt * x.tile_rows + bx * kRows, pol_q);
          }
          __syncwarp();
          if (w) ++nq[1]; else ++nq[0];
        }
      }
    }
    if (!ok && lane == 0) record_failure(abort_flag, L.status);
    // no copy in flight at exit: the last phase issued into each stage has landed
    const volatile int never = 0;
    for (int s = 0; s < C::KS && s < nk; ++s)
      ptx::mbar_wait(bar(C::B_KF + s), ((nk - 1 - s) / C::KS) & 1, &never, kWaitTimeoutNs);
    for (int w = 0; w < kMmaWarps; ++w)
      for (int s = 0; s < spw && s < nq[w]; ++s)
        ptx::mbar_wait(bar(C::B_QF + w * spw + s), ((nq[w] - 1 - s) / spw) & 1, &never, kWaitTimeoutNs);
  } else if (warp < kWarpLse && warp >= kWarpMma) {
    constexpr uint32_t kIdesc0 = ptx::idesc_bf16_f32(kRows, 0, false, false);   // N added per tile
    const int me_w = warp - kWarpMma;
    uint32_t leader = 0;
    int first_leader = -1;
    bool same = true, issued = false;
    int nk = 0, nh = 0, nq = 0;                  // K tiles and heads so far (both warps count all), own steps
    const uint64_t dk = ptx::sdesc_sw128(sbase + C::OFF_K, 16, 1024);
    const uint64_t dq = ptx::sdesc_sw128(sbase + C::OFF_Q, 16, 1024);
    for (int u = blockIdx.x; ok && u < n_units; u += gridDim.x) {
      const Unit x = unit_at(u);
      if (x.n_tt == 0) continue;
      const int ks = nk % C::KS;
      if (!warp_wait(bar(C::B_KF + ks), (nk / C::KS) & 1, abort_flag)) {
        ok = false;
        break;
      }
      ++nk;
      const uint32_t idesc = kIdesc0 | (static_cast<uint32_t>(x.tile_rows >> 3) << 17);
      const uint64_t kd = dk + static_cast<uint64_t>(ks * C::K_BYTES >> 4);
      const int nh_end = nh + x.nh;
      for (; ok && nh < nh_end; ++nh) {
        if ((nh & (kMmaWarps - 1)) != me_w) continue;   // the other warp's head
        const int b = nh & (nb - 1);
        for (int tt = 0; tt < x.n_tt; ++tt, ++nq) {
          const int qs = me_w * spw + nq % spw;
          if (!warp_wait(bar(C::B_QF + qs), (nq / spw) & 1, abort_flag) || !buffer_free(b)) {
            ok = false;
            break;
          }
          ptx::tc_fence_after();
          const bool me = ptx::elect_one(leader);
          if (first_leader < 0) first_leader = static_cast<int>(leader);
          same = same && static_cast<int>(leader) == first_leader;
          if (me && same) {
            const uint64_t qd = dq + static_cast<uint64_t>(qs * q_bytes >> 4);
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              ptx::mma_ss(tmem + b * L.text_cols, kd + static_cast<uint64_t>(((kk / 4) * C::BOX + (kk % 4) * 32) >> 4),
                          qd + static_cast<uint64_t>(((kk / 4) * q_block + (kk % 4) * 32) >> 4), idesc,
                          kk > 0 ? 1u : 0u);
            ptx::mma_commit(bar(C::B_SF + b));
            ptx::mma_commit(bar(C::B_QE + qs));
          }
          __syncwarp();
          issued = true;
          ok = same;
          if (!ok) break;
        }
      }
      // The unit's key tile is free once this warp's MMAs on it are done (at
      // once when it has none: a commit with nothing pending arrives directly).
      if (ok) {
        if (ptx::elect_one(leader)) ptx::mma_commit(bar(C::B_KE + ks));
        same = same && (first_leader < 0 || static_cast<int>(leader) == first_leader);
        __syncwarp();
        ok = same;
      }
    }
    if (!ok) {
      if (lane == 0) record_failure(abort_flag, L.status);
      if (issued && lane == first_leader) {
        const volatile int never = 0;
        ptx::mma_commit(bar(C::B_DRAIN + me_w));
        ptx::mbar_wait(bar(C::B_DRAIN + me_w), 0, &never, kWaitTimeoutNs);
      }
    }
    __syncwarp();
  } else if (warp == kWarpLse) {
    // Per step: -LSE log2e of the tile's text rows, -inf past the tile's rows
    // or the video's text (those columns add 0). Two steps' values are in
    // flight while a third one waits for its buffer: a step takes less time
    // than a load.
    struct Step {
      float lse[kMaxText / 32];
      uint32_t bits[kKeep ? kMaxText / 32 : 1];    // per row: bit shift + i = the unit's i-th block is kept
      int shift, rows, buf;
      bool valid;
    };
    int u = blockIdx.x, hh = 0, tt = 0, nh = 0;
    Unit x{};
    auto seek = [&]() {                            // the next unit with text rows
      for (; u < n_units; u += gridDim.x) {
        x = unit_at(u);
        if (x.n_tt > 0) return;
      }
    };
    auto load = [&](Step& s) {
      s.valid = u < n_units;
      if (!s.valid) return;
      s.rows = x.tile_rows;
      s.buf = nh & (nb - 1);
      const float* lse = L.lse + static_cast<int64_t>(x.h0 + hh) * L.n_tok + x.vis_start + x.n_vis;
      [[maybe_unused]] const uint32_t* words = nullptr;
      if constexpr (kKeep) {
        const int blk0 = x.col0 / L.keep_block;    // a multiple of nblk: the unit's blocks share one word
        s.shift = blk0 & 31;
        words = L.keep + (static_cast<int64_t>(x.h0 + hh) * L.keep_words + (blk0 >> 5)) * L.n_tok + x.vis_start + x.n_vis;
      }
#pragma unroll
      for (int i = 0; i < kMaxText / 32; ++i) {
        const int r = i * 32 + lane, row = tt * x.tile_rows + r;
        const bool in = r < x.tile_rows && row < x.n_text;
        s.lse[i] = in ? __ldg(lse + row) : INFINITY;   // (no branch and no use here: the loads overlap)
        if constexpr (kKeep) {
          s.bits[i] = in ? __ldg(words + row) : 0u;
        }
      }
      if (++tt == x.n_tt) {
        tt = 0;
        ++nh;
        if (++hh == x.nh) {
          hh = 0;
          u += gridDim.x;
          seek();
        }
      }
    };
    auto put = [&](const Step& s) {
      if (!buffer_free(s.buf)) {
        ok = false;
        return;
      }
      for (int kb = 0; kb < nblk; ++kb) {
        float* row = lse_s + (s.buf * nblk + kb) * L.text_cols;
#pragma unroll
        for (int i = 0; i < kMaxText / 32; ++i)
          if (i * 32 < s.rows) {
            const float v = -1.4426950408889634f * s.lse[i];
            if constexpr (kKeep) row[i * 32 + lane] = (s.bits[i] >> (s.shift + kb)) & 1u ? v : -INFINITY;
            else row[i * 32 + lane] = v;
          }
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(bar(C::B_SF + s.buf));
    };
    seek();
    Step s0, s1, s2;
    load(s0);
    load(s1);
    while (ok && s0.valid) {
      load(s2);
      put(s0);
      if (!ok || !s1.valid) break;
      load(s0);
      put(s1);
      if (!ok || !s2.valid) break;
      load(s1);
      put(s2);
    }
    if (!ok && lane == 0) record_failure(abort_flag, L.status);
  } else {
    // Key threads: key = TMEM lane; group `grp` takes every nb-th head that has
    // text rows, in buffer grp (a video without any writes zeros, as its heads come).
    const int grp = warp >> 2, key = threadIdx.x & (kRows - 1);
    const uint32_t tbase = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const uint64_t scale2 = ptx::f2(L.scale_log2, L.scale_log2);
    const int npf = L.tokens_per_frame, w = npf < 32 ? npf : 32;
    const int log_npf = 31 - __clz(npf);           // N_v is a power of two
    const int kblk = kKeep ? key / L.keep_block : 0;   // the key's mask block within the unit
    float* red = reinterpret_cast<float*>(smem + C::OFF_RED);
    int nh = 0;                                    // heads of this CTA so far
    uint32_t step = 0;                             // steps of this group so far
    for (int u = blockIdx.x; u < n_units && grp < nb; u += gridDim.x) {
      const Unit x = unit_at(u);
      const int nkeys = min(kRows, x.n_vis - x.col0);   // a multiple of N_v
      const bool warp_ok = (warp & 3) * 32 < nkeys;     // some key of the warp exists
      for (int hh = 0; hh < x.nh; ++hh) {
        const int turn = x.n_tt > 0 ? nh++ : hh;
        if ((turn & (nb - 1)) != grp) continue;
        uint64_t a2[4] = {0, 0, 0, 0};
        for (int tt = 0; tt < x.n_tt; ++tt, ++step) {
          ok = ok && warp_wait(bar(C::B_SF + grp), step & 1u, abort_flag);
          if (ok && warp_ok) {
            ptx::tc_fence_after();
            const int valid = min(x.tile_rows, x.n_text - tt * x.tile_rows);   // columns past them add 0
            const float* lrow = lse_s + (grp * nblk + kblk) * L.text_cols;
            auto add4 = [&](const uint32_t* r, const float4& nl, int e) {
              float x0, x1, x2, x3;
              ptx::unf2(ptx::fma2(ptx::f2(__uint_as_float(r[0]), __uint_as_float(r[1])), scale2, ptx::f2(nl.x, nl.y)),
                        x0, x1);
              ptx::unf2(ptx::fma2(ptx::f2(__uint_as_float(r[2]), __uint_as_float(r[3])), scale2, ptx::f2(nl.z, nl.w)),
                        x2, x3);
              a2[(2 * e) & 3] = ptx::add2(a2[(2 * e) & 3], ptx::f2(ptx::ex2(x0), ptx::ex2(x1)));
              a2[(2 * e + 1) & 3] = ptx::add2(a2[(2 * e + 1) & 3], ptx::f2(ptx::ex2(x2), ptx::ex2(x3)));
            };
            int c0 = 0;
#pragma unroll 1
            for (; c0 + 32 <= valid; c0 += 32) {
              float4 l4[8];                        // read before the TMEM wait, which covers their latency
              uint32_t r[32];
              ptx::tmem_ld32(tbase + grp * L.text_cols + c0, r);
#pragma unroll
              for (int e = 0; e < 8; ++e) l4[e] = reinterpret_cast<const float4*>(lrow + c0)[e];
              ptx::tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 8; ++e) add4(r + 4 * e, l4[e], e);
            }
            // The last columns by 16: past the video's text rows they are the next
            // video's queries, which may be non-finite, so that their -inf LSE
            // entries alone would not keep them out of the sums.
#pragma unroll 1
            for (; c0 < valid; c0 += 16) {
              float4 l4[4];
              uint32_t r[16];
              ptx::tmem_ld16(tbase + grp * L.text_cols + c0, r);
#pragma unroll
              for (int e = 0; e < 4; ++e) l4[e] = reinterpret_cast<const float4*>(lrow + c0)[e];
              ptx::tmem_wait_ld();
              if (c0 + 16 > valid) {
#pragma unroll
                for (int e = 1; e < 16; ++e)
                  if (c0 + e >= valid) r[e] = 0u;
              }
#pragma unroll
              for (int e = 0; e < 4; ++e) add4(r + 4 * e, l4[e], e);
            }
            ptx::tc_fence_before();
          }
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(bar(C::B_SE + grp));
        }
        // Token map and frame sums of the head (a video without text rows writes 0).
        const int h = x.h0 + hh;
        float s0, s1, s2, s3;
        ptx::unf2(ptx::add2(a2[0], a2[1]), s0, s1);
        ptx::unf2(ptx::add2(a2[2], a2[3]), s2, s3);
        const bool mine = ok && key < nkeys;
        float f = key < nkeys ? (s0 + s1) + (s2 + s3) : 0.f;
        if constexpr (kKeep) {
          if (isnan(f)) f = kept_sum(L, x, h, key);
        }
        if (mine) {
          float* tok = L.tok + static_cast<int64_t>(h) * L.total_vis + x.vis_off + x.col0 + key;
          *tok = L.accumulate ? *tok + f : f;
        }
        for (int off = w / 2; off > 0; off >>= 1) f += __shfl_xor_sync(0xffffffffu, f, off);
        if (npf > 32) {
          if (lane == 0) red[warp] = f;
          ptx::bar_sync(1 + grp, kRows);
          if ((key & (npf - 1)) == 0) {
            float s = 0.f;
            for (int ww = warp; ww < warp + npf / 32; ++ww) s += red[ww];
            f = s;
          }
          ptx::bar_sync(1 + grp, kRows);           // red is read before the group's next head
        }
        if (mine && (key & (npf - 1)) == 0) {
          float* fr = L.frame + static_cast<int64_t>(h) * L.total_frames + x.frame_off + ((x.col0 + key) >> log_npf);
          *fr = L.accumulate ? *fr + f : f;
        }
      }
    }
    if (!ok && lane == 0) record_failure(abort_flag, L.status);
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc<kTmemCols>(tmem);
  }
}

template <int D, bool kKeep>
cudaError_t launch_d(const TextEvidenceLaunch& L, cudaStream_t stream) {
  using C = TeCfg<D>;
  auto kern = text_evidence_kernel<D, kKeep>;
  static PerDeviceAttr smem_once;
  cudaError_t e = raise_smem_limit(smem_once, reinterpret_cast<const void*>(kern), C::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int n_sm = sm_count();
  if (n_sm <= 0) return cudaErrorInvalidDevice;
  // Parts of a KV group's heads: the choice that ends first, by rounds of units
  // times a unit's heads (a later unit's fill runs behind the unit before it).
  TextEvidenceLaunch P = L;
  // One tile per head where it fits (8-video batch, up to 218 text rows: 340 us
  // with 256 columns, 446 with two tiles of 128 or fewer rows).
  P.text_cols = L.max_text > 128 ? 256 : 128;
  const int gq = L.hq / L.hkv, base = L.n_chunks * L.hkv;
  int64_t best = INT64_MAX;
  for (int split = 1; split <= gq; ++split) {
    const int64_t rounds = (static_cast<int64_t>(base) * split + n_sm - 1) / n_sm;
    const int64_t cost = rounds * ((gq + split - 1) / split);
    if (cost < best) {
      best = cost;
      P.head_split = split;
    }
    if (static_cast<int64_t>(base) * split >= 2 * n_sm) break;
  }
  const int n_units = base * P.head_split;
  kern<<<n_units < n_sm ? n_units : n_sm, kThreads, C::SMEM_BYTES, stream>>>(P);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_text_evidence(const TextEvidenceLaunch& L, cudaStream_t stream) {
  if (L.n_chunks == 0) return cudaSuccess;
  if (L.head_dim == 128) return L.keep ? launch_d<128, true>(L, stream) : launch_d<128, false>(L, stream);
  if (L.head_dim == 64) return L.keep ? launch_d<64, true>(L, stream) : launch_d<64, false>(L, stream);
  return cudaErrorInvalidValue;
}

}  // namespace evisel

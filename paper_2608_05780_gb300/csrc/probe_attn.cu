// Block-sparse, causal, grouped-query, varlen prefill attention for sm_103a
// (the paper's sparse probe, Sec. 3.2 Eq. 1, with exact token logits on every
// kept tile: Appendix Eq. 8 in token form and the row normalisation of Eq. 11).
//
// One CTA computes one work item: a query row tile against a list of kept kv
// tiles for two "slots" of query heads of one KV group. A slot is one 128-row
// MMA tile (one head for 128-token tiles, two heads for 64-token tiles); both
// slots use every K/V tile the CTA loads, and each slot's softmax runs while
// the tensor core works on the other slot.
//
// Warp roles (352 threads; 384 for 128-token tiles, where the softmax warpgroups
// take registers over from the third one):
//   warps 0-3  softmax + epilogue of slot 0, one thread per query row (TMEM lane)
//   warps 4-7  softmax + epilogue of slot 1
//   warp 8     block set-up (mbarriers) and the loads of Q (both slots) and
//              K_0, before the block-wide barrier; then K_j into a 3-deep ring
//   warp 10    TMA: V_j into an NS-deep ring (apart from K, so that K tiles
//              run ahead of the V waits)
//   warp 9     MMA issuer; the warp walks the tiles together and one elected
//              lane issues, per kv tile j:
//                O0 += P0_j V_j,  S0_{j+1} = Q0 K_{j+1}^T,
//                O1 += P1_j V_j,  S1_{j+1} = Q1 K_{j+1}^T
// TMEM columns per slot: S (TILE) | O (D). P_j (bf16) is written over the
// first half of its own S_j columns and read from there by the P.V MMA; the
// slot's next S is issued after that P.V, and the tcgen05 MMAs of one thread
// execute in issue order. An item with one slot (the last heads of a KV group
// with an odd head count) uses the idle slot's S columns as a second S
// buffer: S_{j+1} is computed while the softmax works on S_j.
// What bounds it (65,664 tokens, clocks per kv tile of a two-slot item): 2150 of
// tensor pipe; the MMA warp's loop (issue 2140, which blocks while the pipe is
// busy, and its waits) and each slot's chain (softmax 1215, MMAs 1050, hand-overs
// 450) both come to about 2700, so that neither alone can be improved. A K stage
// comes free one kv tile before it is needed again with two stages, about the
// latency of the load under load: the third one took the probe call from 3617 to
// 3515 us (8-video batch 3412 -> 3320, one layer of the 28-layer probe 255 -> 248);
// one pass over S, with P formed before the tile's max is known (see the
// softmax), to 3455 (3304, 246). Taking the softmax's copies after the register
// trade, so that nothing spills, took the step from 3838 to 3759 (3701 to 3660
// for the batch, 1545 to 1487 with the cross-frame partials of 24,704 tokens).
// Online softmax in fp32 (log2 domain) with lazy rescaling: the running max is
// only moved when it grows by more than 2^8, so O in TMEM is rescaled rarely.
// Every wait is bounded; on timeout the CTA records EVISEL_ETIMEOUT,
// drains its own async work and exits.
#include <cstdint>
#include <cuda_runtime.h>

#include "evisel_internal.h"
#include "sm103_ptx.cuh"

namespace evisel {
namespace {

static_assert(kSlots == 2, "the kernel runs two slots per work item");
// 128-token tiles: three warpgroups that trade registers (warp 11 has no role).
template <int TILE>
constexpr int kThreads = TILE == 128 ? 384 : 352;
constexpr int kWarpProducer = 8;   // Q, then the K ring
constexpr int kWarpMma = 9;
constexpr int kWarpVLoader = 10;   // the V ring
constexpr int kRows = 128;
constexpr int NK = 3;                  // stages of the K ring (the V ring has NS; shared memory holds no more)
constexpr float kRescaleThreshold = 8.0f;   // log2 units
constexpr int kWatch = 16;              // tiles that take their max first after one that moved
constexpr float kSharpSum = 4.f;        // row sum of a first tile (its largest P is 1) below which a row counts as sharp
constexpr int kSharpRows = 8;           // sharp rows of a warp that make it take the max first
constexpr float kLn2 = 0.69314718055994531f;

template <int TILE, int D, int NS>
struct Cfg {
  static constexpr int HP = kRows / TILE;        // query heads per slot
  static constexpr int KB = D / 64;              // 128-byte swizzle column blocks along d
  static constexpr int Q_BYTES = kRows * D * 2;  // one slot
  static constexpr int Q_BLOCK = kRows * 128;    // one column block of a slot's Q
  static constexpr int KV_BLOCK = TILE * 128;    // one column block of a K/V tile
  static constexpr int KV_BYTES = TILE * D * 2;
  static constexpr int OFF_Q = 0;                        // two slots
  static constexpr int OFF_K = OFF_Q + 2 * Q_BYTES;
  static constexpr int OFF_V = OFF_K + NK * KV_BYTES;
  static constexpr int OFF_BAR = OFF_V + NS * KV_BYTES;
  // barrier indices
  static constexpr int B_Q = 0;
  static constexpr int B_KF = 1;             // NK: K tile landed
  static constexpr int B_KE = B_KF + NK;     // NK: K tile consumed by both S MMAs
  static constexpr int B_VF = B_KE + NK;     // NS: V tile landed
  static constexpr int B_VE = B_VF + NS;     // NS: V tile consumed by both P.V MMAs
  static constexpr int B_SF = B_VE + NS;     // 2 (per slot): S_j computed
  static constexpr int B_PF = B_SF + 2;      // 2 (per slot): P_j written (128 arrivals)
  static constexpr int B_OF = B_PF + 2;      // 2 (per slot): O complete
  static constexpr int B_DRAIN = B_OF + 2;
  static constexpr int N_BARS = B_DRAIN + 1;
  static constexpr int OFF_MISC = OFF_BAR + N_BARS * 8;
  static constexpr int SMEM_USED = OFF_MISC + 16;
  // TMEM columns (32-bit): slot s occupies [s * SLOT_COLS, (s + 1) * SLOT_COLS)
  static constexpr int SLOT_COLS = TILE + D;
  static constexpr int COL_S = 0;
  static constexpr int COL_O = TILE;
  static constexpr int TMEM_COLS = (2 * SLOT_COLS <= 256) ? 256 : 512;
  // Dynamic smem requested: enough to keep TMEM demand per SM within 512 columns.
  static constexpr int SMEM_MIN = TMEM_COLS == 512 ? 117 * 1024 : 78 * 1024;
  static constexpr int SMEM_BYTES = (SMEM_USED + 1024 > SMEM_MIN) ? SMEM_USED + 1024 : SMEM_MIN;
  static_assert(SMEM_USED + 1024 <= 232448, "shared memory budget");
  static_assert((OFF_K % 1024) == 0 && (OFF_V % 1024) == 0 && (KV_BYTES % 1024) == 0, "1 KB aligned tiles");
  static_assert(2 * SLOT_COLS <= 512, "TMEM budget");
};

__device__ __forceinline__ void record_failure(volatile int* abort_flag, int* status, int code) {
  *abort_flag = 1;
  atomicExch(status, code);
}

// Bounded wait whose outcome is uniform across the warp, so that the warp stays
// converged for the warp-collective tcgen05 operations that follow.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  const bool ok = ptx::mbar_wait(bar, parity, abort_flag, kWaitTimeoutNs);
  return __all_sync(0xffffffffu, ok);
}

struct Wait {
  uint32_t bar, parity;
};
// Waits for `last` after two barriers that are usually over (their tests and the
// wait issue back to back, with one vote).
__device__ __forceinline__ bool warp_wait(Wait a, Wait b, Wait last, volatile int* abort_flag) {
  const bool seen = static_cast<int>(ptx::mbar_test(a.bar, a.parity)) & static_cast<int>(ptx::mbar_test(b.bar, b.parity)) &
                    static_cast<int>(ptx::mbar_try_wait(last.bar, last.parity));
  if (__all_sync(0xffffffffu, seen)) return true;
  return warp_wait(a.bar, a.parity, abort_flag) && warp_wait(b.bar, b.parity, abort_flag) &&
         warp_wait(last.bar, last.parity, abort_flag);
}

// Heads of the item's KV group from its first head on.
__device__ __forceinline__ int heads_left(const ProbeLaunch& L, int head) {
  const int gq = L.hq / L.hkv;
  return gq - head % gq;
}

// Block set-up by the K loader's first lane, before the block-wide barrier:
// the mbarriers and the abort flag, then the loads that the first S MMAs
// wait for (Q of both slots and K tile 0), so that their latency overlaps the
// TMEM allocation and the barrier instead of following them.
template <int TILE, int D, int NS>
__device__ __forceinline__ void setup_and_first_loads(const ProbeLaunch& L, const WorkItem& it, uint32_t sbase,
                                                      volatile int* abort_flag) {
  using C = Cfg<TILE, D, NS>;
  auto bar = [&](int i) { return sbase + C::OFF_BAR + 8u * i; };
  for (int i = 0; i < C::N_BARS; ++i) {
    const bool softmax_arrive = (i == C::B_PF || i == C::B_PF + 1);
    ptx::mbar_init(bar(i), softmax_arrive ? kRows : 1u);
  }
  *abort_flag = 0;
  ptx::fence_mbar_init();
  ptx::tma_prefetch_desc(&L.tm_q);
  ptx::tma_prefetch_desc(&L.tm_k);
  ptx::tma_prefetch_desc(&L.tm_v);
  const int left = heads_left(L, it.head);
  const int nslots = left > C::HP ? 2 : 1;
  const uint64_t pol_q = ptx::l2_policy_evict_first();
  ptx::mbar_arrive_expect_tx(bar(C::B_Q), nslots * C::Q_BYTES);
  for (int slot = 0; slot < nslots; ++slot) {
#pragma unroll
    for (int hp = 0; hp < C::HP; ++hp) {
      // A head past the group's end loads the first head again; its rows are never stored.
      const int h = slot * C::HP + hp < left ? it.head + slot * C::HP + hp : it.head;
#pragma unroll
      for (int kb = 0; kb < C::KB; ++kb)
        ptx::tma_load_3d(sbase + C::OFF_Q + slot * C::Q_BYTES + kb * C::Q_BLOCK + hp * TILE * 128, &L.tm_q,
                         bar(C::B_Q), kb * 64, h, it.q_start, pol_q);
    }
  }
  if (it.kv_count > 0) {
    const int g = it.head / (L.hq / L.hkv);
    ptx::mbar_arrive_expect_tx(bar(C::B_KF), C::KV_BYTES);
#pragma unroll
    for (int kb = 0; kb < C::KB; ++kb)
      ptx::tma_load_3d(sbase + C::OFF_K + kb * C::KV_BLOCK, &L.tm_k, bar(C::B_KF), kb * 64, g,
                       L.kv[it.kv_begin].start, ptx::l2_policy_evict_last());
  }
}

// One TMA warp per ring, so that K tiles run ahead of the V waits. Q and K
// tile 0 were sent by setup_and_first_loads; the K warp goes on from K tile 1.
template <int TILE, int D, int NS, bool IS_V>
__device__ __forceinline__ void producer(const ProbeLaunch& L, const WorkItem& it, uint32_t sbase_in,
                                         volatile int* abort_flag) {
  using C = Cfg<TILE, D, NS>;
  const uint32_t sbase = __shfl_sync(0xffffffffu, sbase_in, 0);
  auto bar = [&](int i) { return sbase + C::OFF_BAR + 8u * i; };
  const int head0 = __shfl_sync(0xffffffffu, it.head, 0);
  const int n = __shfl_sync(0xffffffffu, it.kv_count, 0);
  const int kv_begin = __shfl_sync(0xffffffffu, it.kv_begin, 0);
  const int g = head0 / (L.hq / L.hkv);
  const uint64_t pol_kv = ptx::l2_policy_evict_last();
  uint32_t leader = 0;

  const CUtensorMap* map = IS_V ? &L.tm_v : &L.tm_k;
  const int off = IS_V ? C::OFF_V : C::OFF_K;
  const int b_full = IS_V ? C::B_VF : C::B_KF;
  const int b_empty = IS_V ? C::B_VE : C::B_KE;
  constexpr int R = IS_V ? NS : NK;              // ring stages
  const int first = (IS_V || n == 0) ? 0 : 1;   // K tile 0 went out with the set-up
  int issued = first;
  for (int j = first; j < n; ++j) {
    const int s = j % R;
    const int u = j / R;
    const int kv_start = __shfl_sync(0xffffffffu, L.kv[kv_begin + j].start, 0);
    if (u > 0 && !warp_wait(bar(b_empty + s), (u - 1) & 1, abort_flag)) {
      if ((threadIdx.x & 31) == leader) record_failure(abort_flag, L.status, kStatusTimeout);
      break;
    }
    if (ptx::elect_one(leader)) {
      ptx::mbar_arrive_expect_tx(bar(b_full + s), C::KV_BYTES);
#pragma unroll
      for (int kb = 0; kb < C::KB; ++kb)
        ptx::tma_load_3d(sbase + off + s * C::KV_BYTES + kb * C::KV_BLOCK, map, bar(b_full + s), kb * 64, g, kv_start,
                         pol_kv);
    }
    __syncwarp();
    issued = j + 1;
  }
  {
    // Drain: every load issued here completes on its own; wait for the last
    // phase issued into each stage (and for Q) so that no copy is in flight
    // when the CTA exits, whether or not another warp gave up.
    const volatile int never = 0;
    if (!IS_V) ptx::mbar_wait(bar(C::B_Q), 0, &never, kWaitTimeoutNs);
    for (int s = 0; s < R && s < issued; ++s) {
      const int last = ((issued - 1 - s) / R) * R + s;
      ptx::mbar_wait(bar(b_full + s), (last / R) & 1, &never, kWaitTimeoutNs);
    }
  }
}

// The whole warp walks the tiles on warp-uniform values; one elected lane
// issues every MMA and commit. tcgen05.commit tracks the MMAs of the thread
// that issues it, so the lane must not change: elect.sync picks the same lane
// of a converged warp, and a change is treated as a failure.
template <int TILE, int D, int NS>
__device__ __forceinline__ void mma_issuer(const ProbeLaunch& L, const WorkItem& it, uint32_t sbase_in,
                                           uint32_t tmem_in, volatile int* abort_flag) {
  using C = Cfg<TILE, D, NS>;
  const uint32_t sbase = __shfl_sync(0xffffffffu, sbase_in, 0);
  const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_in, 0);
  const int n = __shfl_sync(0xffffffffu, it.kv_count, 0);
  const bool two = heads_left(L, __shfl_sync(0xffffffffu, it.head, 0)) > C::HP;
  auto bar = [&](int i) { return sbase + C::OFF_BAR + 8u * i; };
  constexpr uint32_t kIdescS = ptx::idesc_bf16_f32(kRows, TILE, false, false);
  constexpr uint32_t kIdescO = ptx::idesc_bf16_f32(kRows, D, false, true);
  uint32_t leader = 0;
  int first_leader = -1;
  bool same_leader = true;
  auto elect = [&]() -> bool {
    const bool me = ptx::elect_one(leader);
    if (first_leader < 0) first_leader = static_cast<int>(leader);
    same_leader = same_leader && static_cast<int>(leader) == first_leader;
    return me && same_leader;
  };
  // Descriptors of every operand buffer, built once; a k-step adds its byte
  // offset / 16 to the address field (the lowest bits; smem offsets < 256 KB
  // never carry out of it).
  const uint64_t dq0 = ptx::sdesc_sw128(sbase + C::OFF_Q, 16, 1024);
  const uint64_t dq1 = ptx::sdesc_sw128(sbase + C::OFF_Q + C::Q_BYTES, 16, 1024);
  const uint64_t dk0 = ptx::sdesc_sw128(sbase + C::OFF_K, 16, 1024);
  const uint64_t dv0 = ptx::sdesc_sw128(sbase + C::OFF_V, C::KV_BLOCK, 1024);
  const uint64_t dv1 = ptx::sdesc_sw128(sbase + C::OFF_V + C::KV_BYTES, C::KV_BLOCK, 1024);
  static_assert(NS == 2, "two ring stages");
  // S[buf] = Q_slot K_j^T (buf: whose S columns receive it)
  auto mma_s = [&](int slot, int j, int buf) {
    const uint64_t qd = slot ? dq1 : dq0;
    const uint64_t kd = dk0 + static_cast<uint64_t>((j % NK) * C::KV_BYTES >> 4);
    const uint32_t d_tmem = tmem + buf * C::SLOT_COLS + C::COL_S;
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
      const uint64_t a = qd + static_cast<uint64_t>(((kk / 4) * C::Q_BLOCK + (kk % 4) * 32) >> 4);
      const uint64_t bd = kd + static_cast<uint64_t>(((kk / 4) * C::KV_BLOCK + (kk % 4) * 32) >> 4);
      ptx::mma_ss(d_tmem, a, bd, kIdescS, kk > 0 ? 1u : 0u);
    }
  };
  // O_slot += P V_j, P from the first TILE/2 columns of S[buf].
  auto mma_pv = [&](int slot, int j, int buf) {
    const uint64_t vd = (j & 1) ? dv1 : dv0;
    const uint32_t d_tmem = tmem + slot * C::SLOT_COLS + C::COL_O;
    const uint32_t p_tmem = tmem + buf * C::SLOT_COLS + C::COL_S;
#pragma unroll
    for (int kk = 0; kk < TILE / 16; ++kk) {
      const uint64_t bd = vd + static_cast<uint64_t>((kk * 16 * 128) >> 4);
      ptx::mma_ts(d_tmem, p_tmem + kk * 8, bd, kIdescO, (j > 0 || kk > 0) ? 1u : 0u);
    }
  };

  bool issued = false;
  bool ok = warp_wait(bar(C::B_Q), 0, abort_flag) && warp_wait(bar(C::B_KF), 0, abort_flag);
  if (!two) {
    // One slot: the second slot's S columns double-buffer S, so S_{j+1} is
    // ready while the softmax works on S_j. Tile j uses buffer b = j & 1
    // (barriers SF[b] / PF[b], phase j >> 1); S_{j+2} reuses b after P_j.V.
    if (ok) {
      ptx::tc_fence_after();
      if (elect()) {
        mma_s(0, 0, 0);
        ptx::mma_commit(bar(C::B_SF));
        ptx::mma_commit(bar(C::B_KE));
      }
      __syncwarp();
      issued = true;
      ok = same_leader;
    }
    if (ok && n > 1) {
      if (!warp_wait(bar(C::B_KF + 1), 0, abort_flag)) {
        ok = false;
      } else {
        if (elect()) {
          mma_s(0, 1, 1);
          ptx::mma_commit(bar(C::B_SF + 1));
          ptx::mma_commit(bar(C::B_KE + 1));
        }
        __syncwarp();
        ok = same_leader;
      }
    }
    for (int j = 0; ok && j < n; ++j) {
      const int b = j & 1;
      const int s = j % NS;
      const int s2 = (j + 2) % NK;
      const bool more = j + 2 < n;
      const Wait v{bar(C::B_VF + s), static_cast<uint32_t>(j / NS) & 1u};
      const Wait kn = more ? Wait{bar(C::B_KF + s2), static_cast<uint32_t>((j + 2) / NK) & 1u} : v;
      if (!warp_wait(v, kn, Wait{bar(C::B_PF + b), static_cast<uint32_t>(j >> 1) & 1u}, abort_flag)) {
        ok = false;
        break;
      }
      ptx::tc_fence_after();
      if (elect()) {
        mma_pv(0, j, b);
        if (j + 1 == n) ptx::mma_commit(bar(C::B_OF));
        ptx::mma_commit(bar(C::B_VE + s));
        if (more) {
          mma_s(0, j + 2, b);
          ptx::mma_commit(bar(C::B_SF + b));
          ptx::mma_commit(bar(C::B_KE + s2));
        }
      }
      __syncwarp();
      ok = same_leader;
    }
  } else {
    if (ok) {
      ptx::tc_fence_after();
      if (elect()) {
        mma_s(0, 0, 0);
        ptx::mma_commit(bar(C::B_SF));
        mma_s(1, 0, 1);
        ptx::mma_commit(bar(C::B_SF + 1));
        ptx::mma_commit(bar(C::B_KE));
      }
      __syncwarp();
      issued = true;
      ok = same_leader;
    }
    for (int j = 0; ok && j < n; ++j) {
      const int s = j % NS;
      const int s1 = (j + 1) % NK;
      const bool more = j + 1 < n;
      // The K/V tiles landed long ago in steady state: they are tested together
      // with P0, whose arrival starts P0.V and the next S0 at once.
      const Wait v{bar(C::B_VF + s), static_cast<uint32_t>(j / NS) & 1u};
      const Wait kn = more ? Wait{bar(C::B_KF + s1), static_cast<uint32_t>((j + 1) / NK) & 1u} : v;
      if (!warp_wait(v, kn, Wait{bar(C::B_PF), static_cast<uint32_t>(j) & 1u}, abort_flag)) {
        ok = false;
        break;
      }
      ptx::tc_fence_after();
      // slot 0: P.V of tile j, then S of tile j + 1
      if (elect()) {
        mma_pv(0, j, 0);
        if (!more) ptx::mma_commit(bar(C::B_OF));
        if (more) {
          mma_s(0, j + 1, 0);
          ptx::mma_commit(bar(C::B_SF));
        }
      }
      __syncwarp();
      // slot 1: P.V of tile j, then S of tile j + 1
      if (!warp_wait(bar(C::B_PF + 1), j & 1, abort_flag)) {
        ok = false;
        break;
      }
      ptx::tc_fence_after();
      if (elect()) {
        mma_pv(1, j, 1);
        if (!more) ptx::mma_commit(bar(C::B_OF + 1));
        ptx::mma_commit(bar(C::B_VE + s));
        if (more) {
          mma_s(1, j + 1, 1);
          ptx::mma_commit(bar(C::B_SF + 1));
          ptx::mma_commit(bar(C::B_KE + s1));
        }
      }
      __syncwarp();
      ok = same_leader;
    }
  }
  const int lane = threadIdx.x & 31;
  if (!ok) {
    if (lane == 0) record_failure(abort_flag, L.status, kStatusTimeout);
    // Wait for every MMA the issuing lane started before TMEM is released.
    if (issued && lane == first_leader) {
      const volatile int never = 0;
      ptx::mma_commit(bar(C::B_DRAIN));
      ptx::mbar_wait(bar(C::B_DRAIN), 0, &never, kWaitTimeoutNs);
    }
  }
  __syncwarp();
}

template <int TILE, int D, int NS, int FSW, int EMB>
__device__ __forceinline__ void softmax_epilogue(const ProbeLaunch& L, const WorkItem& it, int slot, uint32_t sbase,
                                                 uint32_t tmem_base, volatile int* abort_flag) {
  using C = Cfg<TILE, D, NS>;
  auto bar = [&](int i) { return sbase + C::OFF_BAR + 8u * i; };
  const int left = heads_left(L, it.head);
  if (slot * C::HP >= left) return;            // the item has one slot only
  const int warp = (threadIdx.x >> 5) & 3;
  const int row = threadIdx.x & 127;           // TMEM lane
  const int hp = row / TILE;
  const int row_local = row % TILE;
  const bool head_ok = slot * C::HP + hp < left;
  const int head = it.head + slot * C::HP + hp;
  const bool row_ok = head_ok && row_local < it.q_len;
  const int qpos = it.q_start + row_local;
  const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
  const uint32_t tmem = tmem_base + lane_base + slot * C::SLOT_COLS;
  // With one slot, S alternates between both slots' S columns (see the MMA issuer).
  const bool two = left > C::HP;

  // Cross-frame partials (visual rows, when enabled): per kept kv tile and
  // key frame f, m + log2(sum of the frame's P) in log2 units, so that the
  // frame's share of the row's softmax is exp2(value - LSE log2 e).
  // FSW = the key span of one partial, min(N_v, 64), in the instantiation that
  // keeps them (0: not kept), so that the span ends are compile-time positions
  // and the plain probe is unchanged.
  float* fs_row = nullptr;
  if constexpr (FSW > 0) {
    if (it.text_row0 < 0 && row_ok)
      fs_row = L.fspill + (static_cast<int64_t>(head) * L.fs_nnz + it.kv_begin) * (TILE / FSW) * TILE + row_local;
  }

  // Per-row block masks (EMB = their block size; 0: none): the row's bit per
  // block of its video (top-p retention and the own block), applied to the
  // keys of every kv tile before the max and P.
  [[maybe_unused]] const uint32_t* em_row = nullptr;
  [[maybe_unused]] int em_vis_start = 0, em_n_vis = 0;
  if constexpr (EMB > 0) {
    const VideoInfo evi = L.videos[it.video];
    em_vis_start = evi.vis_start;
    em_n_vis = evi.n_vis;
    if (row_ok) em_row = L.keep + static_cast<int64_t>(head) * L.keep_words * L.n_tok + qpos;
  }

  float m_used = -INFINITY;   // running max, log2 units
  float l_sum = 0.f;
  bool ok = true;
  const uint64_t scale2 = ptx::f2(L.scale_log2, L.scale_log2);

  // With per-row masks (EMB) the kv tiles are read two tiles ahead and the
  // row's mask word one tile ahead, so that no global load waits between an
  // S-ready wait and the softmax that follows it. Without them the tile is
  // read before its S-ready wait, which covers the load.
  auto load_kv = [&](int jj) { return jj < it.kv_count ? L.kv[it.kv_begin + jj] : KvTile{0, 0, 0, 0}; };
  [[maybe_unused]] auto mask_word = [&](const KvTile& t) -> uint32_t {
    uint32_t w = 0xffffffffu;   // bit q: the tile's q-th block is attended
    if constexpr (EMB > 0) {
      if (em_row) {
        const int blk0 = t.visual ? (t.start - em_vis_start) / EMB
                                  : em_n_vis / EMB + (t.start - em_vis_start - em_n_vis) / EMB;
        w = em_row[static_cast<int64_t>(blk0 >> 5) * L.n_tok] >> (blk0 & 31);
      }
    }
    return w;
  };
  [[maybe_unused]] KvTile kv_next{0, 0, 0, 0}, kv_after{0, 0, 0, 0};
  [[maybe_unused]] uint32_t em_next = 0xffffffffu;
  if constexpr (EMB > 0) {
    kv_next = load_kv(0);
    kv_after = load_kv(1);
    if (it.kv_count > 0) em_next = mask_word(kv_next);
  }

  // Warp-uniform: tiles to go that take their max before P. A tile formed early
  // that has to be formed again costs about half a tile more, the early start
  // gains a twentieth: after a maximum that moved the next kWatch tiles take the
  // max first, and likewise after a first tile whose row sums say that a few
  // keys hold the mass (sharp logits, whose maxima keep moving): a quarter of the
  // warp's rows, since one row that moves makes the warp form the tile again.
  // Watching one tile only took 3,115 us where the max first everywhere took
  // 2,814 (two videos of 48,000 visual tokens, logits of std 16), this rule 2,845;
  // 64 for 16 the same. Rows with few keys in the first tile or none (above the
  // diagonal, past the tile's rows, dropped by the row's mask) count as sharp:
  // their maxima are still to come. Leaving them out took the sparse layer of
  // 24,704 tokens from 1,096 to 1,107 us and made nothing else faster by more
  // than 0.3%.
  int watch = 1;
  for (int j = 0; j < it.kv_count; ++j) {
    KvTile kv;
    [[maybe_unused]] uint32_t em_bits = 0xffffffffu;
    if constexpr (EMB > 0) {
      kv = kv_next;
      em_bits = em_next;
      kv_next = kv_after;
      if (j + 1 < it.kv_count) em_next = mask_word(kv_next);   // kv_next was read a tile ago
      kv_after = load_kv(j + 2);
    } else {
      kv = L.kv[it.kv_begin + j];
    }
    const int b = two ? slot : (j & 1);
    const uint32_t par = two ? (j & 1) : ((j >> 1) & 1);
    const uint32_t tS = tmem_base + lane_base + b * C::SLOT_COLS + C::COL_S;
    const uint32_t bar_pf = bar(C::B_PF + b);
    if (!warp_wait(bar(C::B_SF + b), par, abort_flag)) { ok = false; break; }
    ptx::tc_fence_after();
    int limit = TILE;                        // keys from here on are masked:
    if (kv.diag || kv.len < TILE) {          // past the tile's end (ragged tile) or above the diagonal
      limit = kv.len;
      if (kv.diag) limit = min(limit, qpos - kv.start + 1);
    }
    // 64 columns of the row's S: masks, then max.
    auto mask64 = [&](uint32_t (&r)[2][32], int h) {
      if constexpr (EMB > 0) {
        if ((em_bits & ((1u << (TILE / EMB)) - 1u)) != (1u << (TILE / EMB)) - 1u) {
#pragma unroll
          for (int c = 0; c < 64; ++c)
            if (!((em_bits >> ((h * 64 + c) / EMB)) & 1u)) r[c / 32][c % 32] = 0xff800000u;   // -inf
        }
      }
      if (limit < TILE) {
#pragma unroll
        for (int c = 0; c < 64; ++c)
          if (h * 64 + c >= limit) r[c / 32][c % 32] = 0xff800000u;
      }
    };
    auto max64 = [&](const uint32_t (&r)[2][32], float (&m4)[4]) {
#pragma unroll
      for (int c = 0; c < 64; c += 8) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          m4[e] = ptx::max3(m4[e], __uint_as_float(r[c / 32][c % 32 + 2 * e]),
                            __uint_as_float(r[c / 32][c % 32 + 2 * e + 1]));
      }
    };
    auto load64 = [&](uint32_t (&r)[2][32], int h) {
      ptx::tmem_ld32(tS + h * 64, r[0]);
      ptx::tmem_ld32(tS + h * 64 + 32, r[1]);
    };
    [[maybe_unused]] float* fs_tile = nullptr;
    if constexpr (FSW > 0) {
      if (fs_row) fs_tile = fs_row + static_cast<int64_t>(j) * (TILE / FSW) * TILE;
    }
    uint64_t l2[4];
    [[maybe_unused]] float l_tile;
    float m_safe;
    uint64_t negm2;
    // P of 32 columns (q-th quarter of the tile): 2^(s * scale * log2 e - m) in
    // packed pairs, as bf16 into pk.
    auto p32 = [&](const uint32_t (&r)[32], int q, uint32_t (&pk)[32]) {
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        float x0, x1;
        ptx::unf2(ptx::fma2(ptx::f2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1])), scale2, negm2), x0, x1);
        const float p0 = ptx::ex2(x0);
        const float p1 = ptx::ex2(x1);
        l2[e & 3] = ptx::add2(l2[e & 3], ptx::f2(p0, p1));
        pk[(q & 1) * 16 + e] = ptx::pack_bf16x2(p0, p1);
        if constexpr (FSW > 0) {
          if ((q * 32 + 2 * e + 2) % FSW == 0) {      // the last keys of span (q * 32 + 2e + 2) / FSW - 1
            float a0, a1, b0, b1, c0, c1, d0, d1;
            ptx::unf2(l2[0], a0, a1);
            ptx::unf2(l2[1], b0, b1);
            ptx::unf2(l2[2], c0, c1);
            ptx::unf2(l2[3], d0, d1);
            const float fsum = ((a0 + a1) + (b0 + b1)) + ((c0 + c1) + (d0 + d1));
            l_tile += fsum;
            l2[0] = l2[1] = l2[2] = l2[3] = 0;
            if (fs_tile)
              __stcs(fs_tile + ((q * 32 + 2 * e + 2) / FSW - 1) * TILE, fsum > 0.f ? m_safe + __log2f(fsum) : -INFINITY);
          }
        }
      }
    };
    auto begin_p = [&]() {
      m_safe = (m_used == -INFINITY) ? 0.f : m_used;
      negm2 = ptx::f2(-m_safe, -m_safe);
      l2[0] = l2[1] = l2[2] = l2[3] = 0;
      l_tile = 0.f;
    };

    uint32_t ra[2][32], rb[2][32], pk[32];   // S: first and second half of the tile
    bool max_first = TILE == 64 || watch > 0;    // (a 64-key tile gains nothing from the early half)
    if (!max_first) {
      // The running max holds for nearly every tile: P of the first half is
      // formed with it while the tile's max is taken, and stands if no row of
      // the warp needs a larger one. The second half loads meanwhile.
      begin_p();
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      load64(ra, 0);
      ptx::tmem_wait_ld();
      if constexpr (TILE == 128) load64(rb, 1);
      mask64(ra, 0);
      max64(ra, m4);
      p32(ra[0], 0, pk);
      if constexpr (TILE == 128) {
        ptx::tmem_wait_ld();
        mask64(rb, 1);
        max64(rb, m4);
      }
      p32(ra[1], 1, pk);
      const float m_tile = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * L.scale_log2;
      max_first = __any_sync(0xffffffffu, m_tile > m_used + kRescaleThreshold);
    }
    if (max_first) {
      // The first tile, a row whose max grew by more than 2^8, or the tiles after
      // such a one (maxima that move tend to move again): the max first, then
      // the lazy rescale of the row sum and (not on the first tile) of the O
      // accumulator. With two slots S_j was issued after P_{j-1}.V, so that
      // MMA has completed; with one slot it is waited for (its V-empty barrier).
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      load64(ra, 0);
      if constexpr (TILE == 128) load64(rb, 1);
      ptx::tmem_wait_ld();
      mask64(ra, 0);
      max64(ra, m4);
      if constexpr (TILE == 128) {
        mask64(rb, 1);
        max64(rb, m4);
      }
      const float m_tile = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * L.scale_log2;
      const bool need = m_tile > m_used + kRescaleThreshold;
      const bool moved = __any_sync(0xffffffffu, need);
      watch = moved ? kWatch : watch - 1;
      const float alpha = need ? ptx::ex2(m_used - m_tile) : 1.f;
      l_sum *= alpha;
      m_used = need ? m_tile : m_used;
      if (moved && j > 0) {
        if (!two && !warp_wait(bar(C::B_VE + (j - 1) % NS), ((j - 1) / NS) & 1, abort_flag)) {
          ok = false;
          break;
        }
        ptx::tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < D / 16; ++c) {
          uint32_t o[16];
          ptx::tmem_ld16(tmem + C::COL_O + c * 16, o);
          ptx::tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
          ptx::tmem_st16(tmem + C::COL_O + c * 16, o);
        }
      }
      begin_p();
      p32(ra[0], 0, pk);
      p32(ra[1], 1, pk);
    }
    // P over the first half of S.
    ptx::tmem_st32(tS, pk);
    if constexpr (TILE == 128) {
      p32(rb[0], 2, pk);
      p32(rb[1], 3, pk);
      ptx::tmem_st32(tS + 32, pk);
    }
    if constexpr (FSW > 0) {
      l_sum += l_tile;
    } else {
      float a0, a1, b0, b1, c0, c1, d0, d1;
      ptx::unf2(l2[0], a0, a1);
      ptx::unf2(l2[1], b0, b1);
      ptx::unf2(l2[2], c0, c1);
      ptx::unf2(l2[3], d0, d1);
      l_sum += ((a0 + a1) + (b0 + b1)) + ((c0 + c1) + (d0 + d1));
    }
    ptx::tmem_wait_st();
    ptx::tc_fence_before();
    ptx::mbar_arrive(bar_pf);
    if (TILE == 128 && j == 0) watch = __popc(__ballot_sync(0xffffffffu, l_sum < kSharpSum)) >= kSharpRows ? kWatch : 0;
  }

  ok = ok && warp_wait(bar(C::B_OF + slot), 0, abort_flag);
  if (!ok) record_failure(abort_flag, L.status, kStatusTimeout);
  ptx::tc_fence_after();

  const float inv_l = l_sum > 0.f ? 1.f / l_sum : 0.f;
  if (it.part < 0 && it.q_len == TILE) {
    // Every warp of the slot reaches the named barrier below, whether or not
    // one of them gave up on a wait, so that the barrier always completes;
    // the barrier then tells all 128 threads whether to store.
    // Full tile: the slot's O goes through its Q region of shared memory (no
    // MMA reads Q any more) in Q's swizzled layout, then out by TMA stores of
    // one 64-column block of one head each: whole 128-byte rows instead of 16
    // bytes per row and store.
    const uint32_t stage = sbase + C::OFF_Q + slot * C::Q_BYTES + hp * TILE * 128 + row_local * 128;
    if (ok) {
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        uint32_t r[32];
        ptx::tmem_ld32(tmem + C::COL_O + c * 32, r);
        ptx::tmem_wait_ld();
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
          uint4 w;
          w.x = ptx::pack_bf16x2(__uint_as_float(r[8 * q4 + 0]) * inv_l, __uint_as_float(r[8 * q4 + 1]) * inv_l);
          w.y = ptx::pack_bf16x2(__uint_as_float(r[8 * q4 + 2]) * inv_l, __uint_as_float(r[8 * q4 + 3]) * inv_l);
          w.z = ptx::pack_bf16x2(__uint_as_float(r[8 * q4 + 4]) * inv_l, __uint_as_float(r[8 * q4 + 5]) * inv_l);
          w.w = ptx::pack_bf16x2(__uint_as_float(r[8 * q4 + 6]) * inv_l, __uint_as_float(r[8 * q4 + 7]) * inv_l);
          // 16-byte chunk k of the row's 128-byte block kb sits at chunk k ^ (row & 7).
          const int kb = c / 2, k = (c % 2) * 4 + q4;
          const uint32_t addr = stage + kb * C::Q_BLOCK + ((k ^ (row_local & 7)) << 4);
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w.x), "r"(w.y), "r"(w.z), "r"(w.w)
                       : "memory");
        }
      }
    }
    if (ok && row_ok) L.lse[static_cast<int64_t>(head) * L.n_tok + qpos] = (m_used + __log2f(l_sum)) * kLn2;
    ptx::fence_proxy_async_smem();
    const bool all_ok = ptx::bar_and(1 + slot, kRows, ok);
    if (all_ok && (threadIdx.x & 127) == 0) {
#pragma unroll
      for (int h = 0; h < C::HP; ++h) {
        if (slot * C::HP + h >= left) break;   // heads past the group's end are not stored
#pragma unroll
        for (int kb = 0; kb < C::KB; ++kb)
          ptx::tma_store_3d(&L.tm_o, sbase + C::OFF_Q + slot * C::Q_BYTES + kb * C::Q_BLOCK + h * TILE * 128, kb * 64,
                            it.head + slot * C::HP + h, it.q_start);
      }
      ptx::bulk_commit();
      ptx::bulk_wait_read();   // the shared memory source must outlive the copy
    }
  } else if (!ok) {
    return;
  } else if (it.part < 0) {
    uint4* dst = reinterpret_cast<uint4*>(static_cast<uint16_t*>(L.o) +
                                          (static_cast<int64_t>(qpos) * L.hq + head) * D);
#pragma unroll
    for (int c = 0; c < D / 32; ++c) {
      uint32_t r[32];
      ptx::tmem_ld32(tmem + C::COL_O + c * 32, r);
      ptx::tmem_wait_ld();
      if (row_ok) {
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
          uint4 w;
          w.x = ptx::pack_bf16x2(__uint_as_float(r[8 * q4 + 0]) * inv_l, __uint_as_float(r[8 * q4 + 1]) * inv_l);
          w.y = ptx::pack_bf16x2(__uint_as_float(r[8 * q4 + 2]) * inv_l, __uint_as_float(r[8 * q4 + 3]) * inv_l);
          w.z = ptx::pack_bf16x2(__uint_as_float(r[8 * q4 + 4]) * inv_l, __uint_as_float(r[8 * q4 + 5]) * inv_l);
          w.w = ptx::pack_bf16x2(__uint_as_float(r[8 * q4 + 6]) * inv_l, __uint_as_float(r[8 * q4 + 7]) * inv_l);
          dst[c * 4 + q4] = w;
        }
      }
    }
    if (row_ok) L.lse[static_cast<int64_t>(head) * L.n_tok + qpos] = (m_used + __log2f(l_sum)) * kLn2;
  } else {
    const int64_t part = it.part + slot;
    float4* dst = reinterpret_cast<float4*>(L.part_o + (part * kRows + row) * D);
#pragma unroll
    for (int c = 0; c < D / 32; ++c) {
      uint32_t r[32];
      ptx::tmem_ld32(tmem + C::COL_O + c * 32, r);
      ptx::tmem_wait_ld();
#pragma unroll
      for (int q4 = 0; q4 < 8; ++q4)
        dst[c * 8 + q4] = make_float4(__uint_as_float(r[4 * q4]), __uint_as_float(r[4 * q4 + 1]),
                                      __uint_as_float(r[4 * q4 + 2]), __uint_as_float(r[4 * q4 + 3]));
    }
    L.part_ml[part * kRows + row] = make_float2(m_used, l_sum);
  }
}

template <int TILE, int D, int NS, int FSW, int EMB>
__global__ void __launch_bounds__(kThreads<TILE>, 1) probe_attn_kernel(const __grid_constant__ ProbeLaunch L) {
  using C = Cfg<TILE, D, NS>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = ptx::smem_addr(smem);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_MISC + 4);
  const int warp = threadIdx.x >> 5;
  const WorkItem it = L.items[blockIdx.x];

  if (threadIdx.x == kWarpProducer * 32) setup_and_first_loads<TILE, D, NS>(L, it, sbase, abort_flag);
  if (warp == 0) {
    ptx::tmem_alloc<C::TMEM_COLS>(sbase + C::OFF_MISC);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();

  // 256 x 192 + 128 x 120 = 384 x 168 registers, what the launch holds: the
  // softmax keeps a whole row of S and its P. What is live at the switch stays
  // under the launch's 168, so the softmax takes its own copies of the item, the
  // shared-memory base and the TMEM address after it (without them, or with 88
  // for the other warps, up to 5 registers spill).
  if (warp >= kWarpProducer) {
    if constexpr (TILE == 128) ptx::setmaxnreg_dec<120>();
    if (warp == kWarpProducer) producer<TILE, D, NS, false>(L, it, sbase, abort_flag);
    else if (warp == kWarpVLoader) producer<TILE, D, NS, true>(L, it, sbase, abort_flag);
    else if (warp == kWarpMma) mma_issuer<TILE, D, NS>(L, it, sbase, *tmem_slot, abort_flag);
  } else {
    if constexpr (TILE == 128) ptx::setmaxnreg_inc<192>();
    const WorkItem own = L.items[blockIdx.x];
    uint32_t own_base = sbase;
    asm volatile("" : "+r"(own_base));
    softmax_epilogue<TILE, D, NS, FSW, EMB>(L, own, warp / 4, own_base, *tmem_slot, abort_flag);
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc<C::TMEM_COLS>(*tmem_slot);
  }
}

template <int TILE, int D, int FSW, int EMB = 0>
cudaError_t launch_cfg(const ProbeLaunch& L, cudaStream_t stream) {
  constexpr int NS = 2;
  using C = Cfg<TILE, D, NS>;
  auto kern = probe_attn_kernel<TILE, D, NS, FSW, EMB>;
  static PerDeviceAttr smem_once;
  cudaError_t e = raise_smem_limit(smem_once, reinterpret_cast<const void*>(kern), C::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  kern<<<L.n_items, kThreads<TILE>, C::SMEM_BYTES, stream>>>(L);
  return cudaGetLastError();
}

// The plain probe (fsw = 0) or the one that keeps cross-frame partials over
// key spans of fsw tokens (16, 32 or 64).
template <int TILE, int D>
cudaError_t launch_fsw(const ProbeLaunch& L, int fsw, cudaStream_t stream) {
  if (L.keep) {                                  // per-row block masks (not with cross-frame partials)
    if (fsw != 0) return cudaErrorInvalidValue;
    switch (L.keep_block) {
      case 16: return launch_cfg<TILE, D, 0, 16>(L, stream);
      case 32: return launch_cfg<TILE, D, 0, 32>(L, stream);
      case 64: return launch_cfg<TILE, D, 0, 64>(L, stream);
      case 128:
        if constexpr (TILE == 128) return launch_cfg<TILE, D, 0, 128>(L, stream);
        return cudaErrorInvalidValue;
      default: return cudaErrorInvalidValue;
    }
  }
  switch (fsw) {
    case 0: return launch_cfg<TILE, D, 0>(L, stream);
    case 16: return launch_cfg<TILE, D, 16>(L, stream);
    case 32: return launch_cfg<TILE, D, 32>(L, stream);
    case 64: return launch_cfg<TILE, D, 64>(L, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_probe_attn(const ProbeLaunch& L, cudaStream_t stream) {
  if (L.n_items == 0) return cudaSuccess;
  const int fsw = L.fspill ? L.fs_span : 0;
  if (L.tile == 128 && L.head_dim == 128) return launch_fsw<128, 128>(L, fsw, stream);
  if (L.tile == 128 && L.head_dim == 64) return launch_fsw<128, 64>(L, fsw, stream);
  if (L.tile == 64 && L.head_dim == 128) return launch_fsw<64, 128>(L, fsw, stream);
  if (L.tile == 64 && L.head_dim == 64) return launch_fsw<64, 64>(L, fsw, stream);
  return cudaErrorInvalidValue;
}

}  // namespace evisel

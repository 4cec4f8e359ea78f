// Evidence from the coarse token-level map of the sparse prefill (Appendix,
// "Detailed Sparse Prefilling", Eq. 10-11). For a text row i of head h:
//   a_im = scale q_i k_m              for the keys of its own block up to i (E_i),
//   a_im = g_ij = scale q_i k_bar_j   for the tokens of each retained block j in S_i,
//   -inf elsewhere;  A~_im = exp(a_im) / sum_n exp(a_in)                (Eq. 11)
// and the maps of Sec. 3.2: tok[h, m] = sum over the text rows of A~_im for the
// visual tokens m, frame sums, head sums and A_qf. All tokens of a retained
// visual block share its weight exp(g_ij - M_i) / Z_i.
//
// coarse_logits_kernel: one CTA per (16 text rows of a video, 256 blocks, head):
//   a lane takes one block for all 16 rows, so that its k_bar values are
//   converted once; the rows' q sit in shared memory as fp32 (broadcast reads),
//   two dims per packed fma. Writes g_ij = scale q_i k_bar_j.
// coarse_rows_kernel: a warp per (text row, head): a running max and sum over
//   the row's retained blocks (B tokens each) and over the exact logits s of
//   its own block's causal prefix E_i (a lane per key), merged over the lanes:
//   M_i and Z_i = sum_{S_i} B exp(g - M) + sum_{E_i} exp(s - M).
// coarse_map_kernel: one CTA per (32 visual blocks, head): a lane per block, the
//   text rows dealt over eight warps whose sums meet in shared memory in warp
//   order (deterministic): c_j = sum over the video's text rows of [j in S_i]
//   exp(g_ij - M_i) / Z_i; writes c_j to the block's tokens and B sum_j c_j to
//   the frame.
// coarse_finalize_kernel: head[b, h] = sum of the video's frames (a warp each);
//   A_qf[t] = sum_h frame[h, t] / (Hq n_text) (a thread per frame), from the
//   (possibly accumulated) frame map.
// What bounds it: a few MB and under 1 GFLOP, so latency: serial loops over a
// row's own keys (a load and a warp sum per key), over the text rows of a frame
// in one thread and over a head's frames in one thread took 64, 40 and 15 us on
// 16,388 tokens (28 heads, 100 text rows, B = 32); here the logits, rows, map and
// finalize kernels take 22, 14, 9 and 3 us, the call 137 -> 56 us (its per-video
// offsets now come with the builder's upload: no copy, no synchronisation).
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "evisel_internal.h"
#include "sm103_ptx.cuh"

namespace evisel {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float warp_sum(float x) {
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(kFull, x, off);
  return x;
}

// Two bf16 values as a packed pair of fp32.
__device__ __forceinline__ uint64_t up2(uint32_t x) {
  return ptx::f2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u));
}

// (m, z) <- the softmax pair of (m, z) and (m2, z2): max and rescaled sum.
__device__ __forceinline__ void merge_mz(float& m, float& z, float m2, float z2) {
  const float mm = fmaxf(m, m2);
  z = mm == -INFINITY ? 0.f : z * __expf(m - mm) + z2 * __expf(m2 - mm);
  m = mm;
}

// The video and group of the i-th group of `per` things (text rows, visual
// blocks), where off(v) is the number of things before video v. Video v's groups
// start at off(v) / per + v: room for a partial group per video, and found by
// bisection (a linear search in every CTA took most of the call from some
// hundred videos on). Groups past a video's last thing are empty.
template <typename Off>
__device__ __forceinline__ int video_of_group(const CoarseLaunch& L, int i, int per, Off off, int& grp) {
  int lo = 0, hi = L.n_videos - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off(L.vids[mid]) / per + mid <= i) lo = mid; else hi = mid - 1;
  }
  grp = i - (off(L.vids[lo]) / per + lo);
  return lo;
}

// The video and group of the i-th group of `per` text rows (false: an empty one).
__device__ __forceinline__ bool row_group(const CoarseLaunch& L, int i, int per, int& v, int& grp) {
  v = video_of_group(L, i, per, [](const ToppVideo& x) { return x.text_off; }, grp);
  return grp * per < L.vids[v].n_text;
}

constexpr int kLogitRows = 16;                   // text rows per CTA of the logits
constexpr int kLogitBlocks = 256;                // blocks per CTA (32 per warp)

template <int D>
__global__ void __launch_bounds__(256) coarse_logits_kernel(const __grid_constant__ CoarseLaunch L) {
  __shared__ __align__(16) float q_s[kLogitRows][D];
  const int h = blockIdx.z;
  int v, grp;
  if (!row_group(L, blockIdx.x, kLogitRows, v, grp)) return;   // CTA-uniform
  const ToppVideo vid = L.vids[v];
  const int row0 = grp * kLogitRows, nr = min(kLogitRows, vid.n_text - row0);
  const int B = L.block, nvb = vid.n_vis / B;
  const int nh = nvb + (row0 + nr - 1) / B;      // blocks that end before the group's last row
  if (static_cast<int>(blockIdx.y) * kLogitBlocks >= nh) return;
  const __nv_bfloat16* q = static_cast<const __nv_bfloat16*>(L.q);
  for (int i = threadIdx.x; i < kLogitRows * D; i += blockDim.x) {
    const int r = i / D, e = i % D;
    q_s[r][e] = r < nr ? __bfloat162float(q[(static_cast<int64_t>(vid.start + vid.n_vis + row0 + r) * L.hq + h) * D + e]) : 0.f;
  }
  __syncthreads();
  const int j = blockIdx.y * kLogitBlocks + threadIdx.x;
  if (j >= nh) return;
  const int g = h / (L.hq / L.hkv);
  const uint4* kb = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(L.kbar) +
                                                   (static_cast<int64_t>(vid.blk_off + j) * L.hkv + g) * D);
  uint64_t acc[kLogitRows];
#pragma unroll
  for (int r = 0; r < kLogitRows; ++r) acc[r] = 0;
#pragma unroll 4
  for (int c = 0; c < D / 8; ++c) {
    const uint4 x = __ldg(kb + c);
    const uint64_t k0 = up2(x.x), k1 = up2(x.y), k2 = up2(x.z), k3 = up2(x.w);
#pragma unroll
    for (int r = 0; r < kLogitRows; ++r) {
      const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(&q_s[r][c * 8]);
      const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(&q_s[r][c * 8 + 4]);
      acc[r] = ptx::fma2(a.x, k0, acc[r]);
      acc[r] = ptx::fma2(a.y, k1, acc[r]);
      acc[r] = ptx::fma2(b.x, k2, acc[r]);
      acc[r] = ptx::fma2(b.y, k3, acc[r]);
    }
  }
  float* out = L.gbuf + (static_cast<int64_t>(h) * L.total_text + vid.text_off + row0) * L.pitch + j;
#pragma unroll
  for (int r = 0; r < kLogitRows; ++r) {
    float lo, hi;
    ptx::unf2(acc[r], lo, hi);
    if (r < nr) out[static_cast<int64_t>(r) * L.pitch] = (lo + hi) * L.scale;
  }
}

constexpr int kRowsPerCta = 8;                   // text rows (warps) per CTA

template <int D>
__global__ void __launch_bounds__(kRowsPerCta * 32) coarse_rows_kernel(const __grid_constant__ CoarseLaunch L) {
  __shared__ __align__(16) float q_s[kRowsPerCta][D];
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.y;
  int v, grp;
  if (!row_group(L, blockIdx.x, kRowsPerCta, v, grp)) return;
  const ToppVideo vid = L.vids[v];
  const int t = grp * kRowsPerCta + wib;         // text row within the video
  if (t >= vid.n_text) return;                   // warp-uniform; no CTA barrier below
  const int trow = vid.text_off + t;             // text row over all videos
  const int pos = vid.n_vis + t;                 // video-local position
  const int row = vid.start + pos;               // global token
  const int B = L.block;
  const int nh = vid.n_vis / B + t / B;          // blocks that end before the row
  const int own0 = vid.n_vis + (t / B) * B;      // first token of its own block
  const int g = h / (L.hq / L.hkv);
  const __nv_bfloat16* q = static_cast<const __nv_bfloat16*>(L.q) + (static_cast<int64_t>(row) * L.hq + h) * D;
  for (int e = lane; e < D; e += 32) q_s[wib][e] = __bfloat162float(q[e]);
  __syncwarp();
  float m = -INFINITY, z = 0.f;
  auto add = [&](float x, float n) {             // n tokens of logit x
    if (x > m) {
      z = (m == -INFINITY) ? 0.f : z * __expf(m - x);
      m = x;
    }
    z += n * __expf(x - m);
  };
  // S_i: the row's retained blocks, eight words at a time.
  const float* grow = L.gbuf + (static_cast<int64_t>(h) * L.total_text + trow) * L.pitch;
  const uint32_t* keep = L.keep + static_cast<int64_t>(h) * L.n_words * L.n_tok + row;
  for (int w0 = 0; w0 * 32 < nh; w0 += 8) {
    float x[8];
    uint32_t word[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int j = (w0 + i) * 32 + lane;
      x[i] = j < nh ? grow[j] : 0.f;
      word[i] = (w0 + i) * 32 < nh ? __ldg(keep + static_cast<int64_t>(w0 + i) * L.n_tok) : 0u;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if ((w0 + i) * 32 + lane < nh && ((word[i] >> lane) & 1u)) add(x[i], static_cast<float>(B));
  }
  // E_i: exact logits of the own block's causal prefix, a lane per key.
  const __nv_bfloat16* k = static_cast<const __nv_bfloat16*>(L.k);
  const bool aligned = (reinterpret_cast<uintptr_t>(k) & 15u) == 0;   // (the caller's k; k_bar is the workspace's)
  for (int mm = own0 + lane; mm <= pos; mm += 32) {
    const __nv_bfloat16* kr = k + (static_cast<int64_t>(vid.start + mm) * L.hkv + g) * D;
    auto load8 = [&](int c) {
      if (aligned) return __ldg(reinterpret_cast<const uint4*>(kr) + c);
      const uint16_t* e = reinterpret_cast<const uint16_t*>(kr) + c * 8;
      return make_uint4(e[0] | e[1] << 16, e[2] | e[3] << 16, e[4] | e[5] << 16, e[6] | e[7] << 16);
    };
    uint64_t acc[2] = {0, 0};
#pragma unroll 4
    for (int c = 0; c < D / 8; ++c) {
      const uint4 x = load8(c);
      const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(&q_s[wib][c * 8]);
      const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(&q_s[wib][c * 8 + 4]);
      acc[0] = ptx::fma2(a.x, up2(x.x), acc[0]);
      acc[1] = ptx::fma2(a.y, up2(x.y), acc[1]);
      acc[0] = ptx::fma2(b.x, up2(x.z), acc[0]);
      acc[1] = ptx::fma2(b.y, up2(x.w), acc[1]);
    }
    float s0, s1, s2, s3;
    ptx::unf2(acc[0], s0, s1);
    ptx::unf2(acc[1], s2, s3);
    add(((s0 + s1) + (s2 + s3)) * L.scale, 1.f);
  }
  __syncwarp();
  for (int off = 16; off > 0; off >>= 1) {       // symmetric merges: all lanes agree
    const float m2 = __shfl_xor_sync(kFull, m, off), z2 = __shfl_xor_sync(kFull, z, off);
    merge_mz(m, z, m2, z2);
  }
  if (lane == 0) {
    L.row_m[static_cast<int64_t>(h) * L.total_text + trow] = m;
    L.row_z[static_cast<int64_t>(h) * L.total_text + trow] = z;
  }
}

constexpr int kMapWarps = 8;

__global__ void __launch_bounds__(kMapWarps * 32) coarse_map_kernel(const __grid_constant__ CoarseLaunch L) {
  __shared__ float part[kMapWarps][32];
  __shared__ float c_s[32];
  const int h = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int npf = L.tokens_per_frame, B = L.block;
  int chunk;                                     // of 32 visual blocks
  const ToppVideo vid =
      L.vids[video_of_group(L, blockIdx.x, 32, [B](const ToppVideo& x) { return x.vis_off / B; }, chunk)];
  const int j0 = chunk * 32, nb = min(32, vid.n_vis / B - j0);
  if (nb <= 0) return;                           // CTA-uniform: an empty group
  const int64_t r0 = static_cast<int64_t>(h) * L.total_text + vid.text_off;
  const float* gcol = L.gbuf + r0 * L.pitch + j0 + lane;
  const uint32_t* keep = L.keep + (static_cast<int64_t>(h) * L.n_words + chunk) * L.n_tok + vid.start + vid.n_vis;
  float c = 0.f;
#pragma unroll 4
  for (int i = warp; i < vid.n_text; i += kMapWarps) {
    const uint32_t word = __ldg(keep + i);
    const float x = lane < nb ? gcol[static_cast<int64_t>(i) * L.pitch] : 0.f;
    const float m = L.row_m[r0 + i], z = L.row_z[r0 + i];
    if (lane < nb && ((word >> lane) & 1u)) c += __expf(x - m) / z;
  }
  part[warp][lane] = c;
  __syncthreads();
  if (warp == 0) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kMapWarps; ++w) s += part[w][lane];
    c_s[lane] = s;
  }
  __syncthreads();
  float* tok = L.tok + static_cast<int64_t>(h) * L.total_vis + vid.vis_off + static_cast<int64_t>(j0) * B;
  for (int i = threadIdx.x; i < nb * B; i += blockDim.x) tok[i] = L.accumulate ? tok[i] + c_s[i / B] : c_s[i / B];
  const int per = npf / B;                       // blocks per frame: 1 .. 8, so frames stay in a chunk
  if (threadIdx.x < nb / per) {
    float f = 0.f;
    for (int i = 0; i < per; ++i) f += static_cast<float>(B) * c_s[threadIdx.x * per + i];
    float* fr = L.frame + static_cast<int64_t>(h) * L.total_frames + vid.vis_off / npf + j0 / per + threadIdx.x;
    *fr = L.accumulate ? *fr + f : f;
  }
}

constexpr int kFinalWarps = 8;

// Blocks [0, n_videos * head_blocks): a warp per (video, head); then a thread per frame.
__global__ void __launch_bounds__(kFinalWarps * 32) coarse_finalize_kernel(const __grid_constant__ CoarseLaunch L,
                                                                          int head_blocks) {
  const int npf = L.tokens_per_frame;
  if (static_cast<int>(blockIdx.x) < L.n_videos * head_blocks) {
    const int v = blockIdx.x / head_blocks, lane = threadIdx.x & 31;
    const int h = (blockIdx.x % head_blocks) * kFinalWarps + (threadIdx.x >> 5);
    if (h >= L.hq) return;
    const ToppVideo vid = L.vids[v];
    const int frames = vid.n_vis / npf;
    const float* fr = L.frame + static_cast<int64_t>(h) * L.total_frames + vid.vis_off / npf;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    int t = lane;
    for (; t + 96 < frames; t += 128) {
#pragma unroll
      for (int i = 0; i < 4; ++i) s[i] += fr[t + 32 * i];
    }
    for (; t < frames; t += 32) s[0] += fr[t];
    const float sum = warp_sum((s[0] + s[1]) + (s[2] + s[3]));
    if (lane == 0) L.head[static_cast<int64_t>(v) * L.hq + h] = sum;
    return;
  }
  const int t = (blockIdx.x - L.n_videos * head_blocks) * blockDim.x + threadIdx.x;
  if (t >= L.total_frames) return;
  int lo = 0, hi = L.n_videos - 1;               // the video that owns frame t
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (L.vids[mid].vis_off / npf <= t) lo = mid; else hi = mid - 1;
  }
  const int n_text = L.vids[lo].n_text;
  float s0 = 0.f, s1 = 0.f;
#pragma unroll 4
  for (int h = 0; h + 1 < L.hq; h += 2) {
    s0 += L.frame[static_cast<int64_t>(h) * L.total_frames + t];
    s1 += L.frame[static_cast<int64_t>(h + 1) * L.total_frames + t];
  }
  if (L.hq & 1) s0 += L.frame[static_cast<int64_t>(L.hq - 1) * L.total_frames + t];
  L.aqf[t] = n_text > 0 ? (s0 + s1) / (static_cast<float>(L.hq) * static_cast<float>(n_text)) : 0.f;
}

template <int D>
cudaError_t launch_rows(const CoarseLaunch& L, cudaStream_t stream) {
  // Row groups per video: at most total / size full ones and a partial one per
  // video; CTAs past the last group return at once. The groups take grid x: y and
  // z end at 65,535.
  dim3 g1(L.total_text / kLogitRows + L.n_videos, (L.max_blocks + kLogitBlocks - 1) / kLogitBlocks, L.hq);
  coarse_logits_kernel<D><<<g1, 256, 0, stream>>>(L);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  dim3 g2(L.total_text / kRowsPerCta + L.n_videos, L.hq);
  coarse_rows_kernel<D><<<g2, kRowsPerCta * 32, 0, stream>>>(L);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_coarse(const CoarseLaunch& L, cudaStream_t stream) {
  if (L.n_videos == 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  if (L.total_text > 0 && L.max_blocks > 0) {
    e = L.head_dim == 128 ? launch_rows<128>(L, stream) : launch_rows<64>(L, stream);
    if (e != cudaSuccess) return e;
  }
  if (L.total_vis > 0) {
    dim3 g((L.total_vis / L.block) / 32 + L.n_videos, L.hq);
    coarse_map_kernel<<<g, kMapWarps * 32, 0, stream>>>(L);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const int head_blocks = (L.hq + kFinalWarps - 1) / kFinalWarps;
  const int aqf_blocks = (L.total_frames + kFinalWarps * 32 - 1) / (kFinalWarps * 32);
  coarse_finalize_kernel<<<L.n_videos * head_blocks + aqf_blocks, kFinalWarps * 32, 0, stream>>>(L, head_blocks);
  return cudaGetLastError();
}

}  // namespace evisel

// Evidence maps of the text rows (Sec. 3.2, "Evidence Decomposition") from the
// token and frame sums that the text-evidence kernel formed.
//
// After a probe with text_evidence = 0 those sums sit in the workspace
// (formed inside the probe call) and evidence_maps_kernel hands them out:
// overwriting, one launch copies the token map and forms the frame, head and
// A_qf maps; accumulating over layers, evidence_add_kernel adds them into the
// caller's maps first. After a probe with text_evidence = 1 the sums were
// written to the caller's maps directly.
//   head map: sum of a video's frames per head (one warp per video and head)
//   A_qf:     sum over heads / (Hq n_text) (one thread per frame)
// Both are recomputed from the resulting frame map, so that they accumulate
// over layers exactly as it does. A few MB move: launches and latency are what
// the call costs (65,664 tokens: 9 us; the pass that read 940 MB of spilled
// logits back took 164 us).
#include <cstdint>
#include <cuda_runtime.h>

#include "evisel_internal.h"

namespace evisel {
namespace {

constexpr int kWarps = 8;
constexpr int kCopyPerThread = 4;                // float4 per thread of a copy block

// tok += src_tok (float4), frame += src_frame.
__global__ void __launch_bounds__(kWarps * 32) evidence_add_kernel(const __grid_constant__ EvidenceLaunch L) {
  const int64_t n4 = static_cast<int64_t>(L.hq) * L.total_vis / 4;   // N_v is a multiple of 4
  const int64_t nf = static_cast<int64_t>(L.hq) * L.total_frames;
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = i0; i < n4; i += stride) {
    float4 a = reinterpret_cast<float4*>(L.tok)[i];
    const float4 b = reinterpret_cast<const float4*>(L.src_tok)[i];
    a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
    reinterpret_cast<float4*>(L.tok)[i] = a;
  }
  for (int64_t i = i0; i < nf; i += stride) L.frame[i] += L.src_frame[i];
}

// Blocks [0, n_videos * head_blocks): head map, one warp per (video, head),
// four independent partial sums per lane. The next aqf_blocks: A_qf, one
// thread per frame, and the frame map where kCopy. The rest (kCopy): the token
// map, 16 bytes a thread. Frames are read from fsrc (the workspace where
// kCopy, else the caller's frame map).
template <bool kCopy>
__global__ void __launch_bounds__(kWarps * 32) evidence_maps_kernel(const __grid_constant__ EvidenceLaunch L,
                                                                   int head_blocks, int aqf_blocks) {
  const float* fsrc = kCopy ? L.src_frame : L.frame;
  int blk = blockIdx.x;
  if (blk < L.n_videos * head_blocks) {
    const int b = blk / head_blocks;
    const int h = (blk % head_blocks) * kWarps + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (h >= L.hq) return;
    const VideoInfo vi = L.videos[b];
    const int frames = vi.n_vis / L.tokens_per_frame;
    const float* fr = fsrc + static_cast<int64_t>(h) * L.total_frames + vi.frame_off;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    int t = lane;
    for (; t + 96 < frames; t += 128) {
      s0 += fr[t];
      s1 += fr[t + 32];
      s2 += fr[t + 64];
      s3 += fr[t + 96];
    }
    for (; t < frames; t += 32) s0 += fr[t];
    float s = (s0 + s1) + (s2 + s3);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) L.head[static_cast<int64_t>(b) * L.hq + h] = s;
    return;
  }
  blk -= L.n_videos * head_blocks;
  if (blk < aqf_blocks) {
    const int t = blk * blockDim.x + threadIdx.x;
    if (t >= L.total_frames) return;
    int lo = 0, hi = L.n_videos - 1;               // video owning frame t
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (L.videos[mid].frame_off <= t) lo = mid; else hi = mid - 1;
    }
    // (the last video whose frame offset is <= t always owns >= 1 frame)
    const int n_text = L.videos[lo].n_text;
    float s0 = 0.f, s1 = 0.f;
    int h = 0;
    for (; h + 3 < L.hq; h += 4) {                 // four loads in flight
      float x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = fsrc[static_cast<int64_t>(h + i) * L.total_frames + t];
      if (kCopy) {
#pragma unroll
        for (int i = 0; i < 4; ++i) L.frame[static_cast<int64_t>(h + i) * L.total_frames + t] = x[i];
      }
      s0 += x[0];
      s1 += x[1];
      s0 += x[2];
      s1 += x[3];
    }
    for (; h < L.hq; ++h) {
      const float x = fsrc[static_cast<int64_t>(h) * L.total_frames + t];
      if (kCopy) L.frame[static_cast<int64_t>(h) * L.total_frames + t] = x;
      if (h & 1) s1 += x; else s0 += x;
    }
    L.aqf[t] = n_text > 0 ? (s0 + s1) / (static_cast<float>(L.hq) * static_cast<float>(n_text)) : 0.f;
    return;
  }
  if constexpr (kCopy) {
    blk -= aqf_blocks;
    const int64_t n4 = static_cast<int64_t>(L.hq) * L.total_vis / 4;   // N_v is a multiple of 4
    const int64_t i0 = static_cast<int64_t>(blk) * blockDim.x * kCopyPerThread + threadIdx.x;
#pragma unroll
    for (int j = 0; j < kCopyPerThread; ++j) {
      const int64_t i = i0 + j * blockDim.x;
      if (i < n4) reinterpret_cast<float4*>(L.tok)[i] = reinterpret_cast<const float4*>(L.src_tok)[i];
    }
  }
}

}  // namespace

cudaError_t launch_evidence(const EvidenceLaunch& L, cudaStream_t stream) {
  constexpr int kThreads = kWarps * 32;
  const int head_blocks = (L.hq + kWarps - 1) / kWarps;
  const int aqf_blocks = (L.total_frames + kThreads - 1) / kThreads;
  const int64_t n4 = static_cast<int64_t>(L.hq) * L.total_vis / 4;
  const bool copy = L.src_tok && !L.accumulate;
  if (L.src_tok && L.accumulate && n4 > 0) {
    const int64_t blocks = (n4 + kThreads - 1) / kThreads;
    evidence_add_kernel<<<static_cast<unsigned>(blocks < 2048 ? blocks : 2048), kThreads, 0, stream>>>(L);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const int64_t per = static_cast<int64_t>(kThreads) * kCopyPerThread;
  const int64_t blocks = static_cast<int64_t>(L.n_videos) * head_blocks + aqf_blocks + (copy ? (n4 + per - 1) / per : 0);
  if (blocks == 0) return cudaSuccess;
  if (copy) evidence_maps_kernel<true><<<static_cast<unsigned>(blocks), kThreads, 0, stream>>>(L, head_blocks, aqf_blocks);
  else evidence_maps_kernel<false><<<static_cast<unsigned>(blocks), kThreads, 0, stream>>>(L, head_blocks, aqf_blocks);
  return cudaGetLastError();
}

}  // namespace evisel
